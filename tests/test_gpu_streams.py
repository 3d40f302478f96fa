"""The calls among other work on the caller's streams: inputs that another stream finishes late, behind a wait on its event, and
capture into a CUDA graph.  Streams against the oracle to the bit, aggregates within the usual tolerance."""
import numpy as np
import pytest

import oracle as O
from gpu_util import assert_aggregate_close, gpu_params, oracle_params, params_dict

pytestmark = pytest.mark.gpu

D, N = 200_003, 3
FORKED = 700_003  # coordinates of clients that cvlc_compress_batch does not give to clusters: the length tuning runs on the side stream
KINDS = ["client", "compress", "separate", "ec", "decode", "unframed", "decode_unframed"]


class Calls:
    """Buffers of N clients.  `load` puts one of two sets of inputs in place, `run` makes the calls of a kind on the current stream,
    `check` compares what they left with the oracle's for a set of inputs."""

    def __init__(self, kind, D=D):
        import torch
        from paper_2402_03770_b200 import binding as B
        self.torch, self.B, self.kind, self.D = torch, B, kind, D
        self.dev = dev = torch.device("cuda:0")
        rng = np.random.default_rng(len(kind))
        self.pds = [params_dict(D, 2 * D, seed=11 + c, client_id=c) for c in range(N)]
        self.params = [gpu_params(pd) for pd in self.pds]
        self.updates = [[rng.laplace(0, 10.0 ** -(3 + s), D).astype(np.float32) for _ in range(N)] for s in range(2)]
        self.weights = np.array([1.0, 2.5, 3.0], np.float32)
        self.plans = [[O.plan(x, oracle_params(pd)) for x, pd in zip(xs, self.pds)] for xs in self.updates]
        encode = O.encode_unframed if "unframed" in kind else O.encode
        self.streams = [[encode(x, oracle_params(pd), pl) for x, pd, pl in zip(xs, self.pds, pls)]
                        for xs, pls in zip(self.updates, self.plans)]
        decode = O.decode_aggregate_unframed if "unframed" in kind else O.decode_aggregate
        self.aggregates = [decode(s, self.weights, D) for s in self.streams]

        self.enc = B.BatchEncoder(self.params, dev)
        self.clients = [B.ClientEncoder(p, dev) for p in self.params]
        self.memory = torch.zeros(N, (D + 3) // 4 * 4, device=dev)
        self.memories = [self.memory[c, :D] for c in range(N)]
        self.side = torch.cuda.Stream(dev)
        size = max(B.cvlc_stream_bytes(self.params[0]), B.cvlc_unframed_stream_capacity(self.params[0]))
        self.bytes_in = [torch.zeros(size, dtype=torch.uint8, device=dev) for _ in range(N)]
        self.bytes_out = [torch.zeros(size, dtype=torch.uint8, device=dev) for _ in range(N)]
        self.sizes = torch.zeros(N, dtype=torch.int64, device=dev)
        self.uf_ws = B.alloc_bytes(B.cvlc_unframed_workspace_bytes(self.params[0], N), dev)
        self.out = torch.zeros(D, device=dev)
        self.agg = B.Aggregator(N, D, dev)
        self.agg.set_clients(self.bytes_in, torch.from_numpy(self.weights))
        self.xs = [torch.zeros(D, device=dev) for _ in range(N)]
        # the sets as they lie on the device, to be copied into place without the host
        if kind.startswith("decode"):
            self.to = self.bytes_in + [self.agg.sizes]
            self.sets = [[torch.nn.functional.pad(torch.from_numpy(s), (0, size - s.size)).to(dev) for s in streams] +
                         [torch.tensor([s.size for s in streams], dtype=torch.int64, device=dev)] for streams in self.streams]
        else:
            self.to = self.xs
            self.sets = [[torch.from_numpy(x).to(dev) for x in xs] for xs in self.updates]
        torch.cuda.synchronize()

    def load(self, which):
        for a, b in zip(self.to, self.sets[which]):
            a.copy_(b)

    def run(self):
        B, kind, enc = self.B, self.kind, self.enc
        if kind == "client":
            for c in range(N):
                self.clients[c].run(self.xs[c])
        elif kind == "compress":
            enc.compress(self.xs, side_stream=self.side)
        elif kind == "separate":
            enc.run(self.xs)
        elif kind == "ec":
            self.memory.zero_()
            B.cvlc_ec_accumulate_batch(self.memories, self.xs)
            B.cvlc_plan_batch(self.memories, self.params, enc.plans, enc.plan_ws)
            B.cvlc_encode_batch_ec(self.memories, self.params, enc.plans, enc.outs, enc.enc_ws, 0, plan_ws=enc.plan_ws)
        elif kind == "decode":
            self.agg.run(N, self.out)
        elif kind == "unframed":
            enc.plan(self.xs)
            B.cvlc_encode_unframed_batch(self.xs, self.params, enc.plans, self.bytes_out, self.sizes, enc.enc_ws, self.uf_ws, 0,
                                         plan_ws=enc.plan_ws)
        else:
            B.cvlc_decode_aggregate_unframed(self.agg.ptrs, self.agg.sizes, self.agg.weights, N, 0.0, self.D, self.out, False, self.agg.ws)

    def check(self, which):
        self.torch.cuda.synchronize()
        if self.kind.startswith("decode"):
            assert self.agg.status() == 0
            assert_aggregate_close(self.out.cpu().numpy(), self.aggregates[which])
            return
        if self.kind == "client":
            assert all(e.status() == 0 for e in self.clients)
            outs = [e.out for e in self.clients]
        else:
            assert self.enc.status() == 0
            outs = self.bytes_out if self.kind == "unframed" else self.enc.outs
        for c, ref in enumerate(self.streams[which]):
            assert (outs[c].cpu().numpy()[:ref.size] == ref).all(), c
            if self.kind == "unframed":
                assert int(self.sizes[c]) == ref.size
            if self.kind == "ec":
                assert (self.memories[c].cpu().numpy() == O.ec_residual(self.updates[which][c], ref)).all()


SIZES = [(kind, D) for kind in KINDS] + [("client", FORKED), ("compress", FORKED)]


@pytest.mark.parametrize("kind,d", SIZES)
def test_inputs_behind_an_event_wait(kind, d):
    """The stream holds a finished call on other inputs, then a wait for the stream that is still making the right ones."""
    calls = Calls(kind, d)
    torch = calls.torch
    work, maker, made = torch.cuda.Stream(calls.dev), torch.cuda.Stream(calls.dev), torch.cuda.Event()
    with torch.cuda.stream(work):
        calls.load(0)
        calls.run()
    calls.check(0)
    for which in (1, 0):
        torch.cuda.synchronize()
        with torch.cuda.stream(maker):
            torch.cuda._sleep(20_000_000)  # about 10 ms
            calls.load(which)
            made.record()
        with torch.cuda.stream(work):
            work.wait_event(made)
            calls.run()
        calls.check(which)


@pytest.mark.parametrize("kind,d", SIZES)
def test_capture_into_a_graph(kind, d):
    """One capture, replayed for two sets of inputs; with the larger clients the length tuning's fork is captured with it."""
    calls = Calls(kind, d)
    torch = calls.torch
    warm = torch.cuda.Stream(calls.dev)
    with torch.cuda.stream(warm):  # attributes are set and modules loaded before the capture
        calls.load(0)
        calls.run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls.run()
    for which in (1, 0, 1):
        calls.load(which)
        graph.replay()
        calls.check(which)


def test_capture_behind_a_call_by_clusters():
    """In a process of its own: a two-stream call of a small client, which forks nothing, is enough for one that does to be captured."""
    import os
    import subprocess
    import sys
    code = """if 1:
        import numpy as np, torch
        from gpu_util import gpu_params, oracle_plan_encode, params_dict
        from paper_2402_03770_b200 import binding as B
        dev = torch.device("cuda:0")
        side, ready = torch.cuda.Stream(dev), []
        for d in (20_001, 700_003):
            x = np.random.default_rng(d).laplace(0, 1e-3, d).astype(np.float32)
            pd = params_dict(d, d)
            ready.append((B.BatchEncoder([gpu_params(pd)], dev), torch.from_numpy(x).to(dev), oracle_plan_encode(x, pd)[1]))
        ready[1][0].run([ready[1][1]])  # its kernels' attributes, without a second stream
        ready[1][0].compress([ready[1][1]])
        ready[0][0].compress([ready[0][1]], side_stream=side)
        torch.cuda.synchronize()
        assert B.cvlc_launch_count("k_client") == 1
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ready[1][0].compress([ready[1][1]], side_stream=side)
        ready[1][0].outs[0].zero_()
        graph.replay()
        torch.cuda.synchronize()
        for enc, _, stream in ready:
            assert enc.status() == 0 and np.array_equal(enc.outs[0].cpu().numpy(), stream)
        """
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([here, os.path.dirname(here)] + os.environ.get("PYTHONPATH", "").split(os.pathsep)))
    done = subprocess.run([sys.executable, "-c", code], env=env, timeout=120, capture_output=True, text=True)
    assert done.returncode == 0, done.stderr


def test_calls_from_several_threads():
    """Every thread on a stream and buffers of its own; no launch is missing from the count.  Four of them share the device's two events."""
    import threading
    import torch
    from paper_2402_03770_b200 import binding as B
    kinds = ["client", "compress", "separate", "ec", "decode", "unframed", "decode_unframed", "compress"]
    work = [Calls(kind) for kind in kinds] + [Calls(kind, FORKED) for kind in ("client", "compress", "compress", "client")]
    each = []
    for calls in work:
        calls.load(0)
        before = B.cvlc_launch_count()
        calls.run()
        each.append(B.cvlc_launch_count() - before)
    torch.cuda.synchronize()
    failed = []

    def repeat(calls):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream(calls.dev)):
                for i in range(30):
                    calls.load((i + 1) % 2)
                    calls.run()
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001
            failed.append((calls.kind, e))

    before = B.cvlc_launch_count()
    threads = [threading.Thread(target=repeat, args=(calls,)) for calls in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    assert B.cvlc_launch_count() - before == 30 * sum(each)
    for calls in work:
        calls.check(0)


def test_encoders_on_two_streams_do_not_wait_for_each_other():
    """More encoders than torch has streams of a kind: those used on one stream finish while the other stream is held up."""
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    pd = params_dict(20_001, 12_000 * 4, seed=1)
    x = np.random.default_rng(3).laplace(0, 1e-3, 20_001).astype(np.float32)
    ref = O.encode(x, oracle_params(pd), O.plan(x, oracle_params(pd)))
    dx = torch.from_numpy(x).to(dev)
    encoders = [B.ClientEncoder(gpu_params(pd), dev) for _ in range(72)]
    held, free = torch.cuda.Stream(dev), torch.cuda.Stream(dev)
    for s in (held, free):
        encoders[0].run(dx, stream=s)
        s.synchronize()
    with torch.cuda.stream(held):
        torch.cuda._sleep(600_000_000)  # about 0.3 s
        encoders[0].run(dx)
    for e in encoders[1:]:
        e.run(dx, stream=free)
    free.synchronize()
    assert not held.query()
    held.synchronize()
    for e in encoders:
        assert e.status() == 0 and (e.out.cpu().numpy() == ref).all()
