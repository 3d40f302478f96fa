"""Performance cases of the compression path: what its users have it do, through the public entry points.

A case is a dict of plain values:

    kind       client    one client compresses its own update (ClientEncoder.run: plan, then encode)
               round     a batch of clients is compressed and aggregated (cvlc_compress_batch with a side stream, then
                         Aggregator.run); with `batches` > 1 the round is streamed through one set of buffers
               ec        a round with error compensation on the clients' side (accumulate, plan, encode with residual)
               server    the parameter server alone: decode, aggregate and model step (Aggregator.apply)
               unframed  a round in the unframed format (plan, encode, decode-aggregate)
    d          coordinates of an update
    clients    clients of the round (over all batches)
    batches    calls the round is split into
    bits       uplink budget in bits per coordinate (packets of 1500 bytes)
    quantizer  "pq" or "qsgd"
    values     the update's distribution, the four recipes of the package's workloads: "laplace", "laplace_blocks",
               "gauss_blocks", "student_blocks"

Inputs are drawn on the GPU from the seed; every client has its own.  Buffers, workspaces, streams, pointer tables and
parameter blocks are made once in `prepare`, as a program that runs many rounds keeps them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_03770_b200 import binding as B
from paper_2402_03770_b200 import workloads as W

QUANTIZERS = {"pq": B.CVLC_QUANT_PQ, "qsgd": B.CVLC_QUANT_QSGD}
N_BLOCKS = {"laplace": 1, "laplace_blocks": 8, "gauss_blocks": 62, "student_blocks": 161}


def _case(name, kind, d, clients, bits, values, quantizer="pq", batches=1):
    return {"name": name, "kind": kind, "d": d, "clients": clients, "batches": batches, "bits": bits,
            "quantizer": quantizer, "values": values}


def listed():
    return [
        # one small update: the smallest call, where launches and the length tuning's latency are all there is
        _case("client_tiny", "client", 100_000, 1, 1.0, "laplace"),
        # a client that compresses a ResNet-18-sized update on its own GPU
        _case("client_resnet18", "client", 11_200_000, 1, 2.0, "gauss_blocks"),
        # the paper's CIFAR-10 setting: a 3-layer CNN, 10 clients a round, 10 packets each
        _case("round_paper_cnn", "round", 300_000, 10, 0.4, "laplace_blocks"),
        # a small CNN with a generous budget
        _case("round_small_cnn", "round", 1_200_000, 20, 2.0, "laplace_blocks"),
        # the benchmark's round: 100 clients of ResNet-18 size
        _case("round_resnet18", "round", 11_200_000, 100, 2.0, "gauss_blocks"),
        # a dense budget on a size that is a multiple of nothing
        _case("round_dense_ragged", "round", 3_000_001, 24, 4.0, "gauss_blocks"),
        # larger model, heavier tail, all-zero layers and exact ties
        _case("round_resnet50", "round", 23_500_000, 50, 1.0, "student_blocks"),
        # the largest model, mostly sparsified, streamed through the aggregation in two batches
        _case("round_stress", "round", 100_000_000, 20, 0.25, "laplace", batches=2),
        # the second quantizer
        _case("round_qsgd_ragged", "round", 3_000_001, 24, 2.0, "gauss_blocks", quantizer="qsgd"),
        # the paper's CIFAR-100 setting (90 packets for a 4-layer CNN) with error compensation
        _case("ec_paper_cnn100", "ec", 5_000_000, 10, 0.216, "gauss_blocks"),
        # the parameter server: 100 clients' packets into a ResNet-18-sized model
        _case("server_resnet18", "server", 11_200_000, 100, 1.0, "gauss_blocks"),
        # the unframed format, both directions
        _case("unframed_small_cnn", "unframed", 1_200_003, 8, 2.0, "laplace_blocks"),
    ]


# most coordinates of a pass, and most coordinates times bits (what is sent), by kind
_LIMITS = {"client": (1.0e8, 4.0e7), "round": (1.1e9, 2.2e9), "ec": (2.0e8, 2.0e8), "server": (1.1e9, 1.1e9),
           "unframed": (2.0e7, 1.9e7)}


def draw(rng):
    def log_uniform(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["client", "round", "round", "round", "round", "ec", "server", "unframed"])
    most, most_sent = _LIMITS[kind]
    bits = round(log_uniform(0.2, 4.0), 3)
    d = int(log_uniform(1e5, min(1e8, most, most_sent / bits)))
    clients = 1 if kind == "client" else int(log_uniform(1.0, max(1.01, min(100.99, most / d, most_sent / (bits * d)))))
    batches = 2 if kind == "round" and d > 30_000_000 and clients >= 2 else 1
    c = _case("", kind, d, clients - clients % batches, bits, rng.choice(sorted(N_BLOCKS)),
              quantizer=rng.choice(["pq", "pq", "qsgd"]), batches=batches)
    del c["name"]
    return c


# ---- inputs -------------------------------------------------------------------------------

class _Updates:
    """Draws the updates of one case on the GPU (client after client from one generator)."""

    def __init__(self, case, seed, device):
        self.d, self.values, self.device = case["d"], case["values"], device
        self.gen = torch.Generator(device=device).manual_seed(seed)
        self.rng = np.random.default_rng(seed)
        n_blocks = N_BLOCKS[self.values]
        self.n_blocks = n_blocks
        if n_blocks > 1:
            sizes = torch.from_numpy(W.block_sizes(self.d, n_blocks, seed=1999)).to(device)
            self.block_of = torch.repeat_interleave(torch.arange(n_blocks, dtype=torch.int32, device=device), sizes, output_size=self.d)

    def _per_block(self, v):
        return torch.from_numpy(np.asarray(v)).to(self.device)[self.block_of]

    def _normal(self):
        return torch.randn(self.d, generator=self.gen, device=self.device)

    def _signed_exponential(self):
        x = torch.empty(self.d, device=self.device).exponential_(generator=self.gen)
        return x.mul_(torch.empty(self.d, device=self.device).bernoulli_(0.5, generator=self.gen).mul_(2.0).sub_(1.0))

    def next(self):
        if self.values == "laplace":
            return self._signed_exponential().mul_(1e-3)
        if self.values == "laplace_blocks":
            return self._signed_exponential().mul_(self._per_block((10.0 ** self.rng.uniform(-4.0, -2.0, self.n_blocks)).astype(np.float32)))
        if self.values == "gauss_blocks":
            std = self._per_block((10.0 ** self.rng.uniform(-5.0, -2.0, self.n_blocks)).astype(np.float32))
            x = self._normal()
            out = torch.rand(self.d, generator=self.gen, device=self.device) < 1e-3
            return torch.where(out, torch.sign(x).mul_(50.0), x).mul_(std)
        # Student-t with 3 degrees of freedom; every tenth block zero, every seventh of the others on a grid (ties)
        x = self._normal()
        chi2 = self._normal().square_()
        for _ in range(2):
            chi2.addcmul_(*[self._normal()] * 2)
        x.mul_(1e-3).div_(chi2.div_(3.0).clamp_(min=1e-12).sqrt_())
        b = np.arange(self.n_blocks)
        zero = b % 10 == 9
        tied = ~zero & (np.cumsum(~zero) % 7 == 0)
        x = torch.where(self._per_block(tied), torch.round(x * 16384.0) / 16384.0, x)
        return x.mul_(self._per_block((~zero).astype(np.float32)))


def _params(case, seed, clients):
    budget = int(math.floor(case["bits"] * case["d"]))
    return [B.make_params(case["d"], budget, quantizer=QUANTIZERS[case["quantizer"]], seed=seed * 4096 + c, client_id=c)
            for c in clients]


def _max_candidates(p):
    s = max(1, math.ceil(math.log2(p.d)))
    R = p.budget_bits // p.packet_bits
    return min(p.d, 3 * R * ((p.packet_bits - p.header_bits) // (s + 1)))


def _bytes(n, device):
    return torch.zeros(n, dtype=torch.uint8, device=device)


def _views(n, size, device):
    """n byte buffers of `size` in one allocation, 256-byte aligned"""
    stride = (size + 255) // 256 * 256
    block = _bytes(n * stride, device).view(n, stride)
    return block, [block[i, :size] for i in range(n)]


def _weights(n, rng):
    return torch.from_numpy(rng.uniform(50.0, 500.0, n).astype(np.float32))  # clients' sample counts


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind, d, n = case["kind"], case["d"], case["clients"]
    updates = _Updates(case, seed, dev)
    s = {"kind": kind, "n": n}
    if kind == "client":
        s["x"] = updates.next()
        s["enc"] = B.ClientEncoder(_params(case, seed, [0])[0], dev)
        s["enc"].plan.zero_()
        return s
    per = n // case["batches"]
    groups = [list(range(i, i + per)) for i in range(0, n, per)]
    params = [_params(case, seed, g) for g in groups]
    p0 = params[0][0]
    # error compensation: the memories flatten against the threshold over the rounds, so any coordinate may become a candidate
    cap = 0 if kind == "ec" else _max_candidates(p0)
    s.update(groups=groups, params=params, cap=cap)
    if kind == "server":
        # the streams come from the clients: compressed here a few at a time, only the packets are kept
        block, outs = _views(n, B.cvlc_stream_bytes(p0), dev)
        few = min(n, 8)
        plans = _bytes(few * B.PLAN_BYTES, dev)
        plan_ws = B.alloc_bytes(B.cvlc_plan_batch_workspace_bytes(p0, few), dev)
        enc_ws = B.alloc_bytes(B.cvlc_encode_batch_workspace_bytes(p0, few, cap), dev)
        for i in range(0, n, few):
            xs = [updates.next() for _ in range(i, min(i + few, n))]
            B.cvlc_compress_batch(xs, params[0][i:i + few], plans, outs[i:i + few], plan_ws, enc_ws, cap)
        torch.cuda.synchronize(dev)
        s.update(streams=block, agg=B.Aggregator(n, d, dev), model=torch.randn(d, generator=updates.gen, device=dev).mul_(0.02),
                 aggregate=torch.zeros(d, device=dev))
        s["agg"].set_clients(outs, _weights(n, updates.rng))
        return s
    xs = [[updates.next() for _ in g] for g in groups]
    s.update(xs=xs, plans=_bytes(per * B.PLAN_BYTES, dev),
             plan_ws=B.alloc_bytes(B.cvlc_plan_batch_workspace_bytes(p0, per), dev),
             enc_ws=B.alloc_bytes(B.cvlc_encode_batch_workspace_bytes(p0, per, cap), dev))
    if kind == "unframed":
        s["block"], s["outs"] = _views(n, B.cvlc_unframed_stream_capacity(p0), dev)
        s["sizes"] = torch.zeros(n, dtype=torch.int64, device=dev)
        s["uf_ws"] = B.alloc_bytes(B.cvlc_unframed_workspace_bytes(p0, n), dev)
    else:
        s["block"], s["outs"] = _views(n, B.cvlc_stream_bytes(p0), dev)
    if kind == "ec":
        s["memory"] = torch.zeros(n, (d + 3) // 4 * 4, device=dev)
        s["memories"] = [s["memory"][i, :d] for i in range(n)]
        return s
    s["side"] = torch.cuda.Stream(dev)
    s["aggs"] = [B.Aggregator(per, d, dev) for _ in groups]
    weights = _weights(n, updates.rng)
    for agg, g in zip(s["aggs"], groups):
        agg.set_clients([s["outs"][c] for c in g], weights[g])
    s["total"] = float(weights.double().sum())
    s["result"] = torch.zeros(d, device=dev)
    return s


# ---- one pass -----------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "client":
        enc = s["enc"]
        return {"stream": enc.run(s["x"]), "plan": enc.plan}
    if kind == "server":
        s["agg"].apply(s["n"], s["model"], s["aggregate"])
        return {"model": s["model"], "aggregate": s["aggregate"]}
    if kind == "ec":
        B.cvlc_ec_accumulate_batch(s["memories"], s["xs"][0])
        B.cvlc_plan_batch(s["memories"], s["params"][0], s["plans"], s["plan_ws"])
        B.cvlc_encode_batch_ec(s["memories"], s["params"][0], s["plans"], s["outs"], s["enc_ws"], s["cap"], plan_ws=s["plan_ws"])
        return {"streams": s["block"], "memory": s["memory"], "plans": s["plans"]}
    if kind == "unframed":
        B.cvlc_plan_batch(s["xs"][0], s["params"][0], s["plans"], s["plan_ws"])
        B.cvlc_encode_unframed_batch(s["xs"][0], s["params"][0], s["plans"], s["outs"], s["sizes"], s["enc_ws"], s["uf_ws"], s["cap"],
                                     plan_ws=s["plan_ws"])
        agg = s["aggs"][0]
        B.cvlc_decode_aggregate_unframed(agg.ptrs, s["sizes"], agg.weights, s["n"], s["total"], agg.d, s["result"], False, agg.ws)
        return {"streams": s["block"], "sizes": s["sizes"], "plans": s["plans"], "aggregate": s["result"]}
    for i, g in enumerate(s["groups"]):
        B.cvlc_compress_batch(s["xs"][i], s["params"][i], s["plans"], [s["outs"][c] for c in g], s["plan_ws"], s["enc_ws"], s["cap"],
                              side_stream=s["side"])
        s["aggs"][i].run(len(g), s["result"], weight_total=s["total"], accumulate=i > 0)
    return {"streams": s["block"], "plans": s["plans"], "aggregate": s["result"]}


def work(case):
    """Inputs once, outputs once: updates, streams and aggregates (the model step reads and writes the model; error
    compensation reads and writes the memories).  Arithmetic: one comparison per coordinate, one multiply-add per record
    of about 30 bits."""
    d, n = case["d"], case["clients"]
    streams = n * math.floor(case["bits"] * d) / 8
    records = 8 * streams / 30
    update = 4.0 * d
    by = {"client": n * update + streams, "round": n * update + streams + update, "ec": 3 * n * update + streams,
          "server": streams + 3 * update, "unframed": n * update + streams + update}[case["kind"]]
    return {"bytes": by, "flops": 2 * records + (0 if case["kind"] == "server" else n * d)}


def tolerance(case):
    """Plans, streams and error-compensation memories are defined to the bit; the aggregate is a sum of fp32 terms in any
    order."""
    return "exact" if case["kind"] in ("client", "ec") else {"rel": 1e-6, "max": 2e-5}
