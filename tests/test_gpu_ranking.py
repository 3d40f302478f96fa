"""GPU parity of the ranking on value distributions at the edges of its buckets: buckets that need the partition, ties of all
sizes up to and beyond what a block holds, zeros among the candidates, mixed batches; plan and stream against the oracle, with the plan's workspace (partition) and without it (digit passes)."""
import numpy as np
import pytest

from gpu_util import assert_plan_equal, gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


def values(kind, d, rng):
    if kind == "narrow":                                    # every candidate in two or three bins: large coarse buckets
        return rng.choice([-1.0, 1.0], d) * (1.0 + 0.06 * rng.random(d))
    x = rng.laplace(0, 1e-3, d)
    if kind.startswith("ties"):                             # one value many times, in the middle of the candidates
        n = int(kind[4:])
        x[rng.choice(d, n, replace=False)] = np.quantile(np.abs(x), 0.97) * rng.choice([-1.0, 1.0], n)
    elif kind == "grid":
        x = np.round(x * 4096.0) / 4096.0
    elif kind == "near_ties":                               # neighbouring floats
        n = d // 20
        x[rng.choice(d, n, replace=False)] = np.float32(0.01) + np.arange(n) % 37 * np.float32(2.0 ** -30)
    elif kind == "wide":
        x = rng.standard_normal(d) * 10.0 ** rng.uniform(-30, 30, d)
    elif kind == "sparse":                                  # fewer values than are sent
        x[rng.random(d) < 0.97] = 0.0
    return x


@pytest.mark.parametrize("kind", ["laplace", "narrow", "ties900", "ties5000", "ties20000", "ties100000", "grid", "near_ties", "wide", "sparse"])
@pytest.mark.parametrize("d,bits", [(2_000_003, 3.0), (70_001, 2.0)])
def test_ranking_matches_the_oracle(kind, d, bits):
    import torch
    from paper_2402_03770_b200 import binding as B
    assert torch.cuda.is_available()
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(d + len(kind))
    if kind.startswith("ties") and int(kind[4:]) > d // 4:
        kind = f"ties{d // 4}"
    xs = [values(kind, d, rng).astype(np.float32), values("laplace", d, rng).astype(np.float32)]
    pds = [params_dict(d, int(bits * d), seed=5 + c, client_id=c) for c in range(2)]
    params = [gpu_params(pd) for pd in pds]
    refs = [oracle_plan_encode(x, pd) for x, pd in zip(xs, pds)]
    dxs = [torch.from_numpy(x).to(dev) for x in xs]
    enc = B.BatchEncoder(params, dev)
    for use_plan_ws in (True, False):
        for o in enc.outs:
            o.fill_(0x3C)
        outs = enc.run(dxs, use_plan_ws=use_plan_ws)
        assert enc.status() == 0
        for c, (fields, stream) in enumerate(refs):
            assert_plan_equal(enc.read_plan(c), fields)
            assert (outs[c].cpu().numpy() == stream).all(), (c, use_plan_ws)


@pytest.mark.parametrize("d", [40_960, 40_961, 40_975, 40_976, 43_007, 43_011])   # multiples of a row and of a warp's piece, and next to them
@pytest.mark.parametrize("bits", [0.5, 4.0])
def test_selection_at_the_edges_of_rows(d, bits):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(d)
    x = rng.laplace(0, 1e-3, d)
    x[d // 2:] *= np.where(rng.random(d - d // 2) < 0.02, 100.0, 0.01)      # a few candidates per step, then whole rows of them
    x[d // 4:d // 4 + 3000] = 0.2 + 0.001 * rng.standard_normal(3000)
    x[-1] = -0.9                                                            # the last coordinate of the last row
    xs = [x.astype(np.float32), np.ascontiguousarray(x[::-1]).astype(np.float32)]
    pds = [params_dict(d, int(bits * d), seed=9 + c, client_id=c) for c in range(2)]
    refs = [oracle_plan_encode(v, pd) for v, pd in zip(xs, pds)]
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    outs = enc.run([torch.from_numpy(v).to(dev) for v in xs], use_plan_ws=True)
    assert enc.status() == 0
    for c, (fields, stream) in enumerate(refs):
        assert_plan_equal(enc.read_plan(c), fields)
        assert (outs[c].cpu().numpy() == stream).all(), c


@pytest.mark.parametrize("n", [48, 49, 50, 256, 257, 290, 4000, 8191, 8193, 12000])   # limits of comparing, of a warp's cell, of a tile
@pytest.mark.parametrize("crowded", [False, True])                                    # indices next to one another
def test_equal_keys_among_others(n, crowded):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    d = 500_009
    rng = np.random.default_rng(n)
    x = rng.laplace(0, 1e-3, d).astype(np.float32)
    tie = np.quantile(np.abs(x), 0.95).astype(np.float32)
    where = np.arange(n) + 1234 if crowded else rng.choice(d, n, replace=False)
    x[where] = tie * rng.choice(np.float32([-1, 1]), n)
    near = rng.choice(d, 20, replace=False)                                           # neighbours of the repeated value
    x[near] = (np.full(20, tie).view(np.int32) + np.arange(-10, 10, dtype=np.int32)).view(np.float32)
    pd = params_dict(d, 3 * d, seed=3, client_id=0)
    fields, stream = oracle_plan_encode(x, pd)
    enc = B.BatchEncoder([gpu_params(pd)], dev)
    outs = enc.run([torch.from_numpy(x).to(dev)], use_plan_ws=True)
    assert enc.status() == 0
    assert_plan_equal(enc.read_plan(0), fields)
    assert (outs[0].cpu().numpy() == stream).all()


@pytest.mark.parametrize("n", [262_000, 300_000])
def test_very_large_buckets(n):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    d = 2_000_003
    rng = np.random.default_rng(n)
    x = values(f"ties{n}", d, rng).astype(np.float32)
    pd = params_dict(d, 6 * d, seed=4, client_id=0)
    fields, stream = oracle_plan_encode(x, pd)
    enc = B.BatchEncoder([gpu_params(pd)], dev)
    outs = enc.run([torch.from_numpy(x).to(dev)], use_plan_ws=True)
    assert enc.status() == 0
    assert_plan_equal(enc.read_plan(0), fields)
    assert (outs[0].cpu().numpy() == stream).all()


def test_large_bucket_found_while_blocks_still_start():
    """The first clients' selections find a very large bucket, while blocks behind the length tuning's (30 of them, one on an SM
    each) have yet to start and others are under way."""
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    d, n = 1_200_003, 30
    rng = np.random.default_rng(30)
    xs = [values("ties300000" if c < 2 else "laplace", d, rng).astype(np.float32) * np.float32(1 + c) for c in range(n)]
    pds = [params_dict(d, 6 * d, seed=6 + c, client_id=c) for c in range(n)]
    refs = {c: oracle_plan_encode(xs[c], pds[c]) for c in (0, 2, n - 1)}
    dxs = [torch.from_numpy(x).to(dev) for x in xs]
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    side = torch.cuda.Stream(dev)
    first = None
    for _ in range(10):
        for o in enc.outs:
            o.fill_(0x3C)
        outs = enc.compress(dxs, side_stream=side)
        assert enc.status() == 0
        if first is None:
            for c, (fields, stream) in refs.items():
                assert_plan_equal(enc.read_plan(c), fields)
                assert (outs[c].cpu().numpy() == stream).all(), c
            first = [o.clone() for o in outs]
        assert all(torch.equal(a, b) for a, b in zip(first, outs))


def _check(xs, pds, **kw):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    refs = [oracle_plan_encode(x, pd) for x, pd in zip(xs, pds)]
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev, **kw)
    outs = enc.run([torch.from_numpy(x).to(dev) for x in xs], use_plan_ws=True)
    assert enc.status() == 0
    for c, (fields, stream) in enumerate(refs):
        assert_plan_equal(enc.read_plan(c), fields)
        assert (outs[c].cpu().numpy() == stream).all(), c


# Buckets beyond a block (8192): one piece and the next, a few parts, several thousand items per part; equal keys spread over the
# update, in one stretch, in two far apart, and several keys of a bucket.
@pytest.mark.parametrize("n", [8192, 8193, 16_385, 24_577, 99_999, 450_000])
@pytest.mark.parametrize("where", ["spread", "stretch", "two", "keys"])
def test_buckets_beyond_a_block(n, where):
    d = 2_400_011
    rng = np.random.default_rng(n)
    x = rng.laplace(0, 1e-3, d).astype(np.float32)
    tie = np.quantile(np.abs(x), 0.8).astype(np.float32)
    if where == "stretch":
        at = d // 3 + np.arange(n)
    elif where == "two":
        at = np.concatenate([np.arange(n // 2), d - 1 - np.arange(n - n // 2)])
    else:
        at = rng.choice(d, n, replace=False)
    key = np.full(n, tie).view(np.int32) + (rng.integers(0, 5, n).astype(np.int32) if where == "keys" else np.int32(0))
    x[at] = key.view(np.float32) * rng.choice(np.float32([-1, 1]), n)
    other = rng.laplace(0, 1e-3, d).astype(np.float32)
    _check([x, other], [params_dict(d, 4 * d, seed=8 + c, client_id=c) for c in range(2)])


@pytest.mark.parametrize("kind", ["bf16", "steps", "signs"])
def test_updates_of_few_values(kind):
    """rounded to 16 bits, on a grid of steps, of one magnitude: every bucket is beyond a block"""
    d = 3_000_017
    rng = np.random.default_rng(len(kind))
    x = rng.standard_normal(d).astype(np.float32)
    if kind == "bf16":
        x = (x.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)
    elif kind == "steps":
        x = np.round(x * 8.0).astype(np.float32) / np.float32(8.0)
    else:
        x = np.sign(x) * np.float32(0.01)
    _check([x], [params_dict(d, 5 * d, seed=2, client_id=1)])


def test_bucket_of_two_rounds():
    """more than 1024 parts that a block can hold: 9.5 M values of one magnitude"""
    d = 9_500_003
    rng = np.random.default_rng(95)
    x = rng.choice(np.float32([-0.25, 0.25]), d)
    _check([x], [params_dict(d, d // 2, seed=2, client_id=1)])


# More coordinates are sent than are not zero: zeros of both signs are ranked behind the rest by their indices, subnormals before
# them; the update's last row and the rows of a warp's step need not be whole.
@pytest.mark.parametrize("d", [63, 64, 65, 1000, 40_961, 40_975, 300_003])
@pytest.mark.parametrize("kind", ["zeros", "few", "subnormal"])
def test_zeros_among_the_candidates(d, kind):
    rng = np.random.default_rng(d)
    xs = []
    for c in range(3):
        x = rng.laplace(0, 1e-3, d).astype(np.float32)
        x[rng.random(d) < (1.0 if kind == "zeros" else 0.99)] = 0.0
        if kind == "subnormal":
            at = rng.random(d) < 0.3
            x[at] = rng.integers(1, 1 << 19, int(at.sum())).astype(np.uint32).view(np.float32)
        x[rng.random(d) < 0.5] *= np.float32(-1.0)
        xs.append(x)
    xs.append(rng.laplace(0, 1e-3, d).astype(np.float32))       # a client of the same batch without zeros
    bits = 12000 if d > 2000 else 32 * 47
    _check(xs, [params_dict(d, max(bits, 2 * d), packet_bits=bits, seed=3 + c, client_id=c) for c in range(4)])


def test_counts_beyond_whole_numbers_of_fp32():
    """17.3 M values of one magnitude in one bin: the sub-buckets are counted in whole numbers"""
    d = 17_300_001
    rng = np.random.default_rng(173)
    x = rng.choice(np.float32([-0.25, 0.25]), d)
    x[::1000] = 0.0
    _check([x], [params_dict(d, d // 8, seed=2, client_id=1)])
