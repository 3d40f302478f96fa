"""GPU parity of cvlc_compress_batch where a cluster of blocks per client plans, selects and ranks: at most 15 clients of up to 327,683
coordinates (eight blocks), at most 7 of 245,764 to 655,363 (sixteen).  Sizes around its limits, its blocks' shares (rows of 16
coordinates, a seventh or a fifteenth each, a ragged tail with the last) and what a block keeps of one (40,960 coordinates), and updates whose candidates crowd into bins that a block cannot hold."""
import numpy as np
import pytest

from gpu_util import gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


def update(kind, d, rng):
    x = rng.standard_normal(d)
    if kind == "layers":
        x *= np.repeat(10.0 ** rng.uniform(-3, 0, 9), d // 9 + 1)[:d]
    elif kind == "equal":  # more equal magnitudes than a block holds, most of them sent
        x = np.where(rng.random(d) < 0.15, np.sign(x) * 3.0, x)
    elif kind == "grid":
        x = np.round(x * 8.0) / 8.0
    elif kind == "zeros":  # fewer that are not zero than are sent
        x[rng.random(d) < 0.999] = 0.0
    elif kind == "signs":
        x = np.sign(x)
    elif kind == "narrow":  # all candidates in one bin of the histogram, a few thousand in each range of it
        x = np.where(rng.random(d) < 0.12, np.sign(x) * rng.uniform(1.0, 1.04, d), x * 1e-3)
    elif kind == "steps":  # ... and on eight values of it
        x = np.where(rng.random(d) < 0.12, np.sign(x) * (1.0 + rng.integers(0, 8, d) / 256.0), x * 1e-3)
    elif kind == "front":  # all candidates in the first block's slice
        x[d // 12:] *= 1e-6
    return x.astype(np.float32)


def check(xs, pds, side, fixed_y=0, checked=3):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    before = B.cvlc_launch_count("k_client")
    outs = enc.compress([torch.from_numpy(x).to(dev) for x in xs], side_stream=torch.cuda.Stream(dev) if side else None, fixed_y=fixed_y)
    assert enc.status() == B.CVLC_OK
    for i in list(range(len(xs)))[-checked:]:
        want = oracle_plan_encode(xs[i], pds[i], fixed_y)
        assert enc.read_plan(i).k == want[0]["k"]
        assert np.array_equal(outs[i].cpu().numpy(), want[1]), i
    return B.cvlc_launch_count("k_client") - before


@pytest.mark.parametrize("d,n", [(2, 1), (5, 2), (127, 1), (129, 3), (2_047, 15), (40_961, 5), (100_003, 1), (300_000, 3), (245_763, 7), (245_764, 7), (327_680, 8), (327_683, 1),
                                 (400_001, 3), (655_363, 7),
                                 (286_720, 8), (286_833, 9), (614_400, 1), (614_465, 1)])
@pytest.mark.parametrize("side", [False, True])
def test_sizes(d, n, side):
    rng = np.random.default_rng(d)
    packet_bits = 128 if d < 1_000 else 1024 if d < 100_000 else 12_000
    pds = [params_dict(d, max(packet_bits, d // 2), packet_bits=packet_bits, seed=c, client_id=c, quantizer=c % 2 if n == 1 else 0) for c in range(n)]
    assert check([update("layers", d, rng) for _ in range(n)], pds, side) == 1


def test_limits():
    rng = np.random.default_rng(0)
    for d, n, bits in [(327_684, 8, 0.3), (655_364, 1, 0.3), (4_000, 16, 0.5), (655_000, 1, 5.0)]:  # coordinates, clients, candidates: the kernels of their own
        pds = [params_dict(d, int(bits * d), seed=c, packet_bits=1024) for c in range(n)]
        assert check([update("normal", d, rng) for _ in range(n)], pds, True, checked=2) == 0


@pytest.mark.parametrize("side", [False, True])
def test_the_limit_holds_for_every_client(side):
    """Clients whose scales differ may send different numbers of records: the call takes clusters only if all of them may send up to
    65,536, whichever stands first."""
    d = 320_001
    rng = np.random.default_rng(7)
    xs = [update("layers", d, rng) for _ in range(3)]
    # 130 packets; shortest lengths of 5 bits (130 * 496 records) and of 2 (130 * 567, beyond the limit)
    few, many = (params_dict(d, 130 * 12_000, seed=c, scale_B=scale) for c, scale in ((1, None), (2, 100.0)))
    assert check(xs, [few] * 3, side) == 1
    assert check(xs, [many] * 3, side) == 0
    assert check(xs, [few, many, few], side) == 0
    assert check(xs, [many, few, few], side) == 0


@pytest.mark.parametrize("kind", ["normal", "equal", "grid", "zeros", "signs", "front", "narrow", "steps"])
@pytest.mark.parametrize("quantizer", [0, 1])
@pytest.mark.parametrize("d,n,bits", [(200_003, 4, 2.0), (327_001, 3, 4.0), (600_001, 2, 2.5)])
def test_distributions(kind, quantizer, d, n, bits):
    rng = np.random.default_rng(3)
    pds = [params_dict(d, int(bits * d), seed=c, client_id=c, quantizer=quantizer) for c in range(n)]
    assert check([update(kind if c % 2 == 0 else "layers", d, rng) for c in range(n)], pds, True, checked=2) == 1


def in_one_bin(m, values, d, rng):
    """m coordinates at scattered places whose keys are 1.0 and the next `values` ones, as evenly as can be; the others a thousand times smaller"""
    x = rng.standard_normal(d).astype(np.float32) * np.float32(1e-3)
    low = rng.permutation(1 << 19)[:m] if values == 1 << 19 else np.arange(m) % values
    at = rng.permutation(d)[:m]
    x[at] = (0x3F800000 + low.astype(np.uint32)).astype(np.uint32).view(np.float32) * np.where(rng.random(m) < 0.5, -1.0, 1.0).astype(np.float32)
    return x


# all different: one cut, where a bin has more than 9216 (up to that many of one key are left to k_rank_rest); 512 neighbouring keys: parts of one cut that are cut again; two and one: by coordinates
@pytest.mark.parametrize("values", [1 << 19, 512, 2, 1])
@pytest.mark.parametrize("m", [8_192, 8_193, 9_216, 9_217, 12_000, 16_384, 16_385, 33_000])
@pytest.mark.parametrize("d,n", [(200_003, 2), (600_001, 1)])
def test_bins_that_a_block_does_not_hold(values, m, d, n):
    """what is sent ends inside the bin and behind it"""
    rng = np.random.default_rng(m + values)
    xs = [in_one_bin(m, values, d, rng) for _ in range(n)]
    for sent in (m * 3 // 5, min(64_000, m + 9_000)):
        pds = [params_dict(d, 12_000 * (sent // 530 + 1), seed=c, client_id=c) for c in range(n)]
        assert check(xs, pds, True) == 1


def test_as_many_bins_as_can_be_too_large():
    """Seven bins of 8193 and more, one after the other and with others between, and one that is sent in part; a bin with seven such parts;
    values next to one another where every cut leaves some too large"""
    rng = np.random.default_rng(8)
    d = 640_003
    pd = params_dict(d, 12_000 * 137, seed=1)  # 65,212 records
    x = rng.standard_normal(d).astype(np.float32) * np.float32(1e-4)
    at = rng.permutation(d)[:80_000]
    x[at] = (1.0 + (np.arange(80_000) // 8_200) / 16 + rng.random(80_000) / 17).astype(np.float32)
    assert check([x], [pd], True) == 1
    x[at] = (2.0 ** (np.arange(80_000) // 8_200) + rng.random(80_000) / 17).astype(np.float32)
    assert check([x], [pd], False) == 1
    x[at] = (0x3F800000 + (np.arange(80_000) // 8_200 * 2048).astype(np.uint32) + rng.integers(0, 512, 80_000).astype(np.uint32)).astype(np.uint32).view(np.float32)
    assert check([x], [pd], True) == 1
    x[at] = (0x3F800000 + (np.arange(80_000) // 20_000 * 1023).astype(np.uint32)).astype(np.uint32).view(np.float32)
    assert check([x], [pd], True) == 1


def test_fixed_length():
    rng = np.random.default_rng(4)
    assert check([update("layers", 150_001, rng)], [params_dict(150_001, 150_001)], False, fixed_y=5) == 1
    assert check([in_one_bin(20_000, 3, 150_001, rng)], [params_dict(150_001, 360_000)], False, fixed_y=5) == 1


def test_errors():
    """Inf in one client; a workspace for fewer candidates than there are: reported, and the buffers serve the next call"""
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(5)
    d, n = 50_001, 3
    pds = [params_dict(d, d, seed=c) for c in range(n)]
    xs = [torch.from_numpy(update("normal", d, rng)).to(dev) for _ in range(n)]
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    bad = xs[1].clone()
    bad[d - 1] = float("inf")
    before = B.cvlc_launch_count("k_client")
    enc.compress([xs[0], bad, xs[2]])
    assert enc.status() == B.CVLC_ERR_NONFINITE_INPUT
    outs = enc.compress(xs)
    assert enc.status() == B.CVLC_OK
    assert np.array_equal(outs[2].cpu().numpy(), oracle_plan_encode(xs[2].cpu().numpy(), pds[2])[1])
    small = B.BatchEncoder([gpu_params(pd) for pd in pds], dev, max_candidates=256)
    small.compress(xs)
    assert small.status() == B.CVLC_ERR_WORKSPACE_TOO_SMALL
    crowded = [torch.from_numpy(update("signs", d, rng)).to(dev)] * n  # bins that would be cut
    small.compress(crowded)
    assert small.status() == B.CVLC_ERR_WORKSPACE_TOO_SMALL
    assert B.cvlc_launch_count("k_client") == before + 4


def test_plan_workspace_serves_the_encoder():
    """the plan's tables that a compress call leaves are those of a plan call"""
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(6)
    d, n = 120_005, 2
    pds = [params_dict(d, d, seed=c) for c in range(n)]
    xs = [torch.from_numpy(update("layers", d, rng)).to(dev) for _ in range(n)]
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    before = B.cvlc_launch_count("k_client")
    want = [o.clone() for o in enc.compress(xs)]
    assert B.cvlc_launch_count("k_client") == before + 1
    for o in enc.outs:
        o.zero_()
    got = enc.encode(xs)
    assert enc.status() == B.CVLC_OK
    for a, b in zip(want, got):
        assert torch.equal(a, b)
