"""GPU parity of the planning front over the ways a batch can be cut: chunks of one client each, whose last block finishes the
client, or chunks of the concatenated clients; exponent fit and tuning per client or shared by clients of one key; with and without a
side stream.  Up to fifteen such small clients are planned by clusters in these calls, so the planning call is checked as well, and
sixteen clients of the same sizes.  Sizes at the edges of rows (16 coordinates) and chunks (256 rows); clients with different scales, so that their
shortest lengths differ."""
import numpy as np
import pytest

import oracle as O
from gpu_util import assert_plan_equal, gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu

SCALES = [None, 1.3, 1.3, 2.0, 1.0]


def make_batch(d, n, seed, bits=2.0, packet_bits=1024):
    rng = np.random.default_rng(seed)
    xs, pds = [], []
    for c in range(n):
        scale = 10.0 ** rng.uniform(-4, -2, 4).astype(np.float32)
        xs.append((rng.laplace(0, 1, d) * scale[np.arange(d) * 4 // d]).astype(np.float32))
        pds.append(params_dict(d, max(packet_bits, int(bits * d)), packet_bits=packet_bits, seed=seed + c, client_id=c,
                               scale_B=SCALES[c % len(SCALES)]))
    return xs, pds


def run_batch(xs, pds, side):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    outs = enc.compress([torch.from_numpy(x).to(dev) for x in xs], side_stream=torch.cuda.Stream(dev) if side else None)
    status = enc.status()
    plans = [B.read_plan(enc.plans[i * B.PLAN_BYTES:(i + 1) * B.PLAN_BYTES]) for i in range(len(xs))]
    return status, plans, [o.cpu().numpy() for o in outs]


def plan_batch(xs, pds):
    import torch
    from paper_2402_03770_b200 import binding as B
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], torch.device("cuda:0"))
    enc.plan([torch.from_numpy(x).to("cuda:0") for x in xs])
    return [enc.read_plan(i) for i in range(len(xs))]


@pytest.mark.parametrize("d,n", [(200, 1), (255, 5), (4095, 1), (4096, 3), (4097, 1), (8193, 2), (20_000, 11), (3_000, 33), (2_000, 148),
                                 (1_500, 149), (400, 400), (100_003, 3), (200, 16), (255, 17), (4095, 16), (4096, 18), (4097, 16), (8193, 17), (700_003, 1)])
def test_every_cut_gives_the_oracles_plan_and_stream(d, n):
    xs, pds = make_batch(d, n, seed=d + n)
    refs = [oracle_plan_encode(x, pd) for x, pd in zip(xs, pds)]
    for side in (False, True):
        status, plans, outs = run_batch(xs, pds, side)
        assert status == 0
        for (fields, stream), plan, out in zip(refs, plans, outs):
            assert_plan_equal(plan, fields)
            assert np.array_equal(out, stream)
    for (fields, _), plan in zip(refs, plan_batch(xs, pds)):
        assert_plan_equal(plan, fields)


@pytest.mark.parametrize("n,bad", [(1, 0), (4, 3), (16, 9), (40, 17), (149, 148)])
def test_non_finite_client_stops_the_batch_and_keeps_the_others_plans(n, bad):
    xs, pds = make_batch(1_777, n, seed=n)
    xs[bad][1_776] = np.inf
    for side in (False, True):
        status, plans, _ = run_batch(xs, pds, side)
        assert status == O.ORC_ERR_NONFINITE_INPUT
        for c, plan in enumerate(plans):
            if c == bad:
                assert plan.status == O.ORC_ERR_NONFINITE_INPUT
            else:
                assert_plan_equal(plan, oracle_plan_encode(xs[c], pds[c])[0])
    assert [plan.status for plan in plan_batch(xs, pds)] == [O.ORC_ERR_NONFINITE_INPUT if c == bad else O.ORC_OK for c in range(n)]
