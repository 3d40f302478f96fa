"""GPU parity of cvlc_compress_batch over where the length tuning runs: in the clusters of few small clients, beside a selection that leaves it SMs, behind a short selection of
many clients, ahead of a long one with the clients tuned each for itself or together, and on one stream.  Every second client's magnitudes
fall as a steep power law, whose tuning takes longer than its selection; both quantizers, fixed lengths, a client that is not finite
and a workspace for too few candidates."""
import numpy as np
import pytest

import oracle as O
from gpu_util import assert_plan_equal, gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu

SHAPES = [(100_003, 3),     # clusters, which tune in the same kernel
          (700_003, 3),     # room left
          (40_000, 33),     # behind
          (4_200_001, 33),  # ahead, one tuning per key, the threshold by the fit's kernel
          (3_150_001, 32),  # ahead, a tuning per client, the threshold by a kernel of its own
          (3_840_001, 29)]  # ahead, a tuning per client, the threshold by the histogram's last blocks


def updates(d):
    rng = np.random.default_rng(d)
    sign = rng.choice([-1.0, 1.0], d)
    return [rng.standard_normal(d).astype(np.float32), (sign * rng.permutation(np.arange(1, d + 1) ** -1.3)).astype(np.float32)]


def compress(xs, pds, n, side, fixed_y=0, max_candidates=0):
    """clients 0, 2, .. have the first update and its parameters, clients 1, 3, .. the second"""
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    dx = [torch.from_numpy(x).to(dev) for x in xs]
    enc = B.BatchEncoder([gpu_params(pds[c % 2]) for c in range(n - 1)] + [gpu_params(pds[-1])], dev, max_candidates)
    for out in enc.outs:
        out.fill_(0xAB)
    enc.compress([dx[c % 2] for c in range(n - 1)] + [dx[-1]], side_stream=torch.cuda.Stream(dev) if side else None, fixed_y=fixed_y)
    return enc


@pytest.mark.parametrize("quantizer,fixed_y", [(0, 0), (1, 0), (0, 6)])
@pytest.mark.parametrize("d,n", SHAPES)
def test_plans_and_streams_are_the_oracles(d, n, quantizer, fixed_y):
    import torch
    xs = updates(d)
    pds = [params_dict(d, d, quantizer=quantizer, seed=7 + i, client_id=i) for i in range(2)]
    xs, pds = xs + xs[:1], pds + pds[:1]  # the last client as the first one
    refs = [oracle_plan_encode(x, pd, fixed_y) for x, pd in zip(xs[:2], pds[:2])]
    streams = [torch.from_numpy(r[1]).to("cuda:0") for r in refs]
    for side in (True, False):
        enc = compress(xs, pds, n, side, fixed_y)
        assert enc.status() == O.ORC_OK
        for c in range(n):
            which = c % 2 if c < n - 1 else 0
            if not fixed_y:
                assert_plan_equal(enc.read_plan(c), refs[which][0])
            assert torch.equal(enc.outs[c], streams[which])


@pytest.mark.parametrize("d,n", SHAPES)
def test_a_refused_client_stops_the_call(d, n):
    from paper_2402_03770_b200 import binding as B
    xs = updates(d)
    xs.append(xs[0].copy())
    xs[2][d - 1] = np.nan
    pds = [params_dict(d, d, seed=i, client_id=i) for i in range(3)]
    for side in (True, False):
        enc = compress(xs, pds, n, side)
        assert enc.status() == O.ORC_ERR_NONFINITE_INPUT
        assert [enc.read_plan(c).status for c in (0, n - 1)] == [O.ORC_OK, O.ORC_ERR_NONFINITE_INPUT]
        enc = compress(xs[:2] + xs[:1], pds, n, side, max_candidates=1024)
        assert enc.status() == B.CVLC_ERR_WORKSPACE_TOO_SMALL
        assert enc.read_plan(n - 1).n_candidates > 1024
