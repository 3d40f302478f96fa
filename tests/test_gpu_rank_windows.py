"""GPU parity of the ranking over the sizes of its tiles: candidates that make one round of the blocks or a little more, from the
smallest tile (1024) to the largest (4096), one client and several of different sizes; the window is whatever makes whole rounds.  (One client of
one packet is ranked by a cluster, sixteen are not.)"""
import numpy as np
import pytest

from gpu_util import gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R", [(1, 1), (16, 1), (1, 620), (1, 700), (1, 1_500), (1, 2_400), (1, 2_700), (3, 260), (20, 41)])
@pytest.mark.parametrize("side", [False, True])
def test_tiles_of_any_size(n, R, side):
    import torch
    from paper_2402_03770_b200 import binding as B
    rng = np.random.default_rng(R)
    d = max(4_000, 620 * R)                       # a packet of 12,000 bits sends about 400 coordinates
    xs, pds = [], []
    for c in range(n):
        x = rng.laplace(0, 1e-3, d)
        x[: d // (c + 2)] *= 10.0 ** rng.uniform(-2, 2)
        xs.append(x.astype(np.float32))
        pds.append(params_dict(d, R * 12_000, seed=c, client_id=c, scale_B=[None, 1.3, 2.0][c % 3]))
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    outs = enc.compress([torch.from_numpy(x).to(dev) for x in xs], side_stream=torch.cuda.Stream(dev) if side else None)
    assert enc.status() == B.CVLC_OK
    for x, pd, out in list(zip(xs, pds, outs))[:3]:
        assert np.array_equal(out.cpu().numpy(), oracle_plan_encode(x, pd)[1])
