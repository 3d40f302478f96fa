"""GPU parity of the length tuning over exponents, sizes and budgets: the operations that concavity settles and those
left to the series arithmetic (steep power laws, whose differences drown in rounding; budgets that could send more than
d coordinates) must give the oracle's plan to the bit."""
import numpy as np
import pytest

import oracle as O
from gpu_util import assert_plan_equal, gpu_params, oracle_params, params_dict

pytestmark = pytest.mark.gpu

ALPHAS = [-0.004, -0.06, -0.2, -0.35, -0.45, -0.492, -0.4999, -0.508, -0.54, -0.7, -1.0, -1.3, -1.8, -2.5, -4.0]


def power_law_histogram(d, alpha):
    """4096-bin histogram of d magnitudes l^alpha (l = 1 .. d), straight from the survival function"""
    edges = np.minimum(np.arange(4096, dtype=np.uint32), 4080) << np.uint32(19)
    lower = edges.view(np.float32).astype(np.float64)
    with np.errstate(divide="ignore", over="ignore", invalid="ignore"):
        rank = np.where(lower > 0, lower ** (1.0 / alpha), np.inf)         # ranks whose magnitude reaches the bin's edge
    survivors = np.floor(np.minimum(np.nan_to_num(rank, nan=0.0, posinf=d), d)).astype(np.int64)
    survivors[0] = d
    survivors[4080:] = 0
    return survivors - np.append(survivors[1:], 0)


@pytest.mark.parametrize("quantizer", [0, 1])
@pytest.mark.parametrize("d,packets", [(2_000, 1), (2_000, 5), (60_001, 40), (300_000, 10), (11_200_000, 1866),
                                       (100_000_000, 33_333), (2 ** 31, 300_000)])
def test_tuned_lengths_match_the_oracle(d, packets, quantizer):
    import torch
    from paper_2402_03770_b200 import binding as B
    assert torch.cuda.is_available()
    dev = torch.device("cuda:0")
    pds, hists = [], []
    for i, alpha in enumerate(ALPHAS):
        for scale in (None, 1.5):
            pds.append(params_dict(d, packets * 12000, quantizer=quantizer, client_id=i, scale_B=scale))
            hists.append(power_law_histogram(d, alpha))
    params = [gpu_params(pd) for pd in pds]
    plans = torch.zeros(len(pds) * B.PLAN_BYTES, dtype=torch.uint8, device=dev)
    ws = B.alloc_bytes(B.cvlc_plan_batch_workspace_bytes(params[0], len(pds)), dev)
    hist = torch.from_numpy(np.stack(hists)).to(dev)
    B.cvlc_plan_from_histogram_batch(hist, params, plans, ws)
    assert B.cvlc_read_status(ws) == 0
    for i, pd in enumerate(pds):
        ref = O.plan_from_histogram(hists[i].astype(np.uint64), oracle_params(pd))
        got = B.read_plan(plans[i * B.PLAN_BYTES:(i + 1) * B.PLAN_BYTES])
        fields = {f: getattr(ref, f) for f in ("s", "R", "y_min", "n_lengths", "k", "alpha", "alpha_q", "beta", "gamma", "B_next")}
        fields["n_y"] = [ref.n_y[y] for y in range(33)]
        fields["cap"] = [ref.cap[y] for y in range(33)]
        assert_plan_equal(got, fields)
