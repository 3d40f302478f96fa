"""GPU parity of the ranking where the candidates crowd at one end of few histogram bins, as the memories of error compensation do
below the threshold after some rounds: by separate calls, and by cvlc_compress_batch, which ranks the smaller two by clusters."""
import numpy as np
import pytest

from gpu_util import gpu_plan_encode, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,R", [(40_000, 30), (300_000, 90), (1_200_000, 200)])
@pytest.mark.parametrize("bins", [1, 3, 40, 200])
@pytest.mark.parametrize("end", ["low", "high"])
def test_candidates_at_one_end_of_their_bins(d, R, bins, end):
    rng = np.random.default_rng(d + bins)
    x = rng.standard_normal(d) * 1e-9
    k = min(d, R * 560)                                           # about what may be sent
    top = 2.0 ** (np.sort(rng.integers(0, bins, k)) / 16 // 1) * (1 + rng.integers(0, min(bins, 16), k) / 16)   # lower ends of bins
    part = rng.random(k) / 16 / 4096
    x[rng.permutation(d)[:k]] = np.where(end == "low", top + top * part, top + 0.0624 - part) * rng.choice([-1.0, 1.0], k)
    x = x.astype(np.float32)
    pd = params_dict(d, R * 12_000, seed=bins)
    ref = oracle_plan_encode(x, pd)[1]
    for compress in (0, 2):
        status, _, out = gpu_plan_encode(x, pd, compress=compress)
        assert status == 0
        assert np.array_equal(out, ref)
