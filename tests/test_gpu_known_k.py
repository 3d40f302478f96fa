"""GPU parity where the selection starts from the bin that holds rank k (separate calls, whose plan is complete) against the
oracle: k at the edges of bins, in the top bin, equal to all candidates, single bins, hundreds of bins."""
import numpy as np
import pytest

from gpu_util import assert_plan_equal, gpu_plan_encode, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


def update(kind, d, rng):
    if kind == "laplace":
        return rng.laplace(0, 1e-3, d)
    if kind == "one_bin":                       # every magnitude in one histogram bin
        return rng.choice([-1.0, 1.0], d) * (1.0 + rng.random(d) / 64)
    if kind == "two_magnitudes":                # the threshold's bin and the top bin far apart
        return rng.choice([-1.0, 1.0], d) * np.where(np.arange(d) < d // 50, 1e3, 1e-3)
    if kind == "wide":                          # more bins than coarse buckets
        return rng.standard_normal(d) * 10.0 ** rng.uniform(-30, 30, d)
    steps = np.repeat(2.0 ** -np.arange(40), d // 40 + 1)[:d]   # bins of equal size, one in sixteen filled
    return rng.permutation(steps) * rng.choice([-1.0, 1.0], d)


@pytest.mark.parametrize("kind", ["laplace", "one_bin", "two_magnitudes", "wide", "steps"])
@pytest.mark.parametrize("d,packets,fixed_y", [(1_000, 1, 0), (40_000, 12, 0), (40_000, 12, 6), (300_001, 90, 0)])
def test_selection_from_the_bin_of_rank_k(kind, d, packets, fixed_y):
    x = update(kind, d, np.random.default_rng(d + packets)).astype(np.float32)
    pd = params_dict(d, packets * 4096, packet_bits=4096, seed=7)
    fields, stream = oracle_plan_encode(x, pd, fixed_y)
    status, plan, out = gpu_plan_encode(x, pd, fixed_y)
    assert status == 0
    if not fixed_y:
        assert_plan_equal(plan, fields)
    assert plan.k == fields["k"] <= plan.n_candidates
    assert np.array_equal(out, stream)
