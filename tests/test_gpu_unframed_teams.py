"""GPU parity of the unframed writer where a thread block shares a block of records and where each of its warps has one: batches at
the line between the two, blocks of fewer records than a warp has lanes and of many, positions spread out and crowded."""
import numpy as np
import pytest

import oracle as O
from gpu_util import oracle_params, params_dict
from test_gpu_unframed import env, gpu_unframed  # noqa: F401  (env is a fixture)

pytestmark = pytest.mark.gpu

LINE = 12 * 148


@pytest.mark.parametrize("quantizer", [0, 1])
@pytest.mark.parametrize("crowded", [False, True])
@pytest.mark.parametrize("packet_bits,R,n,d", [
    (192, 5, 1, 30_011), (192, LINE + 3, 1, 60_011),             # a few records, no multiple of four blocks
    (320, 9, 1, 20_011), (352, 9, 1, 20_011), (576, 7, 1, 20_011), (640, 7, 1, 20_011),  # 14 to 35 records at the shortest length
    (1_024, LINE // 2, 2, 400_003), (1_024, LINE // 2 + 1, 2, 400_003),
    (4_096, LINE + 1, 1, 3_000_001), (9_600, 890, 2, 2_500_001), (9_600, 300, 1, 2_500_001)])
def test_blocks_of_records_at_the_line(env, packet_bits, R, n, d, crowded, quantizer):
    torch, B = env
    rng = np.random.default_rng(packet_bits + R + quantizer)
    xs = []
    for c in range(n):
        x = rng.laplace(0, 1e-3, d)
        if crowded:  # nearly everything that is sent lies in a few places, with gaps of all sizes
            x *= 1e-3
            x[d // 3:d // 3 + d // 8] *= 1e4
        xs.append(x.astype(np.float32))
    pds = [params_dict(d, R * packet_bits, packet_bits=packet_bits, quantizer=quantizer, seed=c + 5, client_id=c) for c in range(n)]
    status, got, _, _ = gpu_unframed(torch, B, xs, pds)
    assert status == 0
    for x, pd, out in zip(xs, pds, got):
        po = oracle_params(pd)
        ref = O.encode_unframed(x, po, O.plan(x, po))
        assert out.size == ref.size and np.array_equal(out, ref)
