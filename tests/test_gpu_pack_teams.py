"""GPU parity of the packing where a block's four warps share a packet and where each has its own: batches at the line between the
two, packets of fewer records than a warp or a block has threads and of many, both quantizers."""
import numpy as np
import pytest

from gpu_util import gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu

SMS = 148


@pytest.mark.parametrize("quantizer,line", [(0, 13 * SMS), (1, 9 * SMS)])
@pytest.mark.parametrize("packet_bits,d", [(192, 30_011), (2_048, 400_003), (12_000, 1_500_001)])
@pytest.mark.parametrize("behind", [0, 1])
@pytest.mark.parametrize("n", [1, 4])
def test_packets_at_the_line(quantizer, line, packet_bits, d, behind, n):
    import torch
    from paper_2402_03770_b200 import binding as B
    R = line // n + behind
    rng = np.random.default_rng(d + n)
    xs = [(rng.laplace(0, 1e-3, d) * np.where(np.arange(d) < d // 3, 1.0, 20.0)).astype(np.float32) for _ in range(n)]
    pds = [params_dict(d, R * packet_bits, packet_bits=packet_bits, quantizer=quantizer, seed=c + 3, client_id=c) for c in range(n)]
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    outs = enc.compress([torch.from_numpy(x).to(dev) for x in xs])
    assert enc.status() == B.CVLC_OK
    for x, pd, out in list(zip(xs, pds, outs))[:2]:
        assert np.array_equal(out.cpu().numpy(), oracle_plan_encode(x, pd)[1])
