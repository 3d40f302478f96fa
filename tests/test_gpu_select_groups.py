"""GPU parity of the selection over the ways its groups of rows are cut: runs of 16 rows (256 coordinates) spread over a client, in
groups of two runs in small batches and of eight in larger ones, the client's last rows and its ragged tail among them.  Nearly all
candidates lie in one layer, at the front, in the middle or at the end; few or many sub-buckets are summed up at a client's end."""
import numpy as np
import pytest

from gpu_util import gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n", [(17, 1), (255, 2), (256, 1), (257, 1), (511, 3), (513, 1), (4_096, 1), (36_867, 1), (40_960, 12),
                                 (360_000, 16), (5_762_049, 1), (5_800_003, 2)])
@pytest.mark.parametrize("layer", ["front", "middle", "end"])
def test_a_dense_layer_anywhere(d, n, layer):
    import torch
    from paper_2402_03770_b200 import binding as B
    rng = np.random.default_rng(d + n)
    dense = max(1, d // 24)
    at = {"front": 0, "middle": d // 2, "end": d - dense}[layer]
    packet_bits = 128 if d < 1_000 else 1024 if d < 100_000 else 12_000
    xs, pds = [], []
    for c in range(n):
        x = rng.standard_normal(d) * 1e-6
        # in one octave (one bin holds a sixteenth of them: many sub-buckets where there are many) or over several
        x[at:at + dense] = rng.choice([-1.0, 1.0], dense) * (rng.uniform(1.0, 2.0, dense) if c % 2 == 0 else rng.exponential(1.0, dense))
        xs.append(x.astype(np.float32))
        pds.append(params_dict(d, max(packet_bits, d), packet_bits=packet_bits, seed=c, client_id=c))
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd) for pd in pds], dev)
    outs = enc.compress([torch.from_numpy(x).to(dev) for x in xs], side_stream=torch.cuda.Stream(dev))
    assert enc.status() == B.CVLC_OK
    for x, pd, out in list(zip(xs, pds, outs))[:2]:
        assert np.array_equal(out.cpu().numpy(), oracle_plan_encode(x, pd)[1])
