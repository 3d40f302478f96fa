"""GPU parity of the selection over the ways its groups of rows are cut: runs of 16 rows (256 coordinates) spread over a client, in
groups of two runs in small batches and of eight in larger ones, the client's last rows and its ragged tail among them.  (Up to fifteen
small clients are selected by clusters; sixteen of the same sizes, and 700,003 coordinates, are not.)  Nearly all
candidates lie in one layer, at the front, in the middle or at the end; few or many sub-buckets are summed up at a client's end."""
import numpy as np
import pytest

from gpu_util import gpu_params, oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n", [(17, 1), (255, 2), (256, 1), (257, 1), (511, 3), (513, 1), (4_096, 1), (36_867, 1), (40_960, 12),
                                 (360_000, 16), (5_762_049, 1), (5_800_003, 2), (17, 16), (255, 17), (256, 16), (257, 16), (511, 18), (513, 16),
                                 (4_096, 16), (36_867, 16), (40_960, 17), (700_003, 1)])
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


@pytest.mark.parametrize("d,n,bits", [(11_800_003, 32, 1.0), (100_000_003, 10, 0.25)])
def test_groups_of_three_sizes(d, n, bits):
    """367 M coordinates and more in at most 32 clients: groups of many pieces, of a quarter as many and of single pieces, spread over a
    client each (8 and 2 pieces of 128 rows, or 21 and 5).  The clients are the same one, so that the oracle runs once."""
    import torch
    from paper_2402_03770_b200 import binding as B
    rng = np.random.default_rng(n)
    x = rng.standard_normal(d, dtype=np.float32)
    for q in range(16):  # layers of different scales, so that rows differ in how many candidates they hold
        x[q * d // 16:(q + 1) * d // 16] *= np.float32(10.0 ** -rng.uniform(0, 2))
    pd = params_dict(d, int(bits * d), seed=n)
    most = 3 * (int(bits * d) // 12_000) * ((12_000 - 80) // (int(d - 1).bit_length() + 1))
    dev = torch.device("cuda:0")
    enc = B.BatchEncoder([gpu_params(pd)] * n, dev, max_candidates=most)
    outs = enc.compress([torch.from_numpy(x).to(dev)] * n, side_stream=torch.cuda.Stream(dev))
    assert enc.status() == B.CVLC_OK
    stream = torch.from_numpy(oracle_plan_encode(x, pd)[1]).to(dev)
    for out in outs:
        assert torch.equal(out, stream)
