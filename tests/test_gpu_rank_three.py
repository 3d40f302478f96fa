"""Partition and ranking with three blocks per SM (batches of 4 M records and more) against the digit passes (the encoder without the plan's
workspace, pinned to the oracle): tiles of smaller windows, buckets about as large as what a block holds, cells and buckets beyond it."""
import pytest

from gpu_util import gpu_params, params_dict

pytestmark = pytest.mark.gpu


def update(kind, d, gen, dev):
    import torch
    x = torch.randn(d, generator=gen, device=dev)
    at = torch.arange(d, device=dev)
    if kind == "layers":
        return x * torch.pow(10.0, -3.0 * torch.rand(32, generator=gen, device=dev))[at * 32 // d]
    if kind == "grid":
        return torch.round(x * 24.0) / 24.0
    if kind == "narrow":  # the candidates in one bin: sub-buckets of thousands
        return torch.where(torch.rand(d, generator=gen, device=dev) < 0.15, x.sign() * (1.0 + 0.03 * torch.rand(d, generator=gen, device=dev)), x * 1e-3)
    if kind == "outliers":  # equal keys at the top
        return torch.where(torch.rand(d, generator=gen, device=dev) < 1e-3, x.sign() * 50.0, x)
    return x


@pytest.mark.parametrize("kind", ["normal", "layers", "grid", "narrow", "outliers"])
@pytest.mark.parametrize("d,n,bits", [(1_200_003, 20, 4.0), (300_002, 80, 4.0)])
def test_streams(kind, d, n, bits):
    import torch
    from paper_2402_03770_b200 import binding as B
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(d)
    xs = [update(kind, d, gen, dev) for _ in range(n)]
    params = [gpu_params(params_dict(d, int(bits * d), seed=c, client_id=c)) for c in range(n)]
    enc = B.BatchEncoder(params, dev)
    assert n * (params[0].budget_bits // 12000) * (11920 // (int(d - 1).bit_length() + 1)) >= 4 << 20
    enc.plan(xs)
    want = [o.clone() for o in enc.encode(xs, use_plan_ws=False)]
    assert enc.status() == B.CVLC_OK
    for o in enc.outs:
        o.zero_()
    got = enc.compress(xs, side_stream=torch.cuda.Stream(dev))
    assert enc.status() == B.CVLC_OK
    for i in range(n):
        assert torch.equal(got[i], want[i]), i
