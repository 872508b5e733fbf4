"""The decode stack's projection kernel at the edges of its sizes, against fp64 products."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def bf(shape, seed, device, scale=1.0):
    g = torch.Generator()
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g) * scale).to(device, torch.bfloat16)


def close(got, want):
    # the sums carry fp32 rounding (about 1e-6 of their size), then one rounding to bf16:
    # half a unit in the last place, 2^-9 relative; a second one where both round apart
    assert ((got.double() - want).abs() <= want.abs() * 2.0 ** -7 + 1e-4).all()


@pytest.mark.parametrize("M", [1, 7, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("K,nq,nkv", [(64, 64, 48), (640, 384, 128), (4096, 544, 64), (1152, 8192, 1024)])
def test_projections(cuda_device, M, K, nq, nkv):
    from paper_2607_05061_gb300 import kvpop
    assert kvpop.kvpop_project_supported(M, K, nq, nkv) == (3 if M <= 16 else 1)
    x = bf((M, K), 1, cuda_device)
    W = [bf((K, n), 2 + i, cuda_device, K ** -0.5) for i, n in enumerate((nq, nkv, nkv))]
    y = [torch.full((M + 1, n), 7.0, dtype=torch.bfloat16, device=cuda_device) for n in (nq, nkv, nkv)]
    kvpop.project_qkv(x, *W, *y)
    for w, t in zip(W, y):
        close(t[:M], x.double() @ w.double())
        assert (t[M] == 7.0).all()
    if M > 16:
        return
    o = torch.randn(M, nq, device=cuda_device)
    Wo, res = bf((nq, K), 9, cuda_device, nq ** -0.5), bf((M, K), 10, cuda_device)
    out = torch.empty_like(res)
    kvpop.project_out(o, Wo, res, out)
    prod = o.to(torch.bfloat16).double() @ Wo.double()
    # the product is rounded to bf16 before the sum is: an error of 2^-8 of the product more
    want = res.double() + prod
    assert ((out.double() - want).abs() <= want.abs() * 2.0 ** -7 + prod.abs() * 2.0 ** -7 + 1e-4).all()
    inplace = res.clone()
    kvpop.project_out(o, Wo, inplace, inplace)
    assert torch.equal(inplace, out)


def test_unsupported_sizes_are_refused(cuda_device):
    from paper_2607_05061_gb300 import kvpop
    for M, K, nq, nkv in ((33, 128, 128, 64), (1, 144, 128, 64), (1, 128, 100, 64), (1, 128, 128, 32),
                          (0, 128, 128, 64)):
        assert kvpop.kvpop_project_supported(M, K, nq, nkv) & 1 == 0
    assert kvpop.kvpop_project_supported(17, 128, 128, 64) == 1
    x, W = bf((1, 144), 1, cuda_device), bf((144, 128), 2, cuda_device)
    y = torch.empty((1, 128), dtype=torch.bfloat16, device=cuda_device)
    with pytest.raises(kvpop.KVpopError):
        kvpop.project_qkv(x, W, W, W, y, y, y)
