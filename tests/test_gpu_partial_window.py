"""Decode attention over windows that fill no whole 16-key group, with NaN left in shared memory
by an earlier kernel: what lies past the last key must not reach the sums."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def randn(shape, seed, device, dtype):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.randn(shape, generator=g).to(device, dtype)


@pytest.mark.parametrize("dtype,tol", [(torch.bfloat16, 1e-2), (torch.float32, 1e-5)])
@pytest.mark.parametrize("B,D,n", [(16, 1, 40), (8, 3, 40), (129, 5, 150), (40, 9, 45), (20, 17, 90), (33, 13, 12)])
@pytest.mark.parametrize("d", [64, 128])
def test_nothing_past_the_last_key(cuda_device, dtype, tol, B, D, n, d):
    from paper_2607_05061_gb300 import kvpop
    b, H, G = 17, 2, 4
    z = torch.zeros
    cache = kvpop.KVpopCache(b, H, G, d, B, D, 4, dtype, z(H, 3 * d, 4), z(H, 4), z(H, 4), z(H))
    K, V, Q = (randn((b, h, n, d), 3 + i, cuda_device, dtype) for i, h in enumerate((H, H, H * G)))
    cache.prefill(Q, K, V, [n] * b)
    nan = torch.full((2048, 2048), float("nan"), dtype=torch.bfloat16, device=cuda_device)
    q = randn((b, H * G * d), 9, cuda_device, dtype)
    out = torch.empty((b, H * G, d), device=cuda_device)
    torch.matmul(nan, nan)
    cache.attend(q, out)
    cache.check()
    # every score is 0: the first B tokens that have left the window are kept, ties to the lower
    for s in (0, b - 1):
        for h in range(H):
            pos, _ = cache.pair_state(s, h)
            keys = sorted(pos) + list(range(max(0, n - D), n))
            k, v = K[s, h, keys].double(), V[s, h, keys].double()
            for g in range(G):
                w = torch.softmax(k @ q.view(b, H * G, d)[s, h * G + g].double() / d ** 0.5, 0)
                # probabilities rounded to bf16: 2^-9 of values of size 1, summed with weights of 1
                assert (out[s, h * G + g].double() - w @ v).abs().max() <= tol
    assert torch.isfinite(out).all()
    cache.free()


@pytest.mark.parametrize("D,B,n", [(5, 40, 60), (17, 129, 200), (16, 40, 60), (16, 40, 50)])
def test_one_kernel_step_past_the_last_key(cuda_device, monkeypatch, D, B, n):
    """The one-kernel step over the same: finite, and equal to the two kernels within the
    rounding of the probabilities."""
    from paper_2607_05061_gb300 import kvpop
    b, H, G, d = 9, 2, 4, 128
    z = torch.zeros
    K, V, Q = (randn((b, h, n, d), 3 + i, cuda_device, torch.bfloat16) for i, h in enumerate((H, H, H * G)))
    q, k, v = (randn((b, h * d), 9 + i, cuda_device, torch.bfloat16) for i, h in enumerate((H * G, H, H)))
    nan = torch.full((2048, 2048), float("nan"), dtype=torch.bfloat16, device=cuda_device)
    outs = []
    for name, other in (("KVPOP_FUSED_STEP", "KVPOP_SPLIT_STEP"), ("KVPOP_SPLIT_STEP", "KVPOP_FUSED_STEP")):
        monkeypatch.delenv(other, raising=False)
        monkeypatch.setenv(name, "1")
        cache = kvpop.KVpopCache(b, H, G, d, B, D, 4, torch.bfloat16, z(H, 3 * d, 4), z(H, 4), z(H, 4), z(H))
        assert kvpop.kvpop_step_is_fused(cache.handle) == (name == "KVPOP_FUSED_STEP")
        cache.prefill(Q, K, V, [n] * b)
        out = torch.empty((b, H * G, d), device=cuda_device)
        torch.matmul(nan, nan)
        cache.step(q, k, v, out)
        cache.check()
        outs.append(out)
        cache.free()
    assert torch.isfinite(outs[0]).all()
    assert (outs[0] - outs[1]).abs().max() <= 1e-2
