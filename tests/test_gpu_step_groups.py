"""The one-kernel step with one, two and four query heads per KV head, against the two kernels, from a
short prompt through the steps that fill the cache to replacements."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("b,H,B,D", [(3, 1, 48, 16), (17, 3, 130, 9)])
def test_one_kernel_equals_two(cuda_device, monkeypatch, G, b, H, B, D):
    from paper_2607_05061_gb300 import kvpop
    d, F, P, n = 128, 32, B + D - 5, 30
    g = torch.Generator()
    g.manual_seed(G + b)
    rn = lambda *s: torch.randn(s, generator=g)  # noqa: E731
    W = dict(W1=rn(H, 3 * d, F) * 0.1, b1=rn(H, F) * 0.1, w2=rn(H, F) * 0.1, b2=rn(H))
    K, V, Q = (rn(b, h, P, d).to(cuda_device, torch.bfloat16) for h in (H, H, H * G))
    q, k, v = (rn(n, b, h, d).to(cuda_device, torch.bfloat16) for h in (H * G, H, H))
    score = rn(n, b, H).to(cuda_device)                      # the same evictions on both sides
    outs, evicted = [], []
    for name, other in (("KVPOP_FUSED_STEP", "KVPOP_SPLIT_STEP"), ("KVPOP_SPLIT_STEP", "KVPOP_FUSED_STEP")):
        monkeypatch.delenv(other, raising=False)
        monkeypatch.setenv(name, "1")
        cache = kvpop.KVpopCache(b, H, G, d, B, D, F, torch.bfloat16, **W)
        assert cache.fused_step == (name == "KVPOP_FUSED_STEP")
        cache.prefill(Q, K, V, [P] * b)
        out = torch.empty((n, b, H * G, d), device=cuda_device)
        ev = torch.empty((n, b, H, 2), dtype=torch.int32, device=cuda_device)
        for t in range(n):
            cache.step(q[t], k[t], v[t], out[t], override=score[t], evict_info=ev[t])
        cache.check()
        outs.append(out)
        evicted.append(ev)
        cache.free()
    assert torch.equal(*evicted)
    # the tokens that change are added in fp32 on one side, with weights rounded to bf16 on the other
    assert (outs[0] - outs[1]).abs().max() <= 2e-2
