"""One-kernel step beside rows that hold no key of the pair: the slots of the next pair (budgets
that are no multiple of 16) and the rows a longer prompt left behind.  Infinities and NaN in them
stay where they are."""
import pytest
import torch

pytestmark = pytest.mark.gpu

H, G, d = 2, 4, 128


def randn(shape, seed, device):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.randn(shape, generator=g).to(device, torch.bfloat16)


def make_cache(monkeypatch, b, B, D, name="KVPOP_FUSED_STEP"):
    from paper_2607_05061_gb300 import kvpop
    for n in ("KVPOP_FUSED_STEP", "KVPOP_SPLIT_STEP"):
        monkeypatch.delenv(n, raising=False)
    monkeypatch.setenv(name, "1")
    z = torch.zeros
    cache = kvpop.KVpopCache(b, H, G, d, B, D, 4, torch.bfloat16, z(H, 3 * d, 4), z(H, 4), z(H, 4), z(H))
    assert cache.fused_step == (name == "KVPOP_FUSED_STEP")
    return cache


def steps(cache, b, n, device):
    q, k, v = (randn((n, b, h * d), 9 + i, device) for i, h in enumerate((H * G, H, H)))
    out = torch.empty((n, b, H * G, d), device=device)
    for t in range(n):
        cache.step(q[t], k[t], v[t], out[t])
    cache.check()
    return out


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("B,D", [(129, 16), (40, 16), (24, 32), (72, 5)])
def test_another_sequence_is_not_finite(cuda_device, monkeypatch, B, D, bad):
    b, n = 5, B + D + 20
    cache = make_cache(monkeypatch, b, B, D)
    K, V, Q = (randn((b, h, n, d), 3 + i, cuda_device) for i, h in enumerate((H, H, H * G)))
    V[2] = bad
    cache.prefill(Q, K, V, [n] * b)
    out = steps(cache, b, 3, cuda_device)
    keep = [s for s in range(b) if s != 2]
    assert torch.isfinite(out[:, keep]).all()
    assert not torch.isfinite(out[:, 2]).all()
    cache.free()


@pytest.mark.parametrize("B,D", [(48, 16), (128, 32), (256, 128), (40, 16)])
@pytest.mark.parametrize("through_import", [False, True])
def test_a_longer_prompt_was_there(cuda_device, monkeypatch, B, D, through_import):
    """From lengths short of the window or the budget on, through the steps that fill the rows."""
    b, n, more = 4, B + D + 20, 40
    lengths = [0, 5, D + 3, B + D - 7]
    K, V, Q = (randn((b, h, n, d), 3 + i, cuda_device) for i, h in enumerate((H, H, H * G)))
    first = make_cache(monkeypatch, b, B, D, "KVPOP_SPLIT_STEP" if through_import else "KVPOP_FUSED_STEP")
    first.prefill(Q, K, torch.full_like(V, float("nan")), [n] * b)
    first.prefill(Q, K, V, lengths)
    cache = first
    if through_import:
        cache = make_cache(monkeypatch, b, B, D)
        cache.import_state(first.export_state())
    got = steps(cache, b, more, cuda_device)
    assert torch.isfinite(got).all()
    fresh = make_cache(monkeypatch, b, B, D)
    fresh.prefill(Q, K, V, lengths)
    # the same keys with the same weights: only the order in which a pair's parts meet may differ
    assert (got - steps(fresh, b, more, cuda_device)).abs().max() <= 1e-5
    for c in {id(c): c for c in (first, cache, fresh)}.values():
        c.free()
