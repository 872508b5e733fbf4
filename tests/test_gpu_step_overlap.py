"""The decode step whose attention streams beside its ingest, against the two calls one after
the other: bit for bit the same outputs, evictions and state, from an empty cache through the
step that fills it to replacements, after a prompt and after an import."""
import numpy as np
import pytest
import torch

from workload import gen

pytestmark = pytest.mark.gpu


def randn(shape, seed, device, dtype=torch.bfloat16):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.randn(shape, generator=g).to(device, dtype)


def same_state(a, b):
    for name in ("slotK", "slotV", "ringK", "ringV", "pos", "nvalid", "len", "mlstm_C", "mlstm_z", "mlstm_m"):
        assert name not in a or np.array_equal(a[name], b[name]), name
    B, D = a["slotK"].shape[1], a["ringK"].shape[1]
    for i, (nv, n) in enumerate(zip(a["nvalid"], a["len"])):   # what is not in use yet holds nothing
        assert np.array_equal(a["score"][i, :nv], b["score"][i, :nv])
        assert np.array_equal(a["ringQm"][i, :min(n, D)], b["ringQm"][i, :min(n, D)])
        for name in ("min_score", "min_slot", "blk_score", "blk_slot") if nv == B else ():
            assert np.array_equal(a[name][i], b[name][i]), name


# budgets at the edges of a 128-slot tile, windows below, at and above one
@pytest.mark.parametrize("batch,H,G,d,B,D,F,mlstm", [
    (1, 2, 4, 128, 127, 16, 32, False), (3, 2, 4, 128, 128, 128, 32, False),
    (17, 1, 1, 128, 129, 5, 16, False), (2, 3, 2, 64, 300, 130, 64, False),
    (5, 2, 4, 128, 64, 7, 260, False), (2, 8, 4, 128, 96, 12, 4, True), (1, 1, 4, 128, 2, 200, 8, False)])
def test_step_equals_ingest_then_attend(cuda_device, monkeypatch, batch, H, G, d, B, D, F, mlstm):
    from paper_2607_05061_gb300 import kvpop
    monkeypatch.delenv("KVPOP_FUSED_STEP", raising=False)
    monkeypatch.setenv("KVPOP_SPLIT_STEP", "1")
    if mlstm:
        from workload import get_config
        w = dict(mlstm=gen.mlstm_weights(get_config("q4b", batch=batch)))
    else:
        w = dict(zip(("W1", "b1", "w2", "b2"), (randn(s, 40 + i, "cpu", torch.float32) * 0.1 for i, s in enumerate(
            ((H, 3 * d, F), (H, F), (H, F), (H,))))))
    make = lambda: kvpop.KVpopCache(batch, H, G, d, B, D, F, torch.bfloat16, **w)
    a, b = make(), make()
    n = 40
    # prompts that leave a sequence a few tokens short of its budget, or of its window, or full
    P = B + D + 30
    lengths = [max(1, (B + D - 4, P, D, B + D)[i % 4]) for i in range(batch)] if batch > 1 else [B + D - 4]
    K, V, Q = (randn((batch, h, P, d), 7 + i, cuda_device) for i, h in enumerate((H, H, H * G)))
    for c in (a, b):
        c.prefill(Q, K, V, lengths)
    q, k, v = (randn((n, batch, h * d), 11 + i, cuda_device) for i, h in enumerate((H * G, H, H)))
    score = randn((n, batch, H), 17, cuda_device, torch.float32)

    def compare(a, b, lo, hi):
        oa, ob = (torch.empty((n, batch, H * G, d), device=cuda_device) for _ in range(2))
        ea, eb = (torch.empty((n, batch * H, 2), dtype=torch.int32, device=cuda_device) for _ in range(2))
        for t in range(lo, hi):          # every other step's evictions as the scorer has them
            ov = score[t] if t % 2 else None
            a.step(q[t], k[t], v[t], oa[t], override=ov, evict_info=ea[t])
        for t in range(lo, hi):
            ov = score[t] if t % 2 else None
            b.ingest(q[t], k[t], v[t], override=ov, evict_info=eb[t])
            b.attend(q[t], ob[t])
        a.check()
        b.check()
        assert torch.equal(ea[lo:hi], eb[lo:hi])
        assert torch.equal(oa[lo:hi], ob[lo:hi])
        blob = a.export_state()
        same_state(kvpop.parse_state(blob, a.cfg), kvpop.parse_state(b.export_state(), b.cfg))
        return blob
    blob = compare(a, b, 0, 25)
    c = make()
    c.import_state(blob)
    compare(c, b, 25, n)
    for x in (a, b, c):
        x.free()
