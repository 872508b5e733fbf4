"""Ranks, cutoffs and the top-B selection of a prompt at the sizes where their split over the
CTAs of a cluster, their items per thread and their last partial chunk change."""
import numpy as np
import pytest
import torch

from oracle import running_topk as rt
from workload import gen

pytestmark = pytest.mark.gpu


def kv():
    from paper_2607_05061_gb300 import kvpop
    return kvpop


@pytest.mark.parametrize("rows,S,levels", [
    (1, 1, None), (1, 513, 3), (1, 1024, None), (3, 2049, 40), (1, 4097, None), (200, 1031, 5),
    (400, 700, None), (40, 8193, None), (330, 5000, 7), (1, 131072, None), (2, 131073, 1000)])
def test_ranks_and_cutoffs_at_the_splits(cuda_device, rows, S, levels):
    s, w, k = 4, 33, max(1, S // 5)
    prio = gen.uniform_scores(31, 77, (rows, S), levels=levels)
    if S > 600:
        prio[0, 5], prio[0, 599], prio[0, 17] = float("nan"), float("inf"), -0.0
    order = torch.full((rows, S), -7, dtype=torch.int32, device=cuda_device)
    rank, tau = kv().topk_cutoff(prio.to(cuda_device), s, w, k, order=order)
    rank, tau, order = rank.cpu().numpy(), tau.cpu().numpy(), order.cpu().numpy()
    for r in sorted({0, rows // 2, rows - 1}):
        want = rt.static_ranks(prio[r].numpy())
        assert np.array_equal(rank[r], want)
        assert np.array_equal(order[r, want], np.arange(S))
        assert np.array_equal(tau[r], rt.fenwick_cutoffs(want, s, w, k))


@pytest.mark.parametrize("dtype,d", [("f32", 64), ("bf16", 128)])
@pytest.mark.parametrize("batch,lengths,B,s,levels", [
    (1, [2048], 100, 0, None), (1, [4099], 1024, 4, 3), (1, [16391], 2048, 4, None),
    (3, [1, 700, 2050], 64, 2, 2), (2, [1037, 1037], 1024, 1, None), (90, [611] * 90, 77, 3, 9)])
def test_selection_at_the_splits(cuda_device, dtype, d, batch, lengths, B, s, levels):
    """Kept positions, priorities and K/V rows against a sort of the injected scores."""
    H, D, P = 2, 13, max(lengths)
    dt = gen.torch_dtype(dtype)
    z = torch.zeros
    cache = kv().KVpopCache(batch, H, 1, d, B, D, 4, dt, z(H, 3 * d, 4), z(H, 4), z(H, 4), z(H),
                            n_sink=s)
    score = gen.uniform_scores(11, 78, (batch, H, P), levels=levels)
    K = gen.uniform_scores(12, 79, (batch, H, P, d), device=cuda_device).to(dt)
    V, Q = K * 2, K * 3
    cache.prefill(Q, K, V, lengths, override=score.to(cuda_device))
    st = kv().parse_state(cache.export_state(), cache.cfg)
    as_raw = lambda t: (t.view(torch.int16) if dtype == "bf16" else t).cpu().numpy()  # noqa: E731
    Kr, Vr = as_raw(K), as_raw(V)
    for b in sorted({0, batch // 2, batch - 1}):
        for h in range(H):
            n = max(0, lengths[b] - D)
            p = score[b, h, :n].numpy()
            if n <= B:
                keep = np.arange(n)
            else:
                rest = np.lexsort((np.arange(s, n), -p[s:]))[:B - s] + s
                keep = np.sort(np.concatenate([np.arange(s), rest]))
            i = b * H + h
            m = keep.size
            assert st["nvalid"][i] == m and st["len"][i] == lengths[b]
            assert np.array_equal(st["pos"][i, :m], keep)
            assert np.array_equal(st["score"][i, :m], p[keep])
            assert np.array_equal(st["slotK"][i, :m].view(Kr.dtype), Kr[b, h, keep])
            assert np.array_equal(st["slotV"][i, :m].view(Vr.dtype), Vr[b, h, keep])
            for t in range(max(0, lengths[b] - D), lengths[b]):
                assert np.array_equal(st["ringK"][i, t % D].view(Kr.dtype), Kr[b, h, t])
            if m == B:
                at = s + int(np.argmin(p[keep][s:]))
                assert (st["min_slot"][i], st["min_score"][i]) == (at, p[keep][at])
    cache.free()
