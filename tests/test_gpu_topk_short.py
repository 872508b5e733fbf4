"""Ranks and cutoffs of short rows: at the edges of the row length up to which one CTA ranks a row,
of its warps' shares of the queries, and of the number of rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def reference(prio, L, s, w, k):
    """Ranks by (priority descending, position ascending) and the min(k, n)-th smallest of the ranks
    eligible at each query."""
    order = torch.argsort(prio[:L], descending=True, stable=True)
    rank = torch.empty(L, dtype=torch.int64)
    rank[order] = torch.arange(L)
    tau = torch.full((L,), -1, dtype=torch.int64)
    for q in range(L):
        r = rank[s:max(s, q - w + 1)]
        if r.numel():
            tau[q] = torch.sort(r).values[min(k, r.numel()) - 1]
    return order, rank, tau


@pytest.mark.parametrize("rows", [1, 305])
@pytest.mark.parametrize("S", [1, 15, 16, 17, 33, 129, 383, 384, 385])
def test_short_rows(cuda_device, rows, S):
    from paper_2607_05061_gb300 import kvpop
    g = torch.Generator()
    g.manual_seed(S + rows)
    prio = torch.randint(-5, 6, (rows, S), generator=g).float()          # many ties
    prio[:, ::7] = torch.randn((rows, S), generator=g)[:, ::7]
    lengths = torch.randint(0, S + 1, (rows,), generator=g, dtype=torch.int32)
    lengths[0] = S
    order = torch.full((rows, S), -7, dtype=torch.int32, device=cuda_device)
    for s, w, k in ((0, 1, 1), (3, 5, 20), (0, 16, 1000)):
        rank, tau = kvpop.topk_cutoff(prio.to(cuda_device), s, w, k, lengths=lengths.to(cuda_device), order=order)
        rank, tau, got = rank.cpu(), tau.cpu(), order.cpu()
        for i in sorted({0, rows // 2, rows - 1}):
            L = int(lengths[i])
            o, r, t = reference(prio[i], L, s, w, k)
            assert torch.equal(got[i, :L].long(), o) and torch.equal(rank[i, :L].long(), r)
            assert torch.equal(tau[i, :L].long(), t)
            assert (rank[i, L:] == -1).all() and (tau[i, L:] == -1).all()
