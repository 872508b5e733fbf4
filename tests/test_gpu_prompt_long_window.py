"""Masked prompt attention (bf16, d = 128) under long windows, at the sizes where a tile's lists take
another form: two stages with lists of their own, packed lists, and the first window past them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 4])
@pytest.mark.parametrize("S,w,k,s", [(13001, 11000, 300, 5), (13001, 12400, 200, 0), (17000, 15000, 700, 70),
                                     (24300, 23800, 64, 4), (24700, 24600, 64, 4)])
def test_long_windows(cuda_device, S, w, k, s, G):
    from paper_2607_05061_gb300 import kvpop
    d, n = 128, 2
    g = torch.Generator(device=cuda_device)
    g.manual_seed(S + w + G)
    make = lambda *z: torch.randn(z, generator=g, device=cuda_device).to(torch.bfloat16)  # noqa: E731
    Q, K, V = make(n, G, S, d) * 2, make(n, 1, S, d), make(n, 1, S, d)
    lengths = torch.tensor([S, S - 777], dtype=torch.int32, device=cuda_device)
    prio = torch.randn((n, S), generator=g, device=cuda_device)
    order = torch.empty((n, S), dtype=torch.int32, device=cuda_device)
    rank, tau = kvpop.topk_cutoff(prio, s, w, k, lengths=lengths, order=order)
    Y, lse = kvpop.prompt_attention(Q, K, V, rank.view(n, 1, S), tau.view(n, 1, S), s, w, k, lengths=lengths,
                                    order=order)
    assert kvpop.kvpop_standalone_status(torch.cuda.current_stream().cuda_stream) == 0
    for b in range(n):
        L = int(lengths[b])
        # the first tiles, those around the window's length, and the last ones
        q = torch.tensor(sorted({x for c in (0, w, w + s, w + k, L - 130) for x in range(c - 3, c + 133, 9)
                                 if 0 <= x < L} | {L - 1}), device=cuda_device)
        t = torch.arange(L, device=cuda_device)
        gap = q[:, None] - t[None]
        keep = (gap >= 0) & ((t < s)[None] | (gap < w) | (rank[b, :L][None] <= tau[b, q][:, None]))
        x = (Q[b][:, q].double() @ K[b, 0, :L].double().T / d ** 0.5).masked_fill(~keep, -float("inf"))
        want_l = torch.logsumexp(x, -1)
        want = torch.exp(x - want_l[..., None]) @ V[b, 0, :L].double()
        # probabilities in bf16 on values of size 1; logits of exact products in fp32 sums
        assert (Y[b][:, q].double() - want).abs().max() <= 2e-2
        assert (lse[b][:, q].double() - want_l).abs().max() <= 1e-3
