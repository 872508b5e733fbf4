"""The fp32 prompt attention and future target at the edges of their tiles, against a plain
fp64 evaluation of the mask and the sums."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def kv():
    from paper_2607_05061_gb300 import kvpop
    return kvpop


def inputs(n, H, G, S, d, device, seed=0):
    g = torch.Generator(device="cpu")
    g.manual_seed(seed)
    mk = lambda *s: torch.randn(s, generator=g).to(device)  # noqa: E731
    return mk(n, H * G, S, d), mk(n, H, S, d), mk(n, H, S, d), mk(n * H, S)


def reference(Q, K, V, rank, tau, lengths, s, w):
    """fp64 outputs and normalisers under the mask rebuilt from its definition."""
    n, H, S, d = K.shape
    G = Q.shape[1] // H
    Y, lse = torch.zeros_like(Q, dtype=torch.float64), torch.zeros(Q.shape[:3], dtype=torch.float64, device=Q.device)
    for b in range(n):
        L = lengths[b]
        q = torch.arange(L, device=Q.device)[:, None]
        t = torch.arange(L, device=Q.device)[None]
        for h in range(H):
            r, c = rank[b, h, :L], tau[b, h, :L]
            ok = (t <= q) & ((t < s) | (q - t < w) | ((t <= q - w) & (r[None] <= c[:, None])))
            for g in range(G):
                x = Q[b, h * G + g, :L].double() @ K[b, h, :L].double().T / math.sqrt(d)
                x = x.masked_fill(~ok, -math.inf)
                lse[b, h * G + g, :L] = torch.logsumexp(x, 1)
                Y[b, h * G + g, :L] = torch.softmax(x, 1) @ torch.where(V[b, h, :L].isnan(), 0, V[b, h, :L]).double()
    return Y, lse


# fp32 sums of up to 128 products of N(0, 1) values and a softmax over N(0, 1) values: about
# 1e-6 absolute each; a wrong key or mask moves an output by more than 1e-2
TOL = 1e-5


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G,lengths,k", [(1, [64, 1], 9), (1, [130], 40), (2, [33, 65], 7), (2, [300, 257], 60),
                                         (4, [16, 17], 5), (4, [301], 100), (2, [200], 50000)])
def test_prompt_f32_tiles(cuda_device, d, G, lengths, k):
    s, w, H, S = 3, 12, 2, max(lengths)
    Q, K, V, prio = inputs(len(lengths), H, G, S, d, cuda_device)
    # the value of the last token is NaN: only the last query may see it
    V[:, :, S - 1] = math.nan
    L = torch.tensor(lengths, dtype=torch.int32, device=cuda_device)
    order = torch.empty((len(lengths) * H, S), dtype=torch.int32, device=cuda_device)
    rank, tau = kv().topk_cutoff(prio, s, w, k, lengths=L.repeat_interleave(H), order=order)
    shape = (len(lengths), H, S)
    Y, lse = kv().prompt_attention(Q, K, V, rank.view(shape), tau.view(shape), s, w, k, lengths=L, order=order)
    want_Y, want_lse = reference(Q, K, V, rank.view(shape), tau.view(shape), lengths, s, w)
    for b, n in enumerate(lengths):
        last = n - 1 if n == S else n
        assert (Y[b, :, :last].double() - want_Y[b, :, :last]).abs().max().item() <= TOL if last else True
        assert (lse[b, :, :n].double() - want_lse[b, :, :n]).abs().max().item() <= TOL
        assert n < S or Y[b, :, n - 1].isnan().all()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G,S,w,la", [(1, 1, 0, 0), (1, 64, 0, 0), (2, 65, 1, 0), (2, 193, 64, 0), (4, 320, 7, 3),
                                      (1, 400, 12, 127), (2, 257, 300, 0)])
def test_target_f32_tiles(cuda_device, d, G, S, w, la):
    H = 2
    Q, K, _, _ = inputs(1, H, G, S, d, cuda_device, seed=1)
    dense = kv().causal_lse(Q, K)
    x = torch.einsum("hgqd,htd->hgqt", Q.view(H, G, S, d).double(), K[0].double()) / math.sqrt(d)
    q, t = torch.arange(S, device=cuda_device)[:, None], torch.arange(S, device=cuda_device)[None]
    want = torch.logsumexp(x.masked_fill(t > q, -math.inf), -1)
    assert (dense[0].double() - want.view(H * G, S)).abs().max().item() <= TOL
    logm, _ = kv().future_target(Q, K, dense, w, lookahead=la)
    ok = (q >= t + w) & (q <= t + w + la if la else q >= 0)
    want = torch.logsumexp((x - want[..., None]).masked_fill(~ok, -math.inf), 2).view(H * G, S)
    got = logm[0].double()
    assert torch.equal(got == -math.inf, want == -math.inf)
    fin = want > -math.inf
    assert not fin.any() or (got[fin] - want[fin]).abs().max().item() <= TOL
