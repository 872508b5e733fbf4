"""Future pass over sequences whose tiles meet at most a block of queries per head, with up to
four heads a tile: the two column halves of a row then part by whole heads."""
import numpy as np
import pytest
import torch

from oracle import future_target as ft

pytestmark = pytest.mark.gpu

TOL = 1e-3                    # bf16 inputs: fp32 sums of exact bf16 products


@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("S,w,la", [(130, 2, 0), (129, 64, 0), (300, 256, 0), (64, 0, 3), (257, 129, 0)])
def test_one_block_per_head(cuda_device, G, S, w, la):
    from paper_2607_05061_gb300 import kvpop
    n, H, d = 24, 8, 128
    g = torch.Generator()
    g.manual_seed(5 * S + G)
    Q = torch.randn((n, H * G, S, d), generator=g).to(torch.bfloat16)
    K = torch.randn((n, H, S, d), generator=g).to(torch.bfloat16)
    x = torch.einsum("nhgqd,nhkd->nhgqk", Q.view(n, H, G, S, d).double(), K.double()) / d ** 0.5
    causal = torch.ones(S, S, dtype=torch.bool).tril()
    lse = torch.logsumexp(x.masked_fill(~causal, -np.inf), -1).reshape(n, H * G, S).float()
    q, k, l = Q.to(cuda_device), K.to(cuda_device), lse.to(cuda_device)
    for _ in range(4):
        logm, _ = kvpop.future_target(q, k, l, w, lookahead=la)
    assert kvpop.kvpop_standalone_status(torch.cuda.current_stream().cuda_stream) == 0
    got = logm.cpu().numpy()
    for b, h in ((0, 0), (7, 5), (n - 1, H - 1)):
        for i in range(G):
            want = ft.future_log_mass(Q[b, h * G + i].double().numpy(), K[b, h].double().numpy(),
                                      lse[b, h * G + i].double().numpy(), w, la)
            fin = np.isfinite(want)
            assert np.array_equal(fin, np.isfinite(got[b, h * G + i]))
            if fin.any():
                assert np.abs(got[b, h * G + i][fin] - want[fin]).max() <= TOL
