"""Normalisers and future pass at the edges of their tiles' rows and columns, with NaN in everything
past a sequence's length."""
import numpy as np
import pytest
import torch

from oracle import future_target as ft

pytestmark = pytest.mark.gpu

TOL = 1e-3                    # bf16 inputs: fp32 sums of exact bf16 products


@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("S,L", [(1, 1), (31, 7), (64, 63), (65, 65), (129, 128), (257, 256), (300, 193), (513, 511)])
def test_tile_edges(cuda_device, G, S, L):
    from paper_2607_05061_gb300 import kvpop
    H, d, w = 3, 128, 5
    lengths = [S, L]
    g = torch.Generator()
    g.manual_seed(7 * S + G)
    Q = torch.randn((2, H * G, S, d), generator=g).to(torch.bfloat16)
    K = torch.randn((2, H, S, d), generator=g).to(torch.bfloat16)
    Q[1, :, L:], K[1, :, L:] = float("nan"), float("nan")
    n = torch.tensor(lengths, dtype=torch.int32, device=cuda_device)
    lse = torch.full((2, H * G, S), float("nan"), device=cuda_device)
    kvpop.causal_lse(Q.to(cuda_device), K.to(cuda_device), lengths=n, lse=lse)
    logm = torch.full((2, H * G, S), 77.0, device=cuda_device)
    kvpop.future_target(Q.to(cuda_device), K.to(cuda_device), lse, w, lengths=n, logm=logm, want_target=False)
    assert kvpop.kvpop_standalone_status(torch.cuda.current_stream().cuda_stream) == 0
    lse, logm = lse.cpu(), logm.cpu()
    assert torch.isnan(lse[1, :, L:]).all() and (logm[1, :, L:] == 77.0).all()
    for b, P in enumerate(lengths):
        for r in range(H * G):
            q, k = Q[b, r, :P].double().numpy(), K[b, r // G, :P].double().numpy()
            want = ft.dense_causal_lse(q, k)
            assert np.abs(lse[b, r, :P].numpy() - want).max() <= TOL
            mass = ft.future_log_mass(q, k, lse[b, r, :P].double().numpy(), w)
            got, fin = logm[b, r, :P].numpy(), np.isfinite(mass)
            assert np.array_equal(fin, np.isfinite(got))
            assert not fin.any() or np.abs(got[fin] - mass[fin]).max() <= TOL
