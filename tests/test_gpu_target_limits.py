"""Future pass with a window or a lookahead beyond the sequence, up to the largest integers."""
import pytest
import torch

pytestmark = pytest.mark.gpu

BIG = 2 ** 31 - 1


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 128), (torch.bfloat16, 64), (torch.float32, 64)])
@pytest.mark.parametrize("w,la,w2,la2", [(BIG, 0, 300, 0), (BIG - 100, BIG, 300, 0), (5, BIG, 5, 0), (5, BIG - 7, 5, 0)])
def test_same_as_the_sequence_length(cuda_device, dtype, d, w, la, w2, la2):
    from paper_2607_05061_gb300 import kvpop
    S, H, G = 300, 2, 2
    g = torch.Generator()
    g.manual_seed(3)
    Q = torch.randn((1, H * G, S, d), generator=g).to(cuda_device, dtype)
    K = torch.randn((1, H, S, d), generator=g).to(cuda_device, dtype)
    lse = kvpop.causal_lse(Q, K)
    got = kvpop.future_target(Q, K, lse, w, lookahead=la)
    want = kvpop.future_target(Q, K, lse, w2, lookahead=la2)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert torch.isneginf(got[0]).all() == (w >= S)
