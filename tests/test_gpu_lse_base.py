"""Dense causal normalisers whose first keys carry far smaller logits than the later ones: the
exponents are formed near the running maximum, not near the first block's."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G", [1, 4])
@pytest.mark.parametrize("low", [0.0, -25.0, -60.0])
def test_base_follows_the_maximum(cuda_device, G, low):
    from paper_2607_05061_gb300 import kvpop
    H, S, d = 2, 4096, 128
    g = torch.Generator()
    g.manual_seed(5 + G)
    Q, K = torch.randn(1, H * G, S, d, generator=g), torch.randn(1, H, S, d, generator=g)
    K[..., [5, 38, 77, 120]] *= 10
    if low:                               # the first keys' logits about 13 or 32 below the others'
        Q[..., 0] = 6
        K[:, :, :256, 0] = low
    Q, K = (t.to(cuda_device, torch.bfloat16) for t in (Q, K))
    got = kvpop.causal_lse(Q, K)
    later = ~torch.ones(S, S, dtype=torch.bool, device=cuda_device).tril()
    err = []
    for r in range(H * G):
        x = (Q[0, r].double() @ K[0, r // G].double().T / d ** 0.5).masked_fill_(later, -float("inf"))
        err.append((got[0, r].double() - torch.logsumexp(x, -1)).abs()[256:])
    err = torch.stack(err)
    print(f"G={G} low={low}: mean {err.mean():.2e} max {err.max():.2e}")
    # values of about 10 (14 in log2 units).  In the mean: half of half a unit in the last place of
    # the sum of base and logarithm (2.4e-7 ln 2 below 16, twice that above) and of the product with
    # ln 2 (2.4e-7); the constants log2(e) / sqrt(d) and ln 2, 9e-9 and 3e-9 of the value, 1.2e-7;
    # logits (fp32 sums of exact products), exponents, 2^x, sums and logarithm 3e-7
    assert err.mean() <= 1.0e-6
