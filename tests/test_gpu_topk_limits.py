"""Cutoffs with sinks or a window beyond the row, up to the largest integers: nothing is eligible."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,w", [(2 ** 31 - 1, 1), (2 ** 31 - 40, 16), (2 ** 31 - 500, 4), (701, 1), (700, 1),
                                 (0, 2 ** 31 - 1), (0, 700), (2 ** 31 - 1, 2 ** 31 - 1)])
@pytest.mark.parametrize("k", [1, 2 ** 31 - 1])
def test_nothing_is_eligible(cuda_device, s, w, k):
    from paper_2607_05061_gb300 import kvpop
    S = 700
    prio = torch.arange(2 * S, dtype=torch.float32, device=cuda_device).view(2, S)
    rank, tau = kvpop.topk_cutoff(prio, s, w, k)
    assert torch.equal(rank.cpu(), torch.arange(S - 1, -1, -1, dtype=torch.int32).expand(2, S))
    assert (tau == -1).all()


@pytest.mark.parametrize("s,w", [(698, 1), (0, 699)])
def test_one_token_is_eligible(cuda_device, s, w):
    from paper_2607_05061_gb300 import kvpop
    S = 700
    prio = torch.arange(S, dtype=torch.float32, device=cuda_device).view(1, S)
    _, tau = kvpop.topk_cutoff(prio, s, w, 5)
    assert (tau[0, :S - 1] == -1).all() and int(tau[0, S - 1]) == S - 1 - max(s, 0)
