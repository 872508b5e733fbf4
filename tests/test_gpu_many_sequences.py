"""Prompt calls over more than 64 sequences: the device copy of the lengths must not share its
bytes with the outputs that follow it in the call's workspace."""
import pytest
import torch

from workload import gen

pytestmark = pytest.mark.gpu


def test_prefill_attend_of_many_sequences_equals_chunks(cuda_device):
    from paper_2607_05061_gb300 import kvpop
    n, H, d, B, D = 80, 1, 64, 16, 4
    lengths = [1 + (37 * i) % 40 for i in range(n)]
    P = max(lengths)
    x = [gen.uniform_scores(5, 90 + i, (n, H, P, d), device=cuda_device) for i in range(3)]
    score = gen.uniform_scores(6, 95, (n, H, P), device=cuda_device)
    z = torch.zeros

    def run(groups):
        cache = kvpop.KVpopCache(n, H, 1, d, B, D, 4, torch.float32, z(H, 3 * d, 4), z(H, 4), z(H, 4), z(H))
        Y = z((n, H, P, d), device=cuda_device)
        for b0, b1 in groups:
            cache.prefill_attend(*(t[b0:b1] for t in x), lengths[b0:b1], Y[b0:b1], first_seq=b0,
                                 override=score[b0:b1])
        blob = cache.export_state()
        cache.free()
        return Y, blob

    whole, parts = run([(0, n)]), run([(0, 40), (40, n)])
    assert torch.equal(whole[0], parts[0])
    assert whole[1] == parts[1]
