"""Which projections a decode stack runs on the weight-streaming kernel: those it takes, within one
wave of CTAs and, for the output, 2^16 values of its input."""
import pytest


@pytest.fixture(scope="module")
def kv():
    from paper_2607_05061_gb300 import build
    build.build()
    from paper_2607_05061_gb300 import kvpop
    return kvpop


# 152 SMs, 6 groups of 8 columns each: 7296 columns at once
@pytest.mark.parametrize("batch,hidden,nq,nkv,want", [
    (1, 4096, 4096, 1024, 3), (16, 4096, 4096, 1024, 3), (17, 4096, 4096, 1024, 1), (32, 4096, 4096, 1024, 1),
    (33, 4096, 4096, 1024, 0), (1, 2560, 4096, 1024, 3), (1, 8192, 8192, 1024, 0), (1, 8192, 4096, 1024, 1),
    (8, 5120, 8192, 2048, 2), (9, 5120, 8192, 2048, 0), (1, 7296, 5248, 1024, 3), (1, 7328, 5256, 1024, 0)])
def test_preferred_projections(kv, batch, hidden, nq, nkv, want):
    got = kv.kvpop_project_preferred(batch, hidden, nq, nkv)
    assert got == want
    assert got & kv.kvpop_project_supported(batch, hidden, nq, nkv) == got


def test_refused_sizes_are_not_preferred(kv):
    for args in ((0, 128, 128, 64), (1, 144, 128, 64), (1, 128, 100, 64), (1, 128, 2 ** 31 - 8, 2 ** 31 - 8)):
        assert kv.kvpop_project_preferred(*args) & 1 == 0
