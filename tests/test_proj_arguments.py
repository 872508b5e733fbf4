"""The projections of the binding refuse tensors they would read or write past the end, before any
launch."""
import pytest
import torch


def bf(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16)


BUF = bf(5, 64)


def call(name, **other):
    from paper_2607_05061_gb300 import kvpop
    M, K, nq, nkv = 4, 64, 96, 48
    qkv = dict(x=bf(M, K), Wq=bf(K, nq), Wk=bf(K, nkv), Wv=bf(K, nkv), q=bf(M, nq), k=bf(M, nkv), v=bf(M, nkv))
    out = dict(o=torch.zeros(M, nq), Wo=bf(nq, K), x=bf(M, K), y=bf(M, K))
    args = qkv if name == "project_qkv" else out
    assert set(other) <= set(args)
    getattr(kvpop, name)(**dict(args, **other))


@pytest.mark.parametrize("name,other", [
    ("project_qkv", dict(Wv=bf(64, 40))), ("project_qkv", dict(v=bf(4, 40))), ("project_qkv", dict(v=bf(3, 48))),
    ("project_qkv", dict(Wk=bf(32, 48))), ("project_qkv", dict(Wq=bf(63, 96))), ("project_qkv", dict(q=bf(4, 88))),
    ("project_qkv", dict(Wq=bf(96, 64).T)), ("project_qkv", dict(x=torch.zeros(4, 64))),
    ("project_qkv", dict(k=torch.zeros(4, 48))),
    ("project_out", dict(o=torch.zeros(4, 64))), ("project_out", dict(o=bf(4, 96))),
    ("project_out", dict(o=torch.zeros(3, 96))),
    ("project_out", dict(Wo=bf(96, 56))), ("project_out", dict(y=bf(4, 56))), ("project_out", dict(y=bf(2, 64))),
    ("project_out", dict(x=bf(64, 4).T)), ("project_out", dict(x=BUF[:4], y=BUF[1:]))])
def test_wrong_tensors_are_refused(name, other):
    from paper_2607_05061_gb300 import build
    build.build()
    with pytest.raises(ValueError, match=name):
        call(name, **other)
