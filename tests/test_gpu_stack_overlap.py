"""A stack's step whose output shares part of its input's memory is refused; in place it is not."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_partly_shared_hidden_states_are_refused(cuda_device):
    from paper_2607_05061_gb300.stack import DecodeStack
    hid, H, G, d, B, D, F, b = 256, 2, 1, 128, 32, 8, 32, 3
    z = torch.zeros
    g = torch.Generator()
    g.manual_seed(1)
    L = {n: (torch.randn(s, generator=g) * s[0] ** -0.5).to(cuda_device, torch.bfloat16) for n, s in (
        ("Wq", (hid, H * G * d)), ("Wk", (hid, H * d)), ("Wv", (hid, H * d)), ("Wo", (H * G * d, hid)))}
    L.update(W1=z(H, 3 * d, F), b1=z(H, F), w2=z(H, F), b2=z(H))
    x = torch.randn((b + 1, hid), generator=g).to(cuda_device, torch.bfloat16)
    stacks = [DecodeStack([L], b, hid, H, G, d, B, D, F) for _ in range(3)]
    want = stacks[0].step(x[:b].clone())
    same = x[:b].clone()
    stacks[1].step(same, same)
    assert torch.equal(same, want)
    with pytest.raises(RuntimeError):
        stacks[2].step(x[:b], x[1:])
    for s in stacks:
        s.free()
