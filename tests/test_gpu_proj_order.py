"""Projections of the decode stack right behind the kernel that writes their weights: the step
multiplies by the new weights, whichever projection comes first after the write."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def bf(shape, seed, device, scale=1.0):
    g = torch.Generator()
    g.manual_seed(seed)
    return (torch.randn(shape, generator=g) * scale).to(device, torch.bfloat16)


@pytest.mark.parametrize("batch", [1, 9])
def test_weights_written_just_before(cuda_device, batch):
    """The last writer before each call is one long product, as one that merges an adapter is;
    the weights it replaces are NaN, so a single stale one would show."""
    from paper_2607_05061_gb300 import kvpop
    K, nq, nkv, rank = 2048, 4096, 512, 1024
    A, B = bf((K, rank), 1, cuda_device), bf((rank, nq), 2, cuda_device, 1e-2)
    x, res = bf((batch, K), 3, cuda_device), bf((batch, nq), 4, cuda_device)
    Wk, Wv = bf((K, nkv), 5, cuda_device), bf((K, nkv), 6, cuda_device)
    o = bf((batch, K), 7, cuda_device).float()
    W = torch.empty((K, nq), dtype=torch.bfloat16, device=cuda_device)
    y = [torch.empty((batch, n), dtype=torch.bfloat16, device=cuda_device) for n in (nq, nkv, nkv)]
    out = torch.empty_like(res)
    torch.matmul(A, B, out=W)
    kvpop.project_qkv(x, W, Wk, Wv, *y)
    kvpop.project_out(o, W, res, out)
    torch.cuda.synchronize()
    want_q, want_out = y[0].clone(), out.clone()
    for _ in range(20):
        W.fill_(float("nan"))
        torch.matmul(A, B, out=W)
        kvpop.project_qkv(x, W, Wk, Wv, *y)
        W.fill_(float("nan"))
        torch.matmul(A, B, out=W)
        kvpop.project_out(o, W, res, out)
        assert torch.equal(y[0], want_q)
        assert torch.equal(out, want_out)


def test_step_behind_a_weight_update(cuda_device):
    """A plain step of the stack behind an update of every layer's weights equals a replay of the
    captured one, which starts after all that is queued before it."""
    from paper_2607_05061_gb300.stack import DecodeStack
    hid, H, G, d, B, D, F = 1024, 2, 4, 128, 64, 16, 32
    z = torch.zeros
    shapes = {"Wq": (hid, H * G * d), "Wk": (hid, H * d), "Wv": (hid, H * d), "Wo": (H * G * d, hid)}
    new = [{n: bf(s, 10 * l + i, cuda_device, s[0] ** -0.5) for i, (n, s) in enumerate(shapes.items())}
           for l in range(2)]
    layers = [{n: torch.full_like(w, float("nan")) for n, w in p.items()} for p in new]
    for L in layers:
        L.update(W1=z(H, 3 * d, F), b1=z(H, F), w2=z(H, F), b2=z(H))
    outs = []
    for plain in (True, False):
        stack = DecodeStack(layers, 2, hid, H, G, d, B, D, F)
        x, y = bf((2, hid), 5, cuda_device), torch.empty((2, hid), dtype=torch.bfloat16, device=cuda_device)
        for p, L in zip(new, layers):
            for n in shapes:
                L[n].fill_(float("nan"))
        torch.matmul(x, new[0]["Wq"])
        if not plain:
            stack.capture(x, y)
        for p, L in zip(reversed(new), reversed(layers)):     # the first layer's Wq last
            for n in reversed(shapes):
                L[n].copy_(p[n])
        if plain:
            stack.step(x, y)
        else:
            stack.graph.replay()
        for c in stack.caches:
            c.check()
        outs.append(y)
        stack.free()
    assert torch.isfinite(outs[0]).all()
    assert torch.equal(outs[0], outs[1])
