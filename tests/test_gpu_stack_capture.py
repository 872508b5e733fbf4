"""A stack captured in a process that has run no library product before, with projections on the
library and without."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = '''
import sys, torch
from paper_2607_05061_gb300.stack import DecodeStack
hid, batch = int(sys.argv[1]), int(sys.argv[2])
H, G, d, B, D, F = 1, 2, 128, 32, 8, 32
z = torch.zeros
g = torch.Generator()
g.manual_seed(1)
L = {n: (torch.randn(s, generator=g) * s[0] ** -0.5).to("cuda", torch.bfloat16) for n, s in (
    ("Wq", (hid, H * G * d)), ("Wk", (hid, H * d)), ("Wv", (hid, H * d)), ("Wo", (H * G * d, hid)))}
L.update(W1=z(H, 3 * d, F), b1=z(H, F), w2=z(H, F), b2=z(H))
x = torch.randn((batch, hid), generator=g).to("cuda", torch.bfloat16)
y = torch.empty_like(x)
stack = DecodeStack([L], batch, hid, H, G, d, B, D, F)
stack.capture(x, y)
stack.graph.replay()
stack.caches[0].check()
other = DecodeStack([L], batch, hid, H, G, d, B, D, F)
assert torch.equal(other.step(x), y)
print("captured")
'''


@pytest.mark.parametrize("hidden,batch", [(7424, 1), (256, 40), (256, 1)])
def test_capture_first(cuda_device, hidden, batch):
    r = subprocess.run([sys.executable, "-c", CODE, str(hidden), str(batch)], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stdout + r.stderr[-2000:]
