"""The first convolution of a process fills the transforms' tables: whatever runs next,
on any stream and before any replay of a captured first call, finds them filled.
Each case is a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import numpy as np, torch
import paper_1511_05690_gb300 as pn
rng = np.random.default_rng(5)
x = rng.random((4, 700), dtype=np.float32) + 0.5
y = rng.random((4, 600), dtype=np.float32) + 0.5
X, Y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
def check(z):
    for a, b, c in zip(x, y, z.cpu().numpy()):
        S = np.convolve((a.astype(np.float64) / a.max()) ** 64, (b.astype(np.float64) / b.max()) ** 64)
        want = S ** (1 / 64) * a.max() * b.max()
        ok = S > 1e-9
        assert ok.sum() > 100 and np.all(np.abs(c - want)[ok] <= 1e-5 * want[ok]), "wrong sums"
"""

CAPTURED = COMMON + """
s = torch.cuda.Stream()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, stream=s):
    z, _ = pn.maxconv_pnorm(X, Y, check=False)
check(pn.maxconv_pnorm(X, Y)[0])
graph.replay()
torch.cuda.synchronize()
check(z)
"""

STREAMS = COMMON + """
a, b = torch.cuda.Stream(), torch.cuda.Stream()
torch.cuda.synchronize()
with torch.cuda.stream(a):
    torch.cuda._sleep(200_000_000)  # about a tenth of a second
    z1, _ = pn.maxconv_pnorm(X, Y, check=False)
with torch.cuda.stream(b):
    z2, _ = pn.maxconv_pnorm(X, Y, check=False)
b.synchronize()
check(z2)
a.synchronize()
check(z1)
"""


@pytest.mark.parametrize("body", [CAPTURED, STREAMS], ids=["captured", "streams"])
def test_first_call(body):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", body], cwd=ROOT, capture_output=True, text=True,
                       timeout=240)
    assert r.returncode == 0, r.stderr[-2000:]
