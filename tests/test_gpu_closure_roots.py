"""Closures (apsp_pnorm) against squarings formed outside the library: the p-sums of
each squaring by maxprod_pnorm, their roots by NumPy -- FP32 square roots one
after another, FP64 ones within a decade of tau -- and the clamp.  All distances
have the same bits: a root that differs in its last bit can select another p in
the next squaring, which moves distances far beyond rounding."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    pn.lib()
    return pn


def _roots(S, p_sel, tau):
    q = p_sel & 0x7F
    near = S < np.float32(10) * np.float32(tau)
    x, d = S.copy(), S.astype(np.float64)
    for t in range(int(q.max())):
        x = np.where(q > t, np.sqrt(x), x)
        d = np.where(q > t, np.sqrt(d), d)
    return np.where(near, d.astype(np.float32), x)


@pytest.mark.parametrize("lo,hi", [(1.0, 10.0), (0.2, 1.0)])
@pytest.mark.parametrize("n,squarings", [(200, 1), (512, 0), (777, 0), (1033, 0), (1800, 0)])
def test_closure_by_numpy_roots(pn, n, squarings, lo, hi):
    g = torch.Generator(device="cuda").manual_seed(n)
    W = torch.rand((n, n), generator=g, device="cuda") * (hi - lo) + lo
    W[torch.rand((n, n), generator=g, device="cuda") >= 0.1] = math.inf
    W.fill_diagonal_(0.0)
    tau = pn.default_tau(n, "f32")
    X = torch.exp(-W)
    for _ in range(squarings or math.ceil(math.log2(n))):
        _, p_sel, S = pn.maxprod_pnorm(X, X, compute="f32")
        x = np.minimum(_roots(S.cpu().numpy(), p_sel.cpu().numpy(), tau), np.float32(1))
        X = torch.from_numpy(x).cuda()
        X.fill_diagonal_(1.0)
    want = torch.where(X > 0, -torch.log(X), math.inf)
    assert torch.equal(pn.apsp_pnorm(W, n_squarings=squarings), want)
