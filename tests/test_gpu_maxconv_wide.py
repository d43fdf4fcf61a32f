"""Max-convolutions whose sums span many decades -- wide ranges of values, sparse
vectors, short y -- so that they fall back to FP64 transforms and direct sums,
against sums formed directly in FP64 by NumPy.

An FP64 transform's error is at most about 16 2^-53 log2(N) (|x|^2 + |y|^2) in a sum; a
root adds (log2 p + 2) 2^-24.  Sums that lie within that error of tau may select
either p; the estimate is checked at the p selected."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TAU = 1e-12


def _values(kind, rng, n):
    u = rng.random(n)
    if kind == "sparse":
        return (u * (rng.random(n) < 0.05)).astype(np.float32)
    if kind == "subnormal":  # one large value over a floor down to 2^-149
        v = np.exp2(-120 - 29 * u).astype(np.float32)
        v[n // 2] = 1.0
        return v
    if kind == "one":
        v = np.zeros(n, np.float32)
        v[n // 3] = 1.5
        return v
    return np.exp2(-float(kind) * u).astype(np.float32)


def _sums(x, y, P):
    """S^(p) of every output for p = 1, 2, .. 2^(P-1), from FP32 powers, and |x|^2 + |y|^2."""
    xs = x * np.float32(1.0 / np.float64(x.max()))
    ys = y * np.float32(1.0 / np.float64(y.max()))
    S, norm = [], []
    for _ in range(P):
        a, b = xs.astype(np.float64), ys.astype(np.float64)
        S.append(np.convolve(a, b))
        norm.append((a * a).sum() + (b * b).sum())
        xs, ys = xs * xs, ys * ys
    return np.array(S), np.array(norm)


@pytest.mark.parametrize("kx,ky", [("4", "4"), ("30", "30"), ("0.01", "30"), ("100", "6"),
                                   ("sparse", "sparse"), ("one", "4"), ("subnormal", "8")])
@pytest.mark.parametrize("nx,ny", [(4096, 8), (4096, 64), (700, 63), (900, 800), (64, 1),
                                   (1, 33), (2500, 2500)])
def test_against_direct_sums(kx, ky, nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    rng = np.random.default_rng(nx + ny)
    X = np.stack([_values(kx, rng, nx) for _ in range(3)])
    Y = np.stack([_values(ky, rng, ny) for _ in range(3)])
    X[:, 0] = Y[:, 0] = 1.0  # no row of zeros
    z, sel = pn.maxconv_pnorm(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    z, sel = z.cpu().numpy().astype(np.float64), sel.cpu().numpy()
    log_n = np.log2(nx + ny) + 1
    for b in range(3):
        S, norm = _sums(X[b], Y[b], 7)
        err = (16 * 2.0 ** -53 * log_n * norm)[:, None] + 2.0 ** -48 * S
        q = np.minimum(sel[b] & 0x7F, 6).astype(int)
        at = np.arange(S.shape[1])
        # the largest p whose sum reaches tau, up to the error of the sums
        for p in range(7):
            assert not np.any((q < p) & (S[p] >= TAU + err[p]))
        stable = sel[b] < 0x80
        assert not np.any(stable & (S[q, at] < TAU - err[q, at]))
        assert not np.any(~stable & ((q != 0) | (S[0] >= TAU + err[0])))
        # z = (S +- err)^(1/p), S and err of the p selected, rounded
        scale, r = float(X[b].max()) * float(Y[b].max()), np.exp2(-q.astype(float))
        lo = np.maximum(S[q, at] - err[q, at], 0.0) ** r * scale
        hi = (S[q, at] + err[q, at]) ** r * scale
        tol = (q + 3) * 2.0 ** -24 * 1.5
        assert np.all((z[b] >= lo * (1 - tol) - 1e-44) & (z[b] <= hi * (1 + tol) + 1e-44))


@pytest.mark.parametrize("nx,ny", [(8000, 150), (150, 8000), (4000, 60)])
def test_one_vector_outweighs_the_other(nx, ny):
    """A long vector of ones and small values against a single 1: the outputs are the
    long vector's values, to one rounding (p = 1 leaves nothing of an error in S)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    n, k = max(nx, ny), min(nx, ny)
    g = torch.Generator().manual_seed(n)
    v, one = torch.ones((40, n)), torch.zeros((40, k))
    small = torch.exp2(-15 + torch.rand((40, n // 17), generator=g))
    v[:, 5:5 + 16 * (n // 17):16] = small
    one[:, 3] = 1.0
    x, y = (v, one) if nx > ny else (one, v)
    z, _ = pn.maxconv_pnorm(x.cuda(), y.cuda(), p_log2=(0,))
    z = z.cpu()[:, 3:3 + n].double()
    assert torch.all((z - v.double()).abs() <= 2.0 ** -24 * v)
