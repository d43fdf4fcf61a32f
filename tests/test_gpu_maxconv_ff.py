"""Max-convolution by transforms in two floats per value against FP64 transforms.

Scales of 2^60 per vector leave every scaled value the same and take the call to
FP64 transforms (a product of scales beyond 1e30), so z / 2^120 and p_sel of the
two calls can be compared."""
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


def _vectors(kind, batch, n, g):
    u = 1.0 - torch.rand((batch, n), generator=g)
    if kind == "wide":
        u = u ** 0.25
    elif kind == "sparse":
        u = u * (torch.rand((batch, n), generator=g) < 0.1)
    elif kind == "decades":  # values over many decades: most sums lie below theta
        u = torch.exp2(-30.0 * u)
    elif kind == "spike":
        u = u * 1e-6
        u[:, n // 2] = 1.0
    return u


# transform lengths 2^4 (FP64 only) .. 2^13, both sides of a power of two
@pytest.mark.parametrize("nx,ny", [(9, 8), (16, 17), (30, 2), (33, 32), (100, 90), (129, 1), (400, 300),
                                   (1024, 1025), (2048, 2049), (3000, 10), (4096, 4096), (4097, 4096)])
@pytest.mark.parametrize("kind", ["uniform", "wide", "sparse", "decades", "spike"])
@pytest.mark.parametrize("tau", [None, 1e-3])
def test_two_float_transforms_equal_fp64_ones(pn, nx, ny, kind, tau):
    g = torch.Generator().manual_seed(nx * 7 + ny)
    x, y = _vectors(kind, 5, nx, g).cuda(), _vectors(kind, 5, ny, g).cuda()
    z, p = pn.maxconv_pnorm(x, y, tau=tau)
    z64, p64 = pn.maxconv_pnorm(x * 2.0 ** 60, y * 2.0 ** 60, tau=tau)
    assert torch.equal(p, p64)
    z, z64 = z.cpu().numpy().astype(np.float64), z64.cpu().numpy().astype(np.float64) * 2.0 ** -120
    # FP64 transforms leave about 1e-15 of the sums' root mean square in every S
    # (an index may be rooted from the direct sum on one side): relative to S,
    # and through the root 1 / p; 2^-20 covers the FP32 roots and scalings
    sxy = (x.amax(1) * y.amax(1)).cpu().numpy().astype(np.float64)[:, None]
    q = (p.cpu().numpy() & 0x7F).astype(np.float64)
    S = np.where(sxy > 0, z64 / np.where(sxy > 0, sxy, 1), 0) ** (2.0 ** q)
    rms = np.sqrt(min(nx, ny)) * min(nx, ny)  # a bound: no sum exceeds its number of terms
    noise = np.where(S > 0, 1e-15 * rms / np.where(S > 0, S, 1), np.inf)
    tol = 2.0 ** -20 + np.minimum(noise, 1e3) / 2.0 ** q
    stable = p.cpu().numpy() < 0x80
    assert np.all(np.abs(z - z64)[stable] <= (tol * z64)[stable])
    # indices no p of which is stable hold the p = 1 sums: only their noise differs
    assert np.all(np.abs(z - z64) <= tol * z64 + 1e-13 * rms * sxy)


def test_rows_do_not_depend_on_the_batch(pn):
    g = torch.Generator().manual_seed(4)
    x, y = _vectors("wide", 40, 300, g).cuda(), _vectors("uniform", 40, 211, g).cuda()
    z, p = pn.maxconv_pnorm(x, y)
    for b in (0, 7, 39):
        z1, p1 = pn.maxconv_pnorm(x[b], y[b])
        assert torch.equal(z[b], z1[0]) and torch.equal(p[b], p1[0])
