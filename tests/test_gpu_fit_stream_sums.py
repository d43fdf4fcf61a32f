"""The affine correction's sample sums by the stream over B's rows, at shapes that take
it (test_image_split.py asks the host's rule), against FP64: a full block of samples and
fewer, N not a multiple of 32, a short last range, a family with gaps, the r = 1
projection, samples outside the product.

A sum's FP32 terms are added in chains of at most 200, a relative error of
200 2^-24; a line fitted to estimates and evaluated at them moves by no more than a
few times that (as in test_gpu_fit_stream.py: 4 x 200 2^-24)."""
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


def _pow2_ceil(m):
    f, e = np.frexp(m.astype(np.float64))
    return np.where(m > 0, np.ldexp(1.0, e - (f == 0.5)), 1.0)


def _samples(A, B, fi, fj, p_log2, tau, estimator):
    """Estimate, exact value and class of the samples, in FP64 (scaled)."""
    a = A[fi].astype(np.float64) / _pow2_ceil(A.max(1))[fi][:, None]
    b = (B[:, fj].astype(np.float64) / _pow2_ceil(B.max(0))[fj]).T
    u = a * b
    S = np.stack([(u ** (2.0 ** q)).sum(1) for q in p_log2])
    cls = np.zeros(len(fi), int)
    for q in range(len(p_log2)):
        cls = np.where(S[q] >= tau, q, cls)
    at = np.arange(len(fi))
    p = 2.0 ** np.array(p_log2)[cls]
    est = S[cls, at] ** (1 / p)
    if estimator == 1:
        half = np.maximum(cls - 1, 0)
        pair = (cls > 0) & (np.array(p_log2)[half] == np.array(p_log2)[cls] - 1)
        est = np.where(pair, (S[cls, at] / S[half, at]) ** (2 / p), est)
    return est, u.max(1), cls


# M, N, K, samples, P, estimator
CASES = [(2048, 4100, 4097, 1024, tuple(range(7)), 0), (2048, 4100, 4500, 1024, (0, 2, 3), 0),
         (2048, 4096, 6001, 700, tuple(range(7)), 1), (1500, 8192, 8200, 513, (0, 1, 4), 1),
         (4000, 1024, 4200, 1000, tuple(range(7)), 0)]


@pytest.mark.parametrize("M,N,K,n_fit,p_log2,estimator", CASES)
@pytest.mark.parametrize("compute", ["bf16", "e4m3"])
def test_lines_against_fp64(pn, compute, M, N, K, n_fit, p_log2, estimator):
    g = torch.Generator().manual_seed(M + N + K)
    A = (1.0 - torch.rand((M, K), generator=g)).cuda() ** 0.25
    B = (1.0 - torch.rand((K, N), generator=g)).cuda() ** 0.25
    fi = torch.randint(0, M, (n_fit,), generator=g, dtype=torch.int32)
    fj = torch.randint(0, N, (n_fit,), generator=g, dtype=torch.int32)
    coef = torch.empty(2 * len(p_log2), device="cuda")
    opts = dict(compute=compute, correction=2, fit_i=fi.cuda(), fit_j=fj.cuda(), fit_coef=coef,
                p_log2=p_log2, estimator=estimator, want_psel=False, want_ssel=False)
    pn.maxprod_pnorm(A, B, **opts)
    line = coef.cpu().numpy().astype(np.float64).reshape(-1, 2)
    x, y, cls = _samples(A.cpu().numpy(), B.cpu().numpy(), fi.numpy(), fj.numpy(), p_log2,
                         pn.default_tau(K, compute), estimator)
    for q in np.unique(cls):
        at = cls == q
        if at.sum() < 8:
            continue
        a, b = np.polyfit(x[at], y[at], 1)
        want, got = a * x[at] + b, line[q, 0] * x[at] + line[q, 1]
        assert np.all(np.abs(got - want) <= 4 * 200 * 2.0 ** -24 * np.abs(want))


def test_samples_outside_the_product(pn):
    M, N, K, n_fit = 2048, 4096, 4200, 1024
    g = torch.Generator().manual_seed(1)
    A, B = torch.rand((M, K), generator=g).cuda(), torch.rand((K, N), generator=g).cuda()
    fi = torch.randint(0, M, (n_fit,), generator=g, dtype=torch.int32).cuda()
    fj = torch.randint(0, N, (n_fit,), generator=g, dtype=torch.int32).cuda()
    opts = dict(compute="bf16", correction=2, want_psel=False, want_ssel=False)
    good = pn.maxprod_pnorm(A, B, fit_i=fi, fit_j=fj, **opts)[0]
    for bad, k in ((M, 0), (-1, 1023), (2 ** 31 - 1, 500)):
        out = fi.clone()
        out[k] = bad
        with pytest.raises(pn.PnError) as ei:
            pn.maxprod_pnorm(A, B, fit_i=out, fit_j=fj, **opts)
        assert ei.value.status == 1  # PN_EINVAL
    assert torch.equal(pn.maxprod_pnorm(A, B, fit_i=fi, fit_j=fj, **opts)[0], good)
