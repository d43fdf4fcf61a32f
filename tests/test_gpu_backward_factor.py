"""The factor x'^(p-1) / s of the gradients at the ends of FP32's range: subnormal
results rounded once, and a NaN or infinite gradient kept where the operand is 0.

One contraction term with W = dC C / S a power of two makes every gradient entry that
factor times a power of two; NumPy forms the same FP32 chain and rounds once."""
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


def _backward(pn, A, B, dC, q, compute):
    M, N = A.shape[0], B.shape[1]
    one = torch.ones((M, N), device="cuda")
    psel = torch.full((M, N), q, dtype=torch.uint8, device="cuda")
    return pn.maxprod_pnorm_backward(A, B, one, one, psel, dC, p_log2=(q,), compute=compute,
                                     check=False)


@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16"])
@pytest.mark.parametrize("q", [2, 4, 6, 7])
@pytest.mark.parametrize("log_w,span", [(-100, 52.0), (0, 149.0), (20, 175.0)])
@pytest.mark.parametrize("K", [96, 131])
def test_subnormal_results(pn, compute, q, K, log_w, span):
    p, M = 2 ** q, 150
    rng = np.random.default_rng(q + K)
    A = np.exp2(-span / (p - 1) * rng.random((M, K))).astype(np.float32)
    A[:, 0] = 1.0  # every row scale is 1
    dC = -2.0 ** log_w
    dA, _ = _backward(pn, torch.from_numpy(A).cuda(), torch.ones((K, 1), device="cuda"),
                      torch.full((M, 1), dC, device="cuda"), q, compute)
    m, e = np.frexp(A)
    y = np.where(m >= 0.75, m, 2 * m).astype(np.float32)
    e = np.where(m >= 0.75, e, e - 1)
    r = np.ones_like(y)
    for _ in range(q):
        r, y = r * y, y * y
    want = np.ldexp(r.astype(np.float64) * dC, e * (p - 1)).astype(np.float32)
    assert np.any((want != 0) & (np.abs(want) < 2.0 ** -126))
    assert np.array_equal(dA.cpu().numpy(), want)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("q", [1, 6, 8])
@pytest.mark.parametrize("K", [96, 131])
def test_a_bad_gradient_is_not_hidden(pn, bad, q, K):
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.rand((64, K), generator=g, device="cuda") * 0.25 + 0.75
    B = torch.rand((K, 40), generator=g, device="cuda") * 0.25 + 0.75
    A[3, 5:9] = 0.0
    B[7, 2] = 0.0
    dC = torch.ones((64, 40), device="cuda")
    dC[3, 2] = bad
    dA, dB = _backward(pn, A, B, dC, q, "f32")
    assert torch.isnan(dA[3, 5:9]).all() and torch.isnan(dB[7, 2])
    assert not torch.isfinite(dA[3]).any() and not torch.isfinite(dB[:, 2]).any()
    keep = torch.ones(64, dtype=torch.bool, device="cuda")
    keep[3] = False
    assert torch.isfinite(dA[keep]).all()
