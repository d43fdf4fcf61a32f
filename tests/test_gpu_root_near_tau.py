"""The 1/p root within a decade of tau, and of sums too small or too large for the
FP32 form, against FP64 square roots rounded to FP32: the same bits.

One contraction term and a one-value family make every entry the root of its
own S_sel; a threshold above every sum puts all entries near it."""
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


def _fp64_roots(S, q):
    r = S.astype(np.float64)
    for _ in range(q):
        r = np.sqrt(r)
    return r.astype(np.float32)


@pytest.mark.parametrize("q", [1, 2, 3, 4, 5, 6, 7, 9])
@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16"])
@pytest.mark.parametrize("shape", [(33, 65), (640, 1024)])
def test_near_tau(pn, compute, q, shape):
    M, N = shape
    p = 2.0 ** q
    g = torch.Generator().manual_seed(M + q)
    # log2 of the powered products from 0 down past 2^-149
    a = torch.exp2(-80.0 / p * torch.rand((M, 1), generator=g))
    b = torch.exp2(-80.0 / p * torch.rand((1, N), generator=g))
    a[0], b[0, 0] = 0.0, 1.0  # a row of zeros
    C, _, S = pn.maxprod_pnorm(a.cuda(), b.cuda(), p_log2=(q,), compute=compute, scaling=0,
                               tau=4.0)
    C, S = C.cpu().numpy(), S.cpu().numpy()
    assert np.array_equal(C, _fp64_roots(S, q))


@pytest.mark.parametrize("q", [1, 2, 3, 6, 7, 9])
@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16"])
def test_large_sums(pn, compute, q):
    # unscaled operands whose sums reach from 2^100 to 2^128 and past it
    p = 2.0 ** q
    g = torch.Generator().manual_seed(q)
    a = torch.exp2((50 + 14.2 * torch.rand((200, 1), generator=g)) / p)
    b = torch.exp2((50 + 14.2 * torch.rand((1, 300), generator=g)) / p)
    C, _, S = pn.maxprod_pnorm(a.cuda(), b.cuda(), p_log2=(q,), compute=compute, scaling=0)
    C, S = C.cpu().numpy(), S.cpu().numpy()
    want = S.astype(np.float64) ** (1.0 / p)
    assert np.array_equal(np.isinf(C), np.isinf(S)) and np.isinf(S).any()
    fin = np.isfinite(S)
    # as test_gpu_root.py: half an ulp and one rounding; two hardware approximations
    tol = 2.0 ** -23 if compute == "f32" else 2.0 ** -21 + 2.0 ** -15 / p
    assert np.all(np.abs(C[fin] - want[fin]) <= tol * want[fin])
    if compute == "f32":
        big = fin & (S >= 2.0 ** 120)
        assert big.any() and np.array_equal(C[big], _fp64_roots(S[big], q))
