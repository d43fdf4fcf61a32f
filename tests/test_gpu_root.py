"""The 1/p root of the 3xTF32 epilogue over the range of the sums, against FP64.

One contraction term and a one-value family make every entry the root of its
own S_sel, also where S_sel lies below the root's range, is subnormal or 0."""
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


@pytest.mark.parametrize("q", [0, 1, 2, 3, 5, 6, 7, 9, 12])
@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16"])
@pytest.mark.parametrize("shape", [(33, 65), (128, 300), (256, 256)])
def test_root_of_the_selected_sum(pn, compute, q, shape):
    M, N = shape
    p = 2.0 ** q
    g = torch.Generator().manual_seed(M + q)
    # log2 of the products from 0 down past 2^-149 once powered
    a = torch.exp2(-80.0 / p * torch.rand((M, 1), generator=g))
    b = torch.exp2(-80.0 / p * torch.rand((1, N), generator=g))
    a[0], b[0, 0] = 0.0, 1.0  # a row of zeros; scales are 1 elsewhere
    C, _, S = pn.maxprod_pnorm(a.cuda(), b.cuda(), p_log2=(q,), compute=compute, scaling=0)
    C, S = C.cpu().numpy().astype(np.float64), S.cpu().numpy().astype(np.float64)
    want = S ** (1.0 / p)
    # 3xTF32: half an ulp of the root, one rounding of the two unit scales' product;
    # the other formats root by two hardware approximations (2^-22 each, the
    # logarithm's rounding 2^-17 / p), but to 3xTF32's accuracy near tau
    tol = 2.0 ** -23 if compute == "f32" else 2.0 ** -21 + 2.0 ** -16 / p
    assert np.all(np.abs(C - want) <= tol * want)
    assert np.all(C[S == 0] == 0)
