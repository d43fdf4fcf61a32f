"""The adjoint's operand images and gradient factor at the edges of their blocks:
gradients against plain FP64 torch, tiles of both shapes against each other."""
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


def _grad64(A, B, C, S, psel, G, plogs):
    """dA, dB of the p-norm product at fixed p*, from the forward's own C and S."""
    def scale(x, dim):
        m, e = torch.frexp(x.amax(dim, keepdim=True).double())
        return torch.where(m > 0, torch.ldexp(torch.ones_like(m), e - (m == 0.5).to(e.dtype)), 1.0)
    r, c = scale(A, 1), scale(B, 0)
    a, b = A.double() / r, B.double() / c
    W = torch.where(S > 0, G.double() * C.double() / S.double(), 0.0)
    dA, dB = torch.zeros_like(a), torch.zeros_like(b)
    for q in plogs:
        p = 2 ** q
        w = torch.where((psel & 0x7F) == q, W, 0.0)
        dA += (w @ (b ** p).t()) * a ** (p - 1) / r
        dB += ((a ** p).t() @ w) * b ** (p - 1) / c
    return dA, dB


# below, at and past the 128 x 128 source blocks and the image blocks of each format
@pytest.mark.parametrize("shape", [(1, 1, 1), (128, 128, 128), (127, 129, 65), (130, 33, 257), (260, 100, 31)])
@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16"])
@pytest.mark.parametrize("plogs", [(0,), (4,), (0, 1, 2, 3, 4, 5, 6), (8,)])
def test_gradients_at_block_edges(pn, shape, compute, plogs):
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.rand((M, K), generator=g, device="cuda")
    B = torch.rand((K, N), generator=g, device="cuda")
    if max(plogs) > 7:  # values near 1: the sums, and W = dC C / S, stay in FP32's range
        A, B = 1 - A / 64, 1 - B / 64
    A[0, 0] = 0.0  # a zero entry: its factor is 0 for p > 1
    G = torch.randn((M, N), generator=g, device="cuda")
    C, psel, S = pn.maxprod_pnorm(A, B, p_log2=plogs, compute=compute)
    outs = [pn.maxprod_pnorm_backward(A, B, C, S, psel, G, p_log2=plogs, compute=compute, tile_m=tm)
            for tm in (0, 128, 256)]
    for o in outs[1:]:
        assert torch.equal(o[0], outs[0][0]) and torch.equal(o[1], outs[0][1])
    # operands: squarings 2 (p - 1) 2^-24, casts 2 u, W two roundings; FP32 sums
    u = {"f32": 2.0 ** -21, "tf32": 2.0 ** -11, "bf16": 2.0 ** -8}[compute]
    p = 2.0 ** max(plogs)
    for out, ref, n in zip(outs[0], _grad64(A, B, C, S, psel, G, plogs), (N, M)):
        tol = 4 * p * 2.0 ** -24 + 2 * u + 2.0 ** -22
        scale = ref.abs().max()  # signs of G cancel: an absolute bound
        assert torch.all((out.double() - ref).abs() <= (tol + n * 2.0 ** -23) * scale * 4 + 2.0 ** -149)
