"""Skewed products, whose merged image launch gives one operand a CTA or two: the
same bits as the product of each half of the wide operand."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("compute", ["bf16", "f32", "e4m3"])
@pytest.mark.parametrize("M,N,K", [(128, 20480, 2048), (20480, 128, 2048), (130, 40000, 520)])
def test_halves_of_the_wide_operand(compute, M, N, K):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    g = torch.Generator(device="cuda").manual_seed(N)
    A = torch.rand((M, K), generator=g, device="cuda")
    B = torch.rand((K, N), generator=g, device="cuda")
    C, p_sel, S = pn.maxprod_pnorm(A, B, compute=compute)
    for part in (0, 1):
        if N > M:
            h = slice(part * (N // 2), (part + 1) * (N // 2))
            got, at = pn.maxprod_pnorm(A, B[:, h], compute=compute), (slice(None), h)
        else:
            h = slice(part * (M // 2), (part + 1) * (M // 2))
            got, at = pn.maxprod_pnorm(A[h], B, compute=compute), (h, slice(None))
        assert all(torch.equal(u, v[at]) for u, v in zip(got, (C, p_sel, S)))


@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16", "f16", "e4m3"])
@pytest.mark.parametrize("M,N,K", [(300, 700, 2000), (129, 1500, 1030), (2000, 130, 260)])
def test_rows_of_one_operand_aligned(compute, M, N, K):
    """A, B or neither with 16-byte aligned rows: each operand's images by the kernel of
    its own, or both by one launch, over several levels, with the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    g = torch.Generator(device="cuda").manual_seed(K)

    def pitch(x, ld):
        y = torch.empty((x.shape[0], ld), device="cuda")[:, :x.shape[1]]
        return y.copy_(x)
    A = torch.rand((M, K), generator=g, device="cuda")
    B = torch.rand((K, N), generator=g, device="cuda")
    A *= torch.exp2(-24 * torch.rand((M, K), generator=g, device="cuda"))
    even = [(pitch(A, (K + 7) // 4 * 4), pitch(B, (N + 7) // 4 * 4))]
    odd = [(pitch(A, K // 4 * 4 + 5), even[0][1]), (even[0][0], pitch(B, N // 4 * 4 + 5)),
           (pitch(A, K // 4 * 4 + 5), pitch(B, N // 4 * 4 + 5))]
    want = pn.maxprod_pnorm(*even[0], compute=compute, tile_m=128)
    for a, b in odd:
        got = pn.maxprod_pnorm(a, b, compute=compute, tile_m=128)
        assert all(torch.equal(u, v) for u, v in zip(got, want))
