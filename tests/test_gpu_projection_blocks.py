"""The projections' last step on whole 32 x 32 blocks: with rows of C 16-byte aligned
(four columns of four rows per lane) it gives what it gives with unaligned rows
(a column per lane), bit for bit; sizes with whole blocks, edges and one block."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K", [(32, 32, 40), (130, 272, 300), (512, 256, 1000)])
@pytest.mark.parametrize("compute", ["bf16", "f32", "e4m3"])
@pytest.mark.parametrize("estimator", [1, 2])
@pytest.mark.parametrize("tile_m", [128, 256])
def test_aligned_rows_equal_unaligned_ones(M, N, K, compute, estimator, tile_m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    g = torch.Generator().manual_seed(M + N + K)
    A = (1.0 - torch.rand((M, K), generator=g)).cuda()
    B = (1.0 - torch.rand((K, N), generator=g)).cuda()
    opts = dict(compute=compute, estimator=estimator, tile_n=128, tile_m=tile_m,
                want_psel=False, want_ssel=False)
    want = pn.maxprod_pnorm(A, B, **opts)[0]
    out = torch.empty((M, N + 1), device="cuda")[:, :N]
    pn.maxprod_pnorm(A, B, out=out, **opts)
    assert torch.equal(out, want)
