"""The affine correction's sample sums by the stream over B's rows (many samples,
aligned rows) against a block per sample (B with a row pitch that is no multiple
of 16 bytes): sizes with a last short range and block of indices, fewer samples
than threads, repeated samples.  Each side adds at most about 200 FP32 terms in
a chain, a relative error of 200 2^-24 in a sum (p = 1; less through the other
roots), so the corrected products agree within 4 x 200 2^-24."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K,n_fit", [(300, 512, 16400, 260), (257, 260, 4100, 1024),
                                         (1024, 2048, 4200, 1000), (2048, 4096, 6001, 700)])
@pytest.mark.parametrize("compute", ["bf16", "e4m3"])
def test_stream_equals_block_per_sample(M, N, K, n_fit, compute):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    g = torch.Generator().manual_seed(M + N + K)
    A = (1.0 - torch.rand((M, K), generator=g)).cuda() ** 0.25
    B = (1.0 - torch.rand((K, N), generator=g)).cuda() ** 0.25
    Bp = torch.empty((K, N + 1), device="cuda")[:, :N]
    Bp.copy_(B)
    fi = torch.randint(0, M, (n_fit,), generator=g, dtype=torch.int32).cuda()
    fj = torch.randint(0, N, (n_fit,), generator=g, dtype=torch.int32).cuda()
    opts = dict(compute=compute, correction=2, fit_i=fi, fit_j=fj, want_psel=False,
                want_ssel=False)
    got = pn.maxprod_pnorm(A, B, **opts)[0]
    want = pn.maxprod_pnorm(A, Bp, **opts)[0]
    assert torch.all((got - want).abs() <= 4 * 200 * 2.0 ** -24 * want.abs())
