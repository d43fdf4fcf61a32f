"""Stores at the product's edges: rows that are not 16-byte aligned, whole 32 x 32
blocks and blocks cut off by the last row or column, against the same product
with B's columns padded to an aligned width (the columns are independent, so the
values agree bit for bit)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pn():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    return pn


def _pair(M, N, K, wide, seed):
    g = torch.Generator().manual_seed(seed)
    A, B = 1.0 - torch.rand((M, K), generator=g), 1.0 - torch.rand((K, N), generator=g)
    if wide:  # many binades: the entries of a block resolve at different p
        A, B = torch.exp2(-40.0 * A), torch.exp2(-40.0 * B)
    A, B = A.cuda(), B.cuda()
    pad = torch.zeros((K, -N % 8), device="cuda")
    return A, B, torch.cat([B, pad], 1).contiguous()


@pytest.mark.parametrize("M,N", [(1, 1), (31, 33), (32, 31), (33, 63), (127, 127), (128, 129),
                                 (129, 95), (160, 257), (300, 1)])
@pytest.mark.parametrize("compute", ["bf16", "f32"])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("K", [64, 3000])
def test_unaligned_rows_equal_aligned_ones(pn, M, N, compute, wide, K):
    A, B, Bp = _pair(M, N, K, wide, M * 1000 + N)
    opts = dict(compute=compute, tile_n=128, tile_m=128)
    for got, want in zip(pn.maxprod_pnorm(A, B, **opts), pn.maxprod_pnorm(A, Bp, **opts)):
        assert torch.equal(got, want[:, :N])
    plan = pn.GroupedProduct([A, A], [B, Bp], compute=compute, tile_n=128)
    got, want = plan.run(check=True)
    assert torch.equal(got, want[:, :N])
