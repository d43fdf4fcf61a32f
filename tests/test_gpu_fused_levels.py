"""The one-launch product over tiles that go through several levels: its epilogue
stages rows in the memory that the next level's operand copies fill, so every
call has to give the level launches' bits (tile_m = 128 selects them)."""
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


@pytest.mark.parametrize("compute", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("shape", [(256, 256, 512), (1024, 2048, 96)])
def test_every_call_over_all_levels(pn, compute, shape):
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.rand((M, K), generator=g, device="cuda")
    B = torch.rand((K, N), generator=g, device="cuda")
    A *= torch.exp2(-24 * torch.rand((M, K), generator=g, device="cuda"))  # open entries at each p
    want = pn.maxprod_pnorm(A, B, compute=compute, tile_m=128)
    for _ in range(10):
        assert all(torch.equal(u, v) for u, v in zip(pn.maxprod_pnorm(A, B, compute=compute), want))


@pytest.mark.parametrize("compute", ["f32", "bf16", "e4m3"])
@pytest.mark.parametrize("shape", [(256, 256, 512), (1024, 2048, 96)])
def test_a_copy_that_never_lands(pn, compute, shape):
    """The first operand block is never copied (debug_flags bit 4): the bounded wait
    runs out, no further copy is started, those in flight land, and the next
    call works."""
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.rand((M, K), generator=g, device="cuda")
    B = torch.rand((K, N), generator=g, device="cuda")
    want = pn.maxprod_pnorm(A, B, compute=compute, tile_m=128)
    with pytest.raises(pn.PnError) as ei:
        pn.maxprod_pnorm(A, B, compute=compute, timeout_ns=100_000_000, debug_flags=16)
    assert ei.value.status == 6  # PN_ETIMEOUT
    assert all(torch.equal(u, v) for u, v in zip(pn.maxprod_pnorm(A, B, compute=compute), want))
