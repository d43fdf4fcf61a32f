"""A group of one problem: its record reaches the kernels (they read a lone
problem's from the launch arguments) and its result is the product's."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K", [(16, 16, 16), (130, 70, 200), (300, 520, 260)])
@pytest.mark.parametrize("tile_n,scaling,flags", [(128, 2, 0), (256, 2, 0), (128, 1, 0), (128, 2, 4),
                                                  (128, 2, 8)])
def test_group_of_one_equals_the_product(M, N, K, tile_n, scaling, flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1511_05690_gb300 as pn
    g = torch.Generator().manual_seed(M + N + K)
    A = (1.0 - torch.rand((M, K), generator=g)).cuda()
    B = (1.0 - torch.rand((K, N), generator=g)).cuda()
    plan = pn.GroupedProduct([A], [B], compute="bf16", tile_n=tile_n, scaling=scaling,
                             debug_flags=flags)
    C = plan.run(check=True)[0]
    # a second, empty problem makes a group of two: the records then come from the table
    E = torch.empty((0, 4), device="cuda"), torch.empty((4, 0), device="cuda")
    two = pn.GroupedProduct([A, E[0]], [B, E[1]], compute="bf16", tile_n=tile_n, scaling=scaling,
                            debug_flags=flags)
    assert torch.equal(C, two.run(check=True)[0])
