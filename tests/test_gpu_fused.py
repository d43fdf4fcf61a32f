"""The one-launch small product (k_fused_product) against the level launches.

tile_m = 128 selects the level launches; both forms build the same operands
and multiply in the same order, so C, p_sel and S_sel are equal bit for bit."""
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


def _operands(M, N, K, pad, levels, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.rand((M, K + pad), generator=g, device="cuda")[:, :K]
    B = torch.rand((K, N + pad), generator=g, device="cuda")[:, :N]
    if levels:  # entries over several levels, a zero row and a zero column
        A *= torch.exp2(-24 * torch.rand((M, K), generator=g, device="cuda"))
        B *= torch.exp2(-3 * torch.rand((K, N), generator=g, device="cuda"))
        A[M // 2] = 0
        B[:, N // 3] = 0
    return A, B


# tile edges: below, at and past 128 rows, 64 and 128 columns, 32 columns of K
# (a raw block) and one image block of every format; outputs of both widths
# (more than 152 tiles of 128 x 64 take the 128 wide form); pad 0 gives aligned
# rows where K and N are multiples of 4, pad 3 never does
SHAPES = [(1, 1, 1), (128, 64, 32), (129, 65, 33), (127, 63, 31), (256, 192, 128), (130, 257, 100),
          (5, 700, 260), (700, 5, 64), (1000, 1400, 68), (1024, 2048, 40)]


@pytest.mark.parametrize("compute", ["f32", "tf32", "bf16", "f16", "e4m3"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("pad", [0, 3])
def test_fused_equals_level_launches(pn, compute, shape, pad):
    M, N, K = shape
    A, B = _operands(M, N, K, pad, True, M + N + K)
    for kw in ({}, {"estimator": 1}, {"correction": 1}, {"scaling": 0, "p_log2": (0, 2, 3)},
               {"p_log2": (4,)}):
        a = pn.maxprod_pnorm(A, B, compute=compute, **kw)
        b = pn.maxprod_pnorm(A, B, compute=compute, tile_m=128, **kw)
        for u, v in zip(a, b):
            assert torch.equal(u, v), kw


def test_large_scales_divide(pn):
    # a maximum above 2^126: the scale's reciprocal is no normal float
    A, B = _operands(150, 90, 70, 0, False, 5)
    A[3, 7] = 1.5e38
    a = pn.maxprod_pnorm(A, B, compute="f32")
    b = pn.maxprod_pnorm(A, B, compute="f32", tile_m=128)
    assert all(torch.equal(u, v) for u, v in zip(a, b))


@pytest.mark.parametrize("policy", [1, 2])
@pytest.mark.parametrize("n", [2, 65, 128, 200, 333])
def test_apsp_fused_equals_level_launches(pn, n, policy):
    g = torch.Generator(device="cuda").manual_seed(n)
    W = 1 + 9 * torch.rand((n, n), generator=g, device="cuda")
    W[torch.rand((n, n), generator=g, device="cuda") > 0.3] = float("inf")
    W.fill_diagonal_(0.0)
    a = pn.apsp_pnorm(W, diag_policy=policy)
    assert torch.equal(a, pn.apsp_pnorm(W, diag_policy=policy, tile_m=128))


@pytest.mark.parametrize("bad", [-1.0, float("nan"), float("inf"), 3e38])
@pytest.mark.parametrize("where", ["A", "B"])
@pytest.mark.parametrize("pad", [0, 1])
def test_domain_errors(pn, bad, where, pad):
    A, B = _operands(140, 80, 72, pad, False, 9)
    (A if where == "A" else B)[-1, -1] = bad
    with pytest.raises(pn.PnError) as ei:
        pn.maxprod_pnorm(A, B, compute="bf16")
    assert ei.value.status == 4
    A, B = _operands(140, 80, 72, pad, False, 9)
    pn.maxprod_pnorm(A, B, compute="bf16")  # the next call is clean


def test_graph_replay_on_new_inputs(pn):
    A, B = _operands(200, 150, 96, 0, False, 11)
    s = torch.cuda.Stream()
    out = torch.empty((200, 150), device="cuda")
    pn.maxprod_pnorm(A, B, out=out)
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(graph, stream=s):
            pn.maxprod_pnorm(A, B, out=out, check=False, stream=s)
    A2, B2 = _operands(200, 150, 96, 0, False, 12)
    A.copy_(A2)
    B.copy_(B2)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, pn.maxprod_pnorm(A2, B2, tile_m=128)[0])
