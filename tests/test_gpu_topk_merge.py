"""The merged NormQueue pops (k <= 2048) against the pops made one after another
(larger k), and the transforms of every length, on the GPU.

Both forms make the same pops in the same order, so the first 2048 of a call
with k = 2049 equal a call with k = 2048 bit for bit."""
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


def _inputs(kind, n):
    g = torch.Generator().manual_seed(n)
    x, y = torch.rand((3, n), generator=g), torch.rand((3, n), generator=g)
    if kind == "equal":       # every product equal: ties between all diagonals
        x, y = torch.ones(3, n), torch.full((3, n), 0.5)
    elif kind == "geometric":  # the terms of a diagonal are equal
        x = y = torch.exp2(-0.25 * torch.arange(n, dtype=torch.float32)).repeat(3, 1)
    elif kind == "few":       # mostly zeros: diagonals without a term above 0
        x, y = x * (x > 0.9), y * (y > 0.9)
    return x.cuda(), y.cuda()


# transform lengths 2^1 .. 2^13, and n on both sides of a power of two
@pytest.mark.parametrize("kind", ["random", "equal", "geometric", "few"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 17, 64, 65, 200, 512, 513, 1500, 4095, 4096])
def test_merged_pops_equal_sequential_pops(pn, kind, n):
    x, y = _inputs(kind, n)
    a = pn.topk_xy(x, y, 2048)
    b = pn.topk_xy(x, y, 2049)
    for u, v in zip(a, b):
        assert torch.equal(u, v[:, :2048])


@pytest.mark.parametrize("k", [1, 31, 32, 33, 1000])
@pytest.mark.parametrize("p_log2", [(0,), (2, 5), tuple(range(13)), tuple(range(16))])
def test_shorter_k_is_a_prefix(pn, k, p_log2):
    x, y = _inputs("random", 700)
    a = pn.topk_xy(x, y, k, p_log2=p_log2)
    b = pn.topk_xy(x, y, 2049, p_log2=p_log2)
    for u, v in zip(a, b):
        assert torch.equal(u, v[:, :k])


@pytest.mark.parametrize("n", [1, 2, 3, 6, 11, 20, 40, 90, 170, 300, 700, 1100, 2100])
def test_first_estimate_in_its_envelope(pn, n):
    # the first pop is the largest p-norm estimate: at least the largest product
    # and at most the n^(1/p*) envelope of the largest p that the products of
    # the top diagonals leave stable (p* >= 32 for values in [0.5, 1])
    g = torch.Generator().manual_seed(n)
    x, y = 0.5 + 0.5 * torch.rand((2, n), generator=g), 0.5 + 0.5 * torch.rand((2, n), generator=g)
    vals, _, _ = pn.topk_xy(x.cuda(), y.cuda(), 1)
    top = (x.double().amax(1) * y.double().amax(1)).numpy()
    v = vals.cpu().numpy()[:, 0].astype(np.float64)
    assert np.all(v >= top * (1 - 1e-6)) and np.all(v <= top * n ** (1 / 32) * (1 + 1e-6))
