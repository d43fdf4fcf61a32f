"""The long max-convolution's transforms at every length they take: 2^14 .. 2^21
(columns of 2^7 .. 2^10, rows of 2^7 .. 2^11; 2^22 is covered by the bench
size), with the upper half of the buffer zero (both vectors at most N / 2 long,
which skips the first stage) and not, one vector much shorter, vectors ending
on and next to a power of two."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_maxconv import _check_long, _pair, _sample_outputs, pn  # noqa: E402,F401


@pytest.mark.parametrize("nx,ny", [(8000, 8192), (16000, 300), (16384, 16384), (16385, 16000),
                                   (1, 20000), (40000, 20000), (65536, 65537), (100000, 7),
                                   (131072, 131072), (200000, 300000), (524288, 524289),
                                   (1500000, 500000)])
def test_long_transform_lengths(pn, orc, nx, ny):
    x, y = _pair(1, nx, ny, 2400 + nx % 1000)
    m = _sample_outputs(nx + ny - 1, 100, 2401)
    _check_long(pn, orc, x[0], y[0], list(range(7)), m)
