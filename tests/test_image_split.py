"""How the CTAs of the merged image launch are shared out between A and B: a CTA's
list of tiles holds 2048 entries, and the busiest CTA sets the time.  The host
function is compiled by itself, no GPU needed."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1511_05690_gb300", "csrc")
LIST = 2048  # tiles per CTA
CTAS = 304   # two on each of 152 SMs


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    d = tmp_path_factory.mktemp("split")
    (d / "s.cpp").write_text(
        '#include "pn_split.h"\n'
        'extern "C" int split(long long a, long long b, int n) { return pn::image_split(a, b, n); }\n'
        'extern "C" int ranges(long long N, long long K, long long f, int n_p, long long room) {\n'
        '  int stages = 0; return pn::fit_stream_ranges(N, K, f, n_p, room, 152, &stages); }\n'
        'extern "C" int even(int bytes, int ctas, int threads, int sms) {\n'
        '  return pn::even_share_smem(bytes, ctas, threads, sms); }\n'
        'static pn::DeviceSet set;\n'
        'extern "C" int add(int d) { int had = set.has(d); set.add(d); return had; }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "s.cpp"),
                    "-o", str(d / "s.so")], check=True)
    f = ctypes.CDLL(str(d / "s.so")).split
    f.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    f.lib = str(d / "s.so")
    return f


def test_what_is_done_once_per_device(split):
    # a kernel's shared-memory limit belongs to a device: each of two needs its own, and
    # one beyond the set's is never taken for done
    add = ctypes.CDLL(split.lib).add
    assert [add(d) for d in (0, 0, 1, 1, 63, 63, 64, 64, -1, -1)] == [0, 1, 0, 1, 0, 1, 0, 0, 0, 0]


def test_the_affine_fit_streams_where_its_tests_mean_it_to(split):
    from test_gpu_fit_stream_sums import CASES
    ranges = ctypes.CDLL(split.lib).ranges
    ranges.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int, ctypes.c_longlong]
    for M, N, K, n_fit, p_log2, _ in CASES:
        got = ranges(N, K, n_fit, len(p_log2), M * (-(-N // 32)))  # the least state array
        assert 16 <= got <= 152 and got * 16 <= K and N % 4 == 0, (M, N, K, got)
    # too few terms, too many columns per sample, no room, more samples than threads
    for N, K, f, room in ((4096, 4095, 1024, 1 << 30), (16388, 8192, 1024, 1 << 30),
                          (4096, 8192, 1024, 15 * 8 * 1024), (4096, 8192, 1025, 1 << 30)):
        assert ranges(N, K, f, 7, room) == 0


def test_an_sm_holds_no_more_than_its_even_share(split):
    even = ctypes.CDLL(split.lib).even
    for threads in (32, 64, 128, 256, 512):
        fit = min(1024 // threads, 32)
        for ctas in (1, 151, 152, 153, 256, 304, 305, 512, 608, 1024, 2000):
            for need in (0, 9000, 24576, 98304):
                got, share = even(need, ctas, threads, 152), -(-ctas // 152)
                assert need <= got <= 226 * 1024 or got == need
                if share >= fit:
                    assert got == need
                    continue
                held = (228 * 1024) // (got + 1024)  # 1 KB of each CTA is the system's
                assert held <= share
                if need <= (228 * 1024) // share - 2048:
                    assert held * 152 >= ctas  # all still fit at once
    assert even(24576, 512, 128, 0 + 152) == (228 * 1024 // 4 - 1024) // 1024 * 1024


def _worst(xa, xb, n, ctas):
    return max(-(-xa // n), -(-xb // (ctas - n)))


def test_no_split_is_better(split):
    rng = random.Random(1)
    for _ in range(3000):
        ctas = rng.choice([2, 3, 8, CTAS, rng.randint(2, CTAS)])
        xa, xb = (int(2 ** rng.uniform(0, 20)) for _ in range(2))
        if xa + xb < ctas:
            ctas = max(2, xa + xb)
        n = split(xa, xb, ctas)
        assert 1 <= n < ctas
        assert _worst(xa, xb, n, ctas) == min(_worst(xa, xb, m, ctas) for m in range(1, ctas))


def test_one_tile_each_when_there_are_fewer_tiles_than_ctas(split):
    for xa, xb in ((1, 1), (1, 200), (200, 1), (100, 150)):
        assert split(xa, xb, xa + xb) == xa


@pytest.mark.parametrize("M,N,K,bk", [
    (1024, 160000, 20480, 64), (128, 19456, 131200, 64), (128, 20480, 16384, 64),
    (19456, 128, 65600, 32), (128, 128 * 2400, 16384, 64)])
def test_skewed_products(split, M, N, K, bk):
    # by the rounded-down share one CTA took all of A: up to 4000 tiles and
    # twice the others' part
    kb = -(-K // bk)
    xa, xb = -(-M // 128) * kb, -(-N // 128) * kb
    n = split(xa, xb, CTAS)
    worst, mean = _worst(xa, xb, n, CTAS), (xa + xb) / CTAS
    assert worst == min(_worst(xa, xb, m, CTAS) for m in range(1, CTAS))
    if mean <= LIST * 0.95:
        assert worst <= LIST and worst <= 1.02 * mean + 1
