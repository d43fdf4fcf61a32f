"""Building a group's table when no memory is left: the C entry may not throw, and the
table holds the problems in the caller's order instead of by descending K.  Host
code only; a process of its own, whose address space is capped."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

BODY = """
import ctypes, resource
import numpy as np
from paper_1511_05690_gb300 import _binding as b
L = b.load()
n = 300_000
mnk = np.zeros((n, 3), np.int64)
mnk[:, 2] = np.arange(n) % 7  # no rows or columns: no tiles
ptrs = np.zeros(n, np.uintp)
o = b.make_opts()
size = L.pn_grouped_table_bytes(n, mnk.ctypes.data, ctypes.byref(o))
assert size > 0
table, ws = np.zeros(size, np.uint8), ctypes.c_size_t(0)
def build():
    p = ptrs.ctypes.data
    return L.pn_grouped_build_table(n, mnk.ctypes.data, p, p, p, ctypes.byref(o),
                                    table.ctypes.data, size, ctypes.byref(ws))
assert build() == 0
by_k = table.copy()
pages = int(open("/proc/self/statm").read().split()[0])
soft, hard = resource.getrlimit(resource.RLIMIT_AS)
resource.setrlimit(resource.RLIMIT_AS, (pages * resource.getpagesize(), hard))
status = build()
resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
assert status == 0
assert not np.array_equal(by_k, table)  # the caller's order
"""


def test_no_memory_for_the_order():
    from paper_1511_05690_gb300 import build
    build.build()
    # large blocks straight from the system, so that the cap meets them
    env = dict(os.environ, MALLOC_MMAP_THRESHOLD_="65536", OPENBLAS_NUM_THREADS="1")
    r = subprocess.run([sys.executable, "-c", BODY], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
