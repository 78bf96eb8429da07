"""Host-side checks of the solve server (no GPU needed)."""
import mmap
import signal
import subprocess
import sys

import pytest

# a child process touches n bytes at offset `at` of a mapping of three pages,
# of which `closed` (in order) have been made read-only or taken away
CHILD = """
import ctypes, mmap, sys
at, n, closed, prot = (int(a) for a in sys.argv[1:5])
sys.path.insert(0, sys.argv[5])
from paper_1304_5546_gb300 import _lib
lib = _lib.load()
page = mmap.PAGESIZE
m = mmap.mmap(-1, 3 * page)
buf = (ctypes.c_ubyte * (3 * page)).from_buffer(m)
for i in range(3 * page):
    buf[i] = i * 31 % 251
libc = ctypes.CDLL(None, use_errno=True)
libc.mprotect.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
base = ctypes.addressof(buf)
if closed >= 0:
    assert libc.mprotect(base + closed * page, page, prot) == 0
status = lib.dg_test_host_touch(base + at, n)
if closed >= 0:
    assert libc.mprotect(base + closed * page, page, 3) == 0
assert status == 0 and all(buf[i] == i * 31 % 251 for i in range(3 * page))
"""


@pytest.fixture(scope="module")
def lib():
    from paper_1304_5546_gb300 import build as B
    B.build()
    from paper_1304_5546_gb300 import _lib
    return _lib


# CUDA error codes: success, not ready, illegal address, launch failure,
# out of memory, context destroyed, unknown
@pytest.mark.parametrize("code,state", [(0, "DONE"), (600, "RUNNING"), (700, "FAILED"),
                                        (719, "FAILED"), (2, "FAILED"), (709, "FAILED"),
                                        (999, "FAILED")])
def test_state_of_a_result_by_its_event(lib, code, state):
    assert lib.load().dg_test_result_state(code) == getattr(lib, "DG_REQUEST_" + state)


@pytest.mark.parametrize("at,pages,less,closed,prot,dies", [
    (0, 3, 0, -1, 0, False),    # everything open: the contents stay
    (0, 3, 0, 2, 1, True),      # the last page read-only
    (8, 2, 0, 2, 1, True),      # eight bytes of it in the range
    (8, 2, 8, 2, 0, False),     # none: a page beside the range is not accessed
    (-4, 1, -4, 0, 0, True),    # four bytes of an unmapped first page
    (0, 1, 0, 0, 0, True),
    (0, 0, 0, 0, 0, False),     # nothing
])
def test_pages_of_a_result_are_touched_by_the_host(lib, at, pages, less, closed, prot, dies):
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    page = mmap.PAGESIZE
    at = at if at >= 0 else page + at
    r = subprocess.run([sys.executable, "-c", CHILD, str(at), str(pages * page - less),
                        str(closed), str(prot), root], capture_output=True, text=True, timeout=300)
    assert r.returncode == (-signal.SIGSEGV if dies else 0), (r.returncode, r.stderr)
