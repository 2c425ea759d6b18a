"""Large host arrays: xy_touch_pages leaves memory that the host may not write alone (each case in
a child process, which a bad touch would end), and a get_state call that fails leaves its output as
it was."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import ctypes as C, mmap, os
from paper_0811_2111_gb300 import _lib as X
libc = C.CDLL(None, use_errno=True)
libc.mmap.restype = C.c_void_p
libc.mmap.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int, C.c_int, C.c_long]
N, PAGE = 32 << 20, os.sysconf("SC_PAGESIZE")
RW = mmap.PROT_READ | mmap.PROT_WRITE
def region(prot):
    p = libc.mmap(None, N, prot, mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS, -1, 0)
    assert p not in (None, C.c_void_p(-1).value)
    return p
def touch(p, n):
    assert X.lib().xy_touch_pages(C.c_void_p(p), n) == X.XY_OK
def present(p):
    v = (C.c_ubyte * (N // PAGE))()
    assert libc.mincore(C.c_void_p(p), C.c_size_t(N), v) == 0
    return [x & 1 for x in v]
"""

CASES = {
    "fresh": "p = region(RW); touch(p, N); assert all(present(p))",
    # an address range without access (as a device pointer's is), and a read-only one
    "no_access": "touch(region(0), N)",
    "read_only": "touch(region(mmap.PROT_READ), N)",
    # unaligned ends keep the bytes outside them; too small to bother; no memory at all
    "edges": """
p = region(RW)
a = (C.c_ubyte * N).from_address(p)
a[11], a[N - 12] = 171, 172
touch(p + 12, N - 24)
assert all(present(p)) and a[11] == 171 and a[N - 12] == 172
p = region(RW)
touch(p, 4096)
assert not any(present(p))
touch(0, N)
assert X.lib().xy_touch_pages(C.c_void_p(p), -1) == X.XY_EINVAL
""",
    # nothing is written where the pages are there already
    "resident": """
p = region(RW)
a = (C.c_ubyte * N).from_address(p)
for i in range(0, N, PAGE):
    a[i] = 171
touch(p, N)
assert all(a[i] == 171 for i in range(0, N, PAGE))
""",
}


@pytest.mark.parametrize("case", CASES)
def test_touching_pages(case):
    r = subprocess.run([sys.executable, "-c", HEAD + CASES[case]], cwd=ROOT, capture_output=True,
                       text=True)
    assert r.returncode == 0, (r.returncode, r.stderr)


@pytest.mark.gpu
def test_a_failed_read_back_leaves_the_callers_array():
    """get_state on a stream that is being captured: its wait is refused, nothing is copied."""
    import ctypes as C
    import numpy as np
    import torch
    from paper_0811_2111_gb300 import _lib as X
    from paper_0811_2111_gb300.hmc import HMC
    cudart = C.CDLL("libcudart.so.13")
    L = 2048                                 # 16 MB: large enough to be touched
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = HMC(L, 1.0, 3, 0.1, 2, stream=s)
        out = [np.empty(L * L, np.float32) for _ in range(2)]
        marks = [slice(i - 64, i + 64) for i in range(5 * 16384, L * L, 17 * 16384)]
        mark = np.full(128, 0x41414141, np.uint32).view(np.float32)
        for a in out:
            for i in marks:                  # across the starts of some pages (4, 16 or 64 KB)
                a[i] = mark
        s.synchronize()
        g = C.c_void_p()
        assert cudart.cudaStreamBeginCapture(C.c_void_p(s.cuda_stream), 2) == 0
        t = C.c_uint64()
        st = X.lib().xy_hmc_get_state(h.h, out[0].ctypes.data_as(C.c_void_p),
                                      out[1].ctypes.data_as(C.c_void_p), C.byref(t))
        cudart.cudaStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(g))
        cudart.cudaGetLastError()                # (which the refused capture leaves behind)
        assert st == X.XY_ECUDA
        for a in out:
            assert all(np.array_equal(a[i], mark) for i in marks)
        h.close()
