"""The kernel that HMC trajectories run (xy_hmc_kernel): AUTO's lines by side, row alignment and
precision, each side of every line against the per-site kernel bit for bit."""
import ctypes as C

import numpy as np
import pytest

from paper_0811_2111_gb300 import _lib as X

LINES = {"accurate": (420, 420, 445), "fast": (470, 470, 522), "libm": (470, 484, 486)}


def _first(line, rest):
    """The first side from `line` on with L % 4 = 0, 2 or odd (rest 0, 1, 2), and the last before."""
    ok = lambda L: L % 128 != 0 and ((L % 2 == 1) if rest == 2 else L % 4 == 2 * rest)
    L = next(L for L in range(line, line + 9) if ok(L))
    return L, next(L for L in range(line - 1, line - 10, -1) if ok(L))


def test_null_arguments():
    k = C.c_int32(-1)
    assert X.lib().xy_hmc_kernel(None, C.byref(k)) == X.XY_EINVAL and k.value == -1


@pytest.mark.gpu
def test_sides_and_explicit_kernels():
    from paper_0811_2111_gb300.hmc import HMC
    for L, kernel, expected in ((3, "auto", "site"), (4, "auto", "resident"), (176, "auto", "resident"),
                                (177, "auto", "site"), (256, "auto", "site"), (384, "auto", "tiled2"),
                                (2048, "auto", "tiled2"), (128, "site", "site"),
                                (128, "cluster", "cluster"), (128, "tiled", "tiled"),
                                (128, "tiled_tma", "tiled_tma")):
        with HMC(L, 1.0, 1, 0.1, 2, kernel=kernel) as h:
            assert h.kernel == expected, L


@pytest.mark.gpu
@pytest.mark.parametrize("rest", [0, 1, 2])
@pytest.mark.parametrize("sincos", LINES)
def test_two_steps_per_launch_from_the_line_on(sincos, rest):
    from paper_0811_2111_gb300.hmc import HMC
    above, below = _first(LINES[sincos][rest], rest)
    for L, kernel in ((above, "tiled2"), (below, "site")):
        with HMC(L, 1.1, 9, 0.2, 5, sincos=sincos) as h, \
                HMC(L, 1.1, 9, 0.2, 5, sincos=sincos, kernel="site") as ref:
            assert h.kernel == kernel, L
            for x in (h, ref):
                x.run(3)
            for a, b in zip(h.state(), ref.state()):
                assert np.array_equal(a, b), L
            a, b = h.observables(), ref.observables()
            for k in b:
                assert np.array_equal(a[k], b[k]), (L, k)
