"""Four replicas held on the chip (XY_ALGO_AUTO, exact sums, 12 <= L <= 1280), four, two or one at a
time, against the two-pass kernels: angles, accept counts and sums of every replica bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BETAS = [0.9, 1.0, 1.1, 1.2]


def _run(L, algorithm, calls, **kw):
    from paper_0811_2111_gb300.lattice import Quad
    with Quad(L, BETAS, 17, lattice_id=5, algorithm=algorithm, **kw) as q:
        for n in calls:
            q.sweep(n)
        return [(q.state(r)[0], q.observables(r)) for r in range(4)]


def _same(a, b):
    for (sa, oa), (sb, ob) in zip(a, b):
        assert np.array_equal(sa, sb)
        for k in ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My"):
            assert np.array_equal(oa[k], ob[k]), k


# below and at the smallest side, one tile column and several, W odd, four / two / one replicas at a
# time, the largest side and one past it
@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
@pytest.mark.parametrize("L", [8, 12, 14, 16, 34, 64, 126, 128, 130, 256, 500, 512, 640, 702, 768, 770,
                               1000, 1024, 1030, 1280, 1282])
def test_replicas_on_the_chip_equal_two_pass(L, sincos):
    _same(_run(L, "auto", (1, 2, 3), sincos=sincos), _run(L, "two_pass", (6,), sincos=sincos))


@pytest.mark.parametrize("L", [64, 98])
def test_without_the_exchange_words_the_other_kernels_run(L):
    from paper_0811_2111_gb300 import _lib as X
    from paper_0811_2111_gb300.lattice import Quad
    ref = _run(L, "two_pass", (5,))
    X.lib().xy_debug_fail_alloc(4)      # after the state and the two scratch buffers
    with Quad(L, BETAS, 17, lattice_id=5) as q:
        X.lib().xy_debug_fail_alloc(0)
        q.sweep(5)
        _same([(q.state(r)[0], q.observables(r)) for r in range(4)], ref)
