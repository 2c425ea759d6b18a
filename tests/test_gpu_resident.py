"""Small lattices held on the chip (XY_ALGO_AUTO, 4 <= L <= 256) against the two-pass kernels.

Every algorithm makes bit-identical decisions and exact sums do not depend on the order of
addition, so angles, accept counts and sums are compared bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one CTA / eight / sixteen, one and two pairs per thread, uneven strips, W odd (L % 4 == 2)
SIDES = [4, 6, 10, 30, 32, 34, 36, 50, 62, 64, 66, 98, 128, 130, 182, 190, 254, 256]


def _run(L, algorithm, calls, **kw):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3, algorithm=algorithm, **kw) as lat:
        for n in calls:
            lat.sweep(n)
        return lat.state()[0], lat.observables()


@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
@pytest.mark.parametrize("L", SIDES)
def test_resident_equals_two_pass(L, sincos):
    a, oa = _run(L, "auto", (1, 2, 6), sincos=sincos)
    b, ob = _run(L, "two_pass", (9,), sincos=sincos)
    assert np.array_equal(a, b)
    for k in ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My"):
        assert np.array_equal(oa[k], ob[k]), k


def test_timing_runs_the_two_timed_kernels():
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(48, 1.0, 2) as lat, Lattice(48, 1.0, 2, algorithm="two_pass") as ref:
        lat.timing(1)
        lat.sweep(3)
        ref.sweep(3)
        assert lat.kernel_time(0)[1] == 3 and lat.kernel_time(1)[1] == 3
        lat.timing(0)
        lat.sweep(3)
        ref.sweep(3)
        assert np.array_equal(lat.state()[0], ref.state()[0])
        assert np.array_equal(lat.observables()["C"], ref.observables()["C"])


def test_a_planted_non_finite_angle_is_flagged():
    import torch
    from paper_0811_2111_gb300 import _lib as X
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(64, 1.0, 2) as lat:
        lat.angles[1234] = float("nan")
        torch.cuda.synchronize()
        lat.sweep(2)
        with pytest.raises(X.XYError):
            lat.observables()
