"""Lattices on the chip and on overlapping tiles hold their first 1024 records in the allocation that
they need anyway: reserving those allocates nothing, and growing past them keeps them."""
import numpy as np
import pytest

from paper_0811_2111_gb300 import _lib as X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,kernel", [(130, "grid"), (512, "grid"), (1282, "overlap"), (1300, "overlap")])
def test_first_records(L, kernel):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3) as lat, \
            Lattice(L, 1.1, 9, lattice_id=3, algorithm="two_pass") as ref:
        X.lib().xy_debug_fail_alloc(1)
        try:
            lat.reserve(1024)               # from what the lattice has already
            lat.sweep(3)
            assert lat.kernel == kernel
        finally:
            X.lib().xy_debug_fail_alloc(0)
        lat.reserve(5000)                   # moves the three records
        lat.sweep(2)
        ref.sweep(5)
        a, b = lat.observables(), ref.observables()
        for k in ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My"):
            assert np.array_equal(a[k], b[k]), k
        lat.reset(11)                       # clears them
        ref.reset(11)
        for x in (lat, ref):
            x.sweep(2)
        assert np.array_equal(lat.observables()["C"], ref.observables()["C"])
        assert np.array_equal(lat.state()[0], ref.state()[0])


def test_growth_that_fails_keeps_the_device_usable():
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(512, 1.0, 5) as lat:
        lat.sweep(1)
        X.lib().xy_debug_fail_alloc(1)
        try:
            with pytest.raises(X.XYError) as e:
                lat.reserve(1 << 16)
        finally:
            X.lib().xy_debug_fail_alloc(0)
        assert e.value.status == X.XY_ENOMEM
    with Lattice(512, 1.0, 5) as lat:
        lat.sweep(3)
        assert lat.observables()["accepted"].size == 3
