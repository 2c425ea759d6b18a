"""The kernels that take over where a cooperative launch finds no room (the refusal made on the
host): which they are, and that angles, accept counts and exact sums are bit for bit the same, also
when later launches of the same context go through."""
import numpy as np
import pytest

from paper_0811_2111_gb300 import _lib as X

KEYS = ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My")


@pytest.fixture
def refuse():
    yield X.lib().xy_debug_fail_cooperative
    X.lib().xy_debug_fail_cooperative(0)


def test_hook_refuses_negative_counts(refuse):
    assert refuse(-1) == X.XY_EINVAL
    assert refuse(0) == X.XY_OK


@pytest.mark.gpu
@pytest.mark.parametrize("L,kernel,instead", [
    (130, "grid", "two_pass"), (512, "grid", "two_pass"), (1282, "overlap", "two_pass"),
    (1300, "overlap", "two_pass"), (1408, "persistent", "fused")])
def test_lattice(refuse, L, kernel, instead):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3) as lat, \
            Lattice(L, 1.1, 9, lattice_id=3, algorithm="two_pass") as ref:
        for n, refused in ((2, False), (3, True), (1, False), (2, True), (2, False)):
            refuse(1 if refused else 0)
            lat.sweep(n)
            assert lat.kernel == (instead if refused else kernel)
        ref.sweep(10)
        assert np.array_equal(lat.state()[0], ref.state()[0])
        a, b = lat.observables(), ref.observables()
        for k in KEYS:
            assert np.array_equal(a[k], b[k]), k


# four, two and one replicas at a time, and the persistent tiles
@pytest.mark.gpu
@pytest.mark.parametrize("L,kernel,instead", [
    (64, "grid", "two_pass"), (130, "grid", "two_pass"), (500, "grid", "two_pass"),
    (768, "grid", "two_pass"), (1030, "grid", "two_pass"), (1312, "persistent", "fused")])
def test_quad(refuse, L, kernel, instead):
    from paper_0811_2111_gb300.lattice import Quad
    betas = [0.9, 1.0, 1.1, 1.2]
    with Quad(L, betas, 17, lattice_id=5) as q, \
            Quad(L, betas, 17, lattice_id=5, algorithm="two_pass") as ref:
        for n, refused in ((2, False), (3, True), (1, False), (2, True), (2, False)):
            refuse(1 if refused else 0)
            q.sweep(n)
            assert q.kernel == (instead if refused else kernel)
        ref.sweep(10)
        for r in range(4):
            assert np.array_equal(q.state(r)[0], ref.state(r)[0])
            a, b = q.observables(r), ref.observables(r)
            for k in KEYS:
                assert np.array_equal(a[k], b[k]), k


@pytest.mark.gpu
def test_an_explicit_persistent_sweep_reports_it(refuse):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(256, 1.0, 1, algorithm="persistent") as lat:
        refuse(1)
        with pytest.raises(X.XYError) as e:
            lat.sweep(1)
        assert e.value.status == X.XY_ECUDA
