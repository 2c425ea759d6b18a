"""Sides that are no multiple of 128 on the persistent sweep's overlapping tiles (XY_ALGO_AUTO)
against the two-pass kernels: angles, accept counts and exact sums bit for bit, and the calls that
keep the two-pass kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(L, algorithm, calls, **kw):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3, algorithm=algorithm, **kw) as lat:
        for n in calls:
            lat.sweep(n)
        return lat.state()[0], lat.observables()


# the smallest overlap (a whole tile but two rows / columns) to the largest, rows of 16, 8 and
# 4-byte alignment (L % 8 = 0, 4, 2 and 6), two tile columns, and more tiles than resident CTAs
@pytest.mark.parametrize("L", [258, 260, 262, 264, 322, 382, 386, 508, 510, 514, 1000, 1022, 1026,
                               2564, 2566])
@pytest.mark.parametrize("sincos", ["accurate", "fast"])
def test_overlapping_tiles_equal_two_pass(L, sincos):
    a, oa = _run(L, "auto", (1, 2, 6), sincos=sincos)
    b, ob = _run(L, "two_pass", (9,), sincos=sincos)
    assert np.array_equal(a, b)
    for k in ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My"):
        assert np.array_equal(oa[k], ob[k]), k


def test_without_the_second_buffer_the_two_pass_kernels_run():
    from paper_0811_2111_gb300 import _lib as X
    from paper_0811_2111_gb300.lattice import Lattice
    X.lib().xy_debug_fail_alloc(2)      # the flag word is the first allocation
    with Lattice(300, 1.1, 9, lattice_id=3) as lat:
        X.lib().xy_debug_fail_alloc(0)
        lat.sweep(9)
        a, oa = lat.state()[0], lat.observables()
    b, ob = _run(300, "two_pass", (9,))
    assert np.array_equal(a, b) and np.array_equal(oa["C"], ob["C"])


def test_timed_and_compensated_runs_keep_the_two_pass_kernels():
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(300, 1.0, 2) as lat, Lattice(300, 1.0, 2, algorithm="two_pass") as ref:
        lat.sweep(3)                    # an odd count: the state moves back to its buffer
        lat.timing(1)
        lat.sweep(2)
        assert lat.kernel_time(0)[1] == 2 and lat.kernel_time(1)[1] == 2
        ref.sweep(5)
        assert np.array_equal(lat.state()[0], ref.state()[0])
    a, oa = _run(300, "auto", (3,), reduce="compensated")
    b, ob = _run(300, "two_pass", (3,), reduce="compensated")
    assert np.array_equal(a, b) and np.array_equal(oa["C"], ob["C"])


@pytest.mark.parametrize("L", [48, 300])
def test_captured_sweeps_replay(L):
    import torch
    from paper_0811_2111_gb300.lattice import Lattice
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        with Lattice(L, 1.0, 3, stream=s) as lat, \
                Lattice(L, 1.0, 3, algorithm="two_pass", stream=s) as ref:
            lat.reserve(8)
            lat.sweep(1)
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lat.sweep(3)
            g.replay()
            ref.sweep(4)
            assert np.array_equal(lat.state()[0], ref.state()[0])


def test_a_large_state_lands_whole_in_a_fresh_array():
    """State read into an array whose pages do not exist yet (touched in parallel first)."""
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(1536, 1.0, 3) as lat:
        a = lat.state()[0]
        b = np.full((1536, 1536), 7.0, np.float32)
        import ctypes as C
        from paper_0811_2111_gb300 import _lib as X
        X.xy_get_state(lat.ctx, b.ctypes.data_as(C.c_void_p))
        assert np.array_equal(a, b)
