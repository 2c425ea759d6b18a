"""Overlapping tiles (XY_ALGO_AUTO, exact sums, L no multiple of 128) where they are what runs,
above the sides that are held on the chip and below without the exchange words, against the
two-pass kernels: angles, accept counts and exact sums bit for bit."""
import numpy as np
import pytest

from paper_0811_2111_gb300 import _lib as X

pytestmark = pytest.mark.gpu


def _result(lat, calls):
    for n in calls:
        lat.sweep(n)
    return lat.state()[0], lat.observables()


def _two_pass(L, sweeps, **kw):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3, algorithm="two_pass", **kw) as lat:
        return _result(lat, (sweeps,))


def _same(a, b):
    assert np.array_equal(a[0], b[0])
    for k in ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My"):
        assert np.array_equal(a[1][k], b[1][k]), k


# rows of 4, 8 and 16 byte alignment (L % 8 = 2 or 6, 4, 0) at two CTAs per SM (to four tiles per SM:
# 608 on 152 SMs, L = 1538) and three; overlaps of two to 62 columns and of two to 30 rows
@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
@pytest.mark.parametrize("L", [1282, 1284, 1288, 1302, 1340, 1376, 1406, 1500, 1504, 1532, 1534, 1544,
                               1546, 1660, 2000, 2002, 2004, 2046])
def test_overlapping_tiles_equal_two_pass(L, sincos):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3, sincos=sincos) as lat:
        got = _result(lat, (1, 2, 3))
        assert lat.kernel == "overlap"
    _same(got, _two_pass(L, 6, sincos=sincos))


# the smallest sides, where a row or column of tiles is one or two of them
@pytest.mark.parametrize("sincos", ["accurate", "libm"])
@pytest.mark.parametrize("L", [258, 260, 264, 288, 382, 508, 516, 520])
def test_small_sides_without_the_exchange_words(L, sincos):
    from paper_0811_2111_gb300.lattice import Lattice
    X.lib().xy_debug_fail_alloc(2)          # the flag word is the first allocation
    with Lattice(L, 1.1, 9, lattice_id=3, sincos=sincos) as lat:
        X.lib().xy_debug_fail_alloc(0)
        got = _result(lat, (1, 2, 6))
        assert lat.kernel == "overlap"
    _same(got, _two_pass(L, 9, sincos=sincos))


@pytest.mark.parametrize("L", [1282, 1300, 2000])
def test_without_the_second_buffer_the_two_pass_kernels_run(L):
    from paper_0811_2111_gb300.lattice import Lattice
    X.lib().xy_debug_fail_alloc(2)          # (above 1280 no exchange words are asked for)
    with Lattice(L, 1.1, 9, lattice_id=3) as lat:
        X.lib().xy_debug_fail_alloc(0)
        got = _result(lat, (4,))
        assert lat.kernel == "two_pass"
    _same(got, _two_pass(L, 4))


def test_the_cluster_takes_a_side_up_to_256_without_the_exchange_words():
    from paper_0811_2111_gb300.lattice import Lattice
    for L in (130, 190, 254, 256):
        X.lib().xy_debug_fail_alloc(2)
        # (L = 256 needs its second buffer besides: the third allocation)
        with Lattice(L, 1.1, 9, lattice_id=3) as lat:
            X.lib().xy_debug_fail_alloc(0)
            got = _result(lat, (2, 3))
            assert lat.kernel == "cluster"
        _same(got, _two_pass(L, 5))


@pytest.mark.parametrize("L", [1300, 1302])
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
            assert lat.kernel == "overlap"
            g.replay()
            ref.sweep(4)
            assert np.array_equal(lat.state()[0], ref.state()[0])
            lat.sweep(2)
            ref.sweep(2)
            assert np.array_equal(lat.state()[0], ref.state()[0])


def test_the_second_buffer_is_the_scratch_of_a_read_back():
    """A state goes to the host and back without another L*L floats."""
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(1300, 1.1, 9, lattice_id=3) as lat:
        lat.reserve(8)
        lat.sweep(3)                        # odd: the state moves back to its buffer
        assert lat.kernel == "overlap"
        X.lib().xy_debug_fail_alloc(1)
        try:
            th, t = lat.state()
            lat.sweep(2)
            lat.set_state(th, t)
            lat.sweep(2)
            got = lat.state()[0]
        finally:
            X.lib().xy_debug_fail_alloc(0)
    assert np.array_equal(th, _two_pass(1300, 3)[0])
    assert np.array_equal(got, _two_pass(1300, 5)[0])
