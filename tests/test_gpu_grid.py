"""Middling lattices whose tiles stay with their CTAs (XY_ALGO_AUTO, 128 < L <= 1280) against the
two-pass kernels: angles, accept counts and exact sums bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("accepted", "beta", "C", "Ix", "Iy", "Mx", "My")


def _run(L, algorithm, calls, **kw):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.1, 9, lattice_id=3, algorithm=algorithm, **kw) as lat:
        for n in calls:
            lat.sweep(n)
        return lat.state()[0], lat.observables()


def _same(a, b):
    assert np.array_equal(a[0], b[0])
    for k in KEYS:
        assert np.array_equal(a[1][k], b[1][k]), k


# every shape (one row a warp, few and many threads; two rows; four), tiles of uneven width and
# height, W odd (L % 4 == 2), rows that do not fill the last warp
@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
@pytest.mark.parametrize("L", [130, 132, 134, 252, 260, 510, 512, 542, 546, 600, 702, 704, 766, 768,
                               1000, 1002, 1024, 1026, 1030, 1150, 1152, 1278, 1280, 1282])
def test_tiles_on_the_chip_equal_two_pass(L, sincos):
    _same(_run(L, "auto", (1, 2, 6), sincos=sincos), _run(L, "two_pass", (9,), sincos=sincos))


@pytest.mark.parametrize("L", [200, 258, 322, 512, 514, 1026])
def test_without_the_exchange_words_the_other_kernels_run(L):
    from paper_0811_2111_gb300 import _lib as X
    from paper_0811_2111_gb300.lattice import Lattice
    ref = _run(L, "two_pass", (5,))
    X.lib().xy_debug_fail_alloc(2)      # the flag word is the first allocation
    with Lattice(L, 1.1, 9, lattice_id=3) as lat:
        X.lib().xy_debug_fail_alloc(0)
        lat.sweep(5)
        _same((lat.state()[0], lat.observables()), ref)


def test_a_captured_launch_replays_and_launches_mix():
    import torch
    from paper_0811_2111_gb300.lattice import Lattice
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        with Lattice(512, 1.0, 3, stream=s) as lat, \
                Lattice(512, 1.0, 3, algorithm="two_pass", stream=s) as ref:
            lat.reserve(16)
            lat.sweep(1)
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lat.sweep(3)            # sweeps 1 .. 3 whenever it is replayed
            g.replay()
            ref.sweep(4)
            assert np.array_equal(lat.state()[0], ref.state()[0])
            lat.sweep(2)
            ref.sweep(2)
            assert np.array_equal(lat.state()[0], ref.state()[0])


def test_two_lattices_on_two_streams():
    import torch
    from paper_0811_2111_gb300.lattice import Lattice
    streams = [torch.cuda.Stream() for _ in range(2)]
    lats = [Lattice(L, 1.0, 3, stream=s) for L, s in zip((512, 1024), streams)]
    for _ in range(5):
        for lat in lats:
            lat.sweep(40)
    got = [lat.state()[0] for lat in lats]
    for lat in lats:
        lat.close()
    for L, a in zip((512, 1024), got):
        with Lattice(L, 1.0, 3, algorithm="two_pass") as ref:
            ref.sweep(200)
            assert np.array_equal(a, ref.state()[0])
