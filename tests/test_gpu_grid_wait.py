"""The failure path of the sweep that keeps its tiles on the chip, made on purpose without a fault:
one tile's CTA is not launched, so the bounded waits for its edge sites run out, every warp of the
others leaves, and the call reports XY_ETIMEOUT.  The device stays usable."""
import ctypes as C

import numpy as np
import pytest

from paper_0811_2111_gb300 import _lib as X

pytest.importorskip("torch")

SELFTESTS = [("xy_selftest_grid_wait", "xy_last_error"),
             ("xy_selftest_quad_grid_wait", "xy_quad_last_error")]


@pytest.mark.parametrize("name,error", SELFTESTS)
def test_polls_out_of_range_are_refused(name, error):
    for polls in (0, -1, (1 << 22) + 1):
        assert getattr(X.lib(), name)(None, polls) == X.XY_EINVAL
        assert b"polls must be in" in getattr(X.lib(), error)(None)


@pytest.mark.gpu
@pytest.mark.parametrize("polls", [1, 4096])
@pytest.mark.parametrize("name,error", SELFTESTS)
def test_waits_run_out_and_report_timeout(name, error, polls):
    import torch
    from paper_0811_2111_gb300.lattice import Lattice, Quad
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert getattr(X.lib(), name)(stream, polls) == X.XY_ETIMEOUT
    assert b"ran out" in getattr(X.lib(), error)(None)
    torch.cuda.synchronize()
    with Lattice(256, 1.0, 3) as lat, Lattice(256, 1.0, 3, algorithm="two_pass") as ref:
        lat.sweep(5)
        ref.sweep(5)
        assert np.array_equal(lat.state()[0], ref.state()[0])
        assert np.array_equal(lat.observables()["C"], ref.observables()["C"])
    betas = [0.9, 1.0, 1.1, 1.2]
    with Quad(64, betas, 3) as q, Quad(64, betas, 3, algorithm="two_pass") as ref:
        q.sweep(5)
        ref.sweep(5)
        for r in range(4):
            assert np.array_equal(q.state(r)[0], ref.state(r)[0])
            assert np.array_equal(q.observables(r)["C"], ref.observables(r)["C"])
