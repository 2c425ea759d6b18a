"""The kernel that a sweep ran (xy_sweep_kernel): what AUTO takes by side, precision, sums and plan,
so that a test of a kernel can say which one it reached."""
import ctypes as C

import pytest

from paper_0811_2111_gb300 import _lib as X


def test_null_arguments():
    k = C.c_int32(-1)
    for f in (X.lib().xy_sweep_kernel, X.lib().xy_quad_sweep_kernel):
        assert f(None, C.byref(k)) == X.XY_EINVAL and k.value == -1


@pytest.mark.gpu
@pytest.mark.parametrize("L,kw,expected", [
    (2, {}, "two_pass"), (4, {}, "cluster"), (128, {}, "cluster"), (130, {}, "grid"),
    (1280, {}, "grid"), (1282, {}, "overlap"), (1408, {}, "persistent"), (4098, {}, "overlap"),
    (4224, {}, "fused"),
    (64, {"reduce": "compensated"}, "two_pass"), (512, {"reduce": "compensated"}, "persistent"),
    (512, {"ctas_per_sm": 3}, "persistent"), (300, {"ctas_per_sm": 3}, "two_pass"),
    (128, {"algorithm": "two_pass"}, "two_pass"), (256, {"algorithm": "persistent"}, "persistent"),
    (256, {"algorithm": "fused"}, "fused"), (256, {"algorithm": "fused2"}, "fused2")])
def test_lattice(L, kw, expected):
    from paper_0811_2111_gb300.lattice import Lattice
    with Lattice(L, 1.0, 1, **kw) as lat:
        assert lat.kernel is None
        lat.sweep(2)
        assert lat.kernel == expected


@pytest.mark.gpu
@pytest.mark.parametrize("L,kw,expected", [
    (8, {}, "two_pass"), (12, {}, "grid"), (672, {}, "grid"), (704, {}, "persistent"),
    (704, {"sincos": "libm"}, "grid"), (1024, {"sincos": "fast"}, "persistent"), (1280, {}, "grid"),
    (1536, {}, "persistent"), (1568, {}, "fused"), (1290, {}, "two_pass"),
    (64, {"reduce": "compensated"}, "persistent"), (64, {"algorithm": "fused"}, "fused"),
    (64, {"algorithm": "two_pass"}, "two_pass")])
def test_quad(L, kw, expected):
    from paper_0811_2111_gb300.lattice import Quad
    with Quad(L, [0.9, 1.0, 1.1, 1.2], 1, **kw) as q:
        assert q.kernel is None
        q.sweep(1)
        assert q.kernel == expected
