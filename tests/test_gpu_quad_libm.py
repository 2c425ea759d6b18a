"""Four replicas with CUDA's sincosf, one launch per sweep: the packed kernel up to four waves of CTAs
(L = 1344 on 152 SMs) and the scalar one beyond, against the two-pass kernels: angles, accept
counts and exact sums of every replica bit for bit; compensated sums to their rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BETAS = [0.9, 1.0, 1.1, 1.2]


def _run(L, algorithm, calls, reduce):
    from paper_0811_2111_gb300.lattice import Quad
    with Quad(L, BETAS, 17, lattice_id=5, algorithm=algorithm, sincos="libm", reduce=reduce) as q:
        for n in calls:
            q.sweep(n)
        return q.kernel, [(q.state(r)[0], q.observables(r)) for r in range(4)]


@pytest.mark.parametrize("reduce", ["exact", "compensated"])
@pytest.mark.parametrize("L", [1344, 1376, 1632, 2048])
def test_one_launch_per_sweep_equals_two_pass(L, reduce):
    kernel, a = _run(L, "auto", (1, 2), reduce)
    assert kernel == "fused"
    _, b = _run(L, "two_pass", (3,), reduce)
    for (sa, oa), (sb, ob) in zip(a, b):
        assert np.array_equal(sa, sb)
        assert np.array_equal(oa["accepted"], ob["accepted"])
        for k in ("C", "Ix", "Iy", "Mx", "My"):
            if reduce == "exact":
                assert np.array_equal(oa[k], ob[k]), k
            else:                       # two FP32 groupings of the same terms, 2e-3 sqrt(N / 1024) each
                assert np.abs(oa[k] - ob[k]).max() <= 4e-3 * L / 32, k
