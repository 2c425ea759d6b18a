"""Which one-side batches run in clusters (XY_ALGO_AUTO, exact sums): n lattices of side L go to the
faster of the cluster and the whole-lattice kernel, as measured in rounds of ten sweeps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
@pytest.mark.parametrize("L,n,clusters", [
    (36, 41, False), (40, 8, False), (40, 64, False), (44, 16, False), (44, 41, False), (40, 1, True),
    (52, 100, False), (52, 41, True), (52, 1, True), (42, 41, True), (46, 64, True), (48, 41, True),
    (64, 16, True), (64, 152, False), (96, 16, True)])
def test_the_faster_kernel_is_taken(L, n, clusters, sincos):
    from paper_0811_2111_gb300.lattice import Batch
    betas = np.linspace(0.9, 1.2, n)
    with Batch([L] * n, betas, 5, sweeps_per_round=4, sincos=sincos) as b, \
            Batch([L] * n, betas, 5, sweeps_per_round=4, sincos=sincos, algorithm="two_pass") as ref:
        assert (b.info()[3] > 0) == clusters         # CTAs of clusters and bands
        b.run(2)
        ref.run(2)
        for i in (0, n // 2, n - 1):
            assert np.array_equal(b.state(i), ref.state(i))
            assert np.array_equal(b.observables(i)["C"], ref.observables(i)["C"])
