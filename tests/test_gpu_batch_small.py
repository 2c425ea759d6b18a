"""Whole-lattice batches (sides whose lattice fits one CTA's shared memory) in each precision and sum:
packed or scalar pairs (L % 4 == 0) and single sites, several pairs a thread and fewer pairs than
threads, against the two-pass single lattice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDES = [4, 6, 16, 30, 32, 46, 48, 64, 66, 92, 96]


@pytest.mark.parametrize("reduce", ["exact", "compensated"])
@pytest.mark.parametrize("sincos", ["accurate", "fast", "libm"])
def test_whole_lattices_equal_the_single_lattice(sincos, reduce):
    from paper_0811_2111_gb300.lattice import Batch, Lattice
    betas = list(np.linspace(0.8, 1.3, len(SIDES)))
    with Batch(SIDES, betas, 21, sweeps_per_round=3, sincos=sincos, reduce=reduce,
               lattice_id0=4) as b:
        b.run(3)                                # both parities of the first sweep
        for i, L in enumerate(SIDES):
            with Lattice(L, betas[i], 21, lattice_id=4 + i, sincos=sincos, reduce=reduce,
                         algorithm="two_pass") as ref:
                ref.sweep(9)
                assert np.array_equal(b.state(i), ref.state()[0]), L
                o, r = b.observables(i), ref.observables()
                assert np.array_equal(o["accepted"], r["accepted"]), L
                for k in ("C", "Ix", "Iy", "Mx", "My"):
                    if reduce == "exact":
                        assert np.array_equal(o[k], r[k]), (L, k)
                    else:               # two FP32 groupings of the same terms, 2e-3 sqrt(N / 1024) each
                        tol = 4e-3 * max(1.0, L / 32)
                        assert np.abs(o[k] - r[k]).max() <= tol, (L, k)
