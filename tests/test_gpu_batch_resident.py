"""Batches whose lattices AUTO's default plan holds on the chip (one cluster each), against the
explicit tile / whole-lattice / band paths: states, records and exchange bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(Ls, betas, ladders, rounds, spr, **kw):
    from paper_0811_2111_gb300.lattice import Batch
    with Batch(Ls, betas, 23, ladders=ladders, lattice_id0=5, sweeps_per_round=spr, **kw) as b:
        for n in rounds:
            b.run(n)
        return ([b.state(i) for i in range(b.n)], [b.observables(i) for i in range(b.n)],
                b.betas(), b.exchange_stats(), b.info()[3])


# one side in the batch: one, eight and sixteen CTAs, L / 2 odd, more clusters than run at a time;
# mixed sides: only those that would be banded are held
@pytest.mark.parametrize("Ls", [[34] * 5, [64] * 9, [96] * 3, [128] * 2, [256] * 2, [98] * 30,
                                [130] * 7, [250] * 12, [16, 100, 130, 254, 128, 100]])
@pytest.mark.parametrize("sincos", ["accurate", "fast"])
def test_resident_batches_equal_the_other_paths(Ls, sincos):
    betas = [0.8 + 0.02 * i for i in range(len(Ls))]
    ladders = [0] * len(Ls) if len(set(Ls)) == 1 else None
    a = _run(Ls, betas, ladders, (1, 2), 5, sincos=sincos)
    b = _run(Ls, betas, ladders, (3,), 5, sincos=sincos, algorithm="fused")
    assert a[4] != b[4] or set(Ls) == {34}          # clusters in the plan (L = 34: may be whole)
    for x, y in zip(a[0], b[0]):
        assert np.array_equal(x, y)
    for x, y in zip(a[1], b[1]):
        for k in x:
            assert np.array_equal(x[k], y[k]), k
    assert np.array_equal(a[2], b[2])
    for x, y in zip(a[3], b[3]):
        assert np.array_equal(x, y)
