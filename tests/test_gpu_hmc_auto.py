"""HMC's AUTO paths -- many trajectories per cluster launch on small sides, two steps per launch
on overlapping tiles on large ones -- against the per-site kernel: angles, momenta, records, dH,
counters and plain integrations bit for bit (every sum is an exact integer)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _chain(L, kernel, sincos, eps, n_md, runs):
    from paper_0811_2111_gb300.hmc import HMC
    with HMC(L, 1.1, 9, eps, n_md, sincos=sincos, lattice_id=3, kernel=kernel) as h:
        for n in runs:
            h.run(n)
        out = [h.observables(), h.state(), h.info(), h.last_sums()]
        h.refresh()
        h.integrate(5)
        return out + [h.state(), h.last_sums()]


# one, eight and sixteen CTAs, one and two pairs a thread, odd sides, uneven strips; per-site
# sides; overlapping tiles of 16, 8 and 4-byte rows, the smallest and nearly whole overlaps
@pytest.mark.parametrize("L", [4, 5, 25, 32, 33, 63, 64, 65, 100, 127, 128, 160, 175, 176, 177, 256,
                               352, 385, 386, 510, 513, 1001])
@pytest.mark.parametrize("sincos,eps,n_md", [("accurate", 0.3, 7), ("accurate", 0.05, 1),
                                             ("fast", 0.3, 6), ("libm", 0.3, 2)])
def test_auto_equals_the_per_site_kernel(L, sincos, eps, n_md):
    a = _chain(L, "auto", sincos, eps, n_md, (1, 2, 5))
    b = _chain(L, "site", sincos, eps, n_md, (8,))
    for k in b[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    for i in (1, 4):
        assert np.array_equal(a[i][0], b[i][0]) and np.array_equal(a[i][1], b[i][1])
        assert a[i][2] == b[i][2]
    assert a[2] == b[2] and a[3] == b[3] and a[5] == b[5]


def test_rejections_restore_the_state():
    """A step far too long: both kinds of decision occur, and agree."""
    a = _chain(48, "auto", "accurate", 0.55, 6, (40,))
    b = _chain(48, "site", "accurate", 0.55, 6, (40,))
    acc = b[0]["accepted"]
    assert 0 < acc.sum() < 40
    assert np.array_equal(a[0]["accepted"], acc) and np.array_equal(a[0]["dH"], b[0]["dH"])
    assert np.array_equal(a[1][0], b[1][0])
