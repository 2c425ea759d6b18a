"""HMC's two steps per launch by rows (AUTO from L = 1792, from 1500 where the side is no multiple of
128) against the per-site kernel: angles, momenta, records, dH, counters and plain integrations bit
for bit."""
import numpy as np
import pytest

from test_gpu_hmc_auto import _chain

pytestmark = pytest.mark.gpu


# the first sides of each rule, rows of 16, 8 and 4-byte accesses (L % 4 = 0, 2, odd), a last strip
# of one access and of a whole strip (L % 120 = 0, 4, 2, 1), a last segment of few rows
@pytest.mark.parametrize("L", [1500, 1501, 1502, 1560, 1564, 1562, 1681, 1792, 1920, 2048, 2177, 3000])
@pytest.mark.parametrize("sincos,eps,n_md", [("accurate", 0.1, 8), ("fast", 0.05, 3),
                                             ("libm", 0.1, 4)])
def test_rows_equal_the_per_site_kernel(L, sincos, eps, n_md):
    a = _chain(L, "auto", sincos, eps, n_md, (1, 2))
    b = _chain(L, "site", sincos, eps, n_md, (3,))
    for k in b[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    for i in (1, 4):
        assert np.array_equal(a[i][0], b[i][0]) and np.array_equal(a[i][1], b[i][1])
        assert a[i][2] == b[i][2]
    assert a[2] == b[2] and a[3] == b[3] and a[5] == b[5]
