"""The autotuner knows the library's default plan (GPU): for batches of one side, which only that
plan holds on the chip, and for the sides that are no multiple of 128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(64, 10), (128, 4)])
def test_a_one_side_batch_tries_the_default_plan(L, n):
    from paper_0811_2111_gb300 import autotune
    from paper_0811_2111_gb300.lattice import Batch
    betas = np.linspace(0.9, 1.2, n)
    plan = autotune.tune_batch([L] * n, betas, rounds=2, use_cache=False, group_ctas=(16, 128),
                               ctas_per_sm=(3,))
    times = plan.pop("ms_per_round")
    assert set(times) == {"16/3/8192", "128/3/8192", "0/0/0"}
    assert "/".join(str(plan[k]) for k in ("group_ctas", "ctas_per_sm", "target_band_sites")) == \
        min(times, key=times.get)
    # held on the chip: a few CTAs' worth of clusters and two launches a round
    with Batch([L] * n, betas, 9) as b, Batch([L] * n, betas, 9, **plan) as t, \
            Batch([L] * n, betas, 9, algorithm="two_pass") as ref:
        assert b.launches_per_round() == 2
        for x in (b, t, ref):
            x.run(2)
        for i in range(n):
            assert np.array_equal(b.state(i), ref.state(i))
            assert np.array_equal(t.state(i), ref.state(i))


@pytest.mark.parametrize("L", [100, 1000])
def test_candidates_of_other_sides_are_timed(L):
    from paper_0811_2111_gb300 import autotune
    plan = autotune.tune_lattice(L, sweeps=20, repeats=2, use_cache=False,
                                 candidates=autotune.OTHER_SIDE_CANDIDATES)
    times = plan["ms_per_sweep"]
    assert set(times) == {"auto/0", "two_pass/0"}
    assert f"{plan['algorithm']}/{plan['ctas_per_sm']}" == min(times, key=times.get)
