"""The front ends' read-back: observables as arrays of the C structs' fields."""
import numpy as np

from paper_0811_2111_gb300 import _lib as X


def test_obs_arrays_equal_the_fields():
    for n in (0, 1, 3):
        obs = (X.xy_obs * n)()
        for i, o in enumerate(obs):
            for j, (name, _) in enumerate(X.xy_obs._fields_):
                setattr(o, name, (1 << 63) + i if name == "accepted" else 10.0 * i + j)
        out = X.obs_arrays(obs)
        assert list(out) == list(X.OBS_NAMES)
        for name in X.OBS_NAMES:
            assert out[name].dtype == (np.uint64 if name == "accepted" else np.float64)
            assert out[name].flags.owndata and out[name].shape == (n,)
            assert [v for v in out[name].tolist()] == [getattr(o, name) for o in obs]
