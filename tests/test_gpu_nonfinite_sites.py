"""Sites that are not numbers (GPU): one NaN component of phi leaves the plaquettes of
its site to the FP64 formula, whose counts the EXACT_DIAG pass gives."""
import numpy as np
import pytest

import paper_1809_00995_gb300 as ah
from inputs import random_state
from test_gpu_parity import sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("component", [0, 1])
@pytest.mark.parametrize("precision,N", [(p, n) for p in (ah.AH_FP32, ah.AH_FP64) for n in (33, 44)])
def test_one_nan_component_of_phi(precision, N, component):
    f = random_state(N, 8).astype(np.float32).astype(np.float64)
    for k, (z, y, x) in enumerate([(3, 7, 9), (8, 15, 31), (0, 0, 0), (N - 1, N - 1, N - 1)]):
        f[component, z, y, x] = np.nan
        f[1 - component, z, y, x] = (0.5, -0.5)[k % 2]
    got = []
    for flags in (0, ah.AH_FLAG_EXACT_DIAG):
        with sim(N, precision, ah.AH_KERNEL_FUSED, flags=flags) as g:
            g.set_fields(f, 6)
            got.append(g.observables(check_finite=False))
    fast, exact = got
    assert exact["nonfinite"] > 0
    assert list(fast["wind_abs_plane"]) == list(exact["wind_abs_plane"])
    assert list(fast["wind_plane"]) == list(exact["wind_plane"])
    assert fast["n_pierced"] == exact["n_pierced"]
