"""The FP32 step from copied planes and the diagnostics bit for bit (GPU): the value of
a site does not depend on how the lattice was cut into pieces, which other lattices
run, or on the run."""
import numpy as np
import pytest

import paper_1809_00995_gb300 as ah
from inputs import random_state

pytestmark = pytest.mark.gpu


def test_batched_lattice_equals_the_simulation_in_any_mix():
    """Strong plaquettes (e0 = 2), where the sines of some are reduced and of others
    not: 64^3 alone (short chunks of planes), in a mix (longer ones) and stepped by
    ah_step gives the same fields."""
    kw = dict(era=ah.AH_RADIATION, s=0.0, e0=2.0)
    cfg = ah.config(64, seed=21, **kw)
    steps = int(round((cfg.tau_end - cfg.tau0) / cfg.dt))
    with ah.Sim(64, seed=21, **kw) as g:
        g.step(steps)
        ref = g.fields()
    for others in ([], [68, 128], [192, 20]):
        cfgs = [cfg] + [ah.config(N, seed=N, tau_end=cfg.tau_end, **kw) for N in others]
        _, _, fields = ah.ah_batch_run_ex(cfgs, [(0, 0, 0, 0, 64, 64, 64)])
        np.testing.assert_array_equal(fields[0], ref, err_msg=str(others))


@pytest.mark.parametrize("th_amp", [0.2, 0.9, 30.0])
@pytest.mark.parametrize("N", [64, 100])
def test_steps_and_sums_repeat(N, th_amp):
    """The same steps and passes twice, and from a checkpoint half way."""
    f = random_state(N, N, th_amp=th_amp)
    runs = []
    for half in (False, False, True):
        with ah.Sim(N, era=ah.AH_RADIATION, s=0.0) as g:
            g.set_fields(f, 30)
            if half:
                g.step(3)
                mid = g.fields()
                g.set_fields(np.zeros_like(mid), 0)
                g.set_fields(mid, 33)
                g.step(3)
            else:
                g.step(6)
            first = g.observables()
            for _ in range(3):
                again = g.observables()
                assert again["sums"] == first["sums"] and again["gauss_max"] == first["gauss_max"]
                assert again["wind_plane"] == first["wind_plane"] and again["n_pierced"] == first["n_pierced"]
            runs.append((g.fields(), first["sums"]))
    for fields, sums in runs[1:]:
        np.testing.assert_array_equal(fields, runs[0][0])
        assert sums == runs[0][1]
