"""The z-marching walks at the sizes and link phases where they change course (GPU):
the FP64 step and its ranges of sine and cosine, the FP32 step from copied planes
(rows that can be copied in 16 bytes, ragged tiles, several z chunks, wrapped
windows), the whole-lattice diagnostics and its winding turns, and batches that
mix lattices of the two FP32 walks.  Against the oracle with the tolerances of the
parity tests: fields 1e-12 (FP64) and 1e-5 (FP32), sums as compare_obs, windings
exactly."""
import numpy as np
import pytest

import oracle as O
import paper_1809_00995_gb300 as ah
from inputs import random_state, straight_strings
from test_gpu_batch_serve import oracle_fields, short_config
from test_gpu_parity import TOL, compare_obs, oparams, rel_err, sim

pytestmark = pytest.mark.gpu

# link phases within the short polynomials, the middle and the long ones, past
# pi / 4 (reduced) and past several turns
AMPLITUDES = [0.015, 0.09, 0.18, 0.7, 3.0, 40.0]


@pytest.mark.parametrize("th_amp", AMPLITUDES)
@pytest.mark.parametrize("precision,name,N", [(ah.AH_FP64, "ty8_b2_w", n) for n in (4, 31, 33, 41)]
                         + [(ah.AH_FP32, "ty16_b2_w", n) for n in (40, 44, 64, 68, 100)])
def test_step_walk_matches_oracle(precision, name, N, th_amp):
    f = random_state(N, 7, th_amp=th_amp).astype(np.float32).astype(np.float64)
    wrap = th_amp == 3.0
    with sim(N, precision, ah.AH_KERNEL_FUSED, era=ah.AH_MATTER, s=1.0,
             flags=ah.AH_FLAG_WRAP_THETA if wrap else 0) as g:
        for k in range(g.info["n_variants"]):
            try:
                g.set_variant(k)
            except ah.AhError:
                continue
            if g.info["variant_name"] == name:
                break
        assert g.info["variant_name"] == name
        g.set_fields(f, 30)
        g.step(3)
        got = g.fields()
    ref = O.evolve(oparams(N, era=O.MATTER, s=1.0, wrap_theta=wrap), f, 30, 3)
    assert max(rel_err(got, ref)) <= TOL[precision]


@pytest.mark.parametrize("th_amp", AMPLITUDES + [200.0])
@pytest.mark.parametrize("precision,N", [(p, n) for p in (ah.AH_FP32, ah.AH_FP64) for n in (5, 31, 33, 42, 44)])
def test_diagnostics_walk_matches_oracle(precision, N, th_amp):
    f = random_state(N, 11, th_amp=th_amp).astype(np.float32).astype(np.float64)
    with sim(N, precision, ah.AH_KERNEL_FUSED) as g:
        g.set_fields(f, 12)
        compare_obs(g.observables(), O.observables(oparams(N), f, 12), precision)


def test_batch_of_both_walks():
    Ns, steps = [64, 20, 66, 68], 6
    cfgs = [short_config(N, ah.AH_RADIATION, 0.0, 60 + N, steps) for N in Ns]
    wins = [(i, 0, 0, 0, N, N, N) for i, N in enumerate(Ns)]
    _, st, fields = ah.ah_batch_run_ex(cfgs, wins)
    assert st["launches"] == 3 * steps              # two walks and the advance per step
    for c, got in zip(cfgs, fields):
        assert max(rel_err(got, oracle_fields(c, steps)[0])) <= TOL[ah.AH_FP32], c.N
    for i in (0, 1):
        _, st, alone = ah.ah_batch_run_ex([cfgs[i]], [(0, 0, 0, 0, Ns[i], Ns[i], Ns[i])])
        assert st["launches"] == 2 * steps
        np.testing.assert_array_equal(alone[0], fields[i])


@pytest.mark.parametrize("N,fused", [(64, 1), (68, 0)])
def test_deferred_observables_ride_only_on_small_lattices(N, fused):
    """Few pierced plaquettes, no flag: the two-step launch takes the pass up to 64^3,
    above it the separate pass runs, bit for bit that of ah_observables."""
    with ah.Sim(N, precision=ah.AH_FP32, era=ah.AH_RADIATION, seed=4, flags=ah.AH_FLAG_TWO_STEP) as g:
        g.set_fields(straight_strings(N, axis=1, x0=0.5, y0=0.25), 8)
        ref = g.observables()
        g.observables_start()
        g.step(2)
        got = g.observables_finish()
        assert g.info["fused_diag_passes"] == fused
    assert got["wind_abs_plane"] == ref["wind_abs_plane"] == [0, 4 * N, 0]
    assert got["gauss_max"] == ref["gauss_max"]
    assert fused or got["sums"] == ref["sums"]
