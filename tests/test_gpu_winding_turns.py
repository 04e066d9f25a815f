"""Windings at link phases of many turns and at fields of any size (GPU): the
whole-lattice pass counts what the FP64 formula counts, and takes no longer for it.  Sides of the one-row and of the
two-row walk, each with ragged tiles."""
import time

import numpy as np
import pytest

import oracle as O
import paper_1809_00995_gb300 as ah
from inputs import random_state
from test_gpu_parity import oparams, sim

pytestmark = pytest.mark.gpu

WALKS = [(p, n) for p in (ah.AH_FP32, ah.AH_FP64) for n in (33, 44)]
TURN = 2 * np.pi


def same_windings(N, precision, f, step, size=1.0):
    """The windings of f, phi and Pi times `size`, are the oracle's of f."""
    if precision == ah.AH_FP32:
        f = f.astype(np.float32).astype(np.float64)
    scaled = f.copy()
    scaled[0:4] *= size
    with sim(N, precision, ah.AH_KERNEL_FUSED) as g:
        g.set_fields(scaled, step)
        go = g.observables()
    oo = O.observables(oparams(N), f, step)
    assert list(go["wind_abs_plane"]) == list(oo["sum_abs_W_plane"])
    assert list(go["wind_plane"]) == list(oo["sum_W_plane"])
    assert go["n_pierced"] == oo["n_pierced"]


def pass_time(N, precision, f):
    with sim(N, precision, ah.AH_KERNEL_FUSED) as g:
        g.set_fields(f, 6)
        g.observables()
        runs = []
        for _ in range(9):
            t0 = time.perf_counter()
            g.observables()
            runs.append(time.perf_counter() - t0)
        return min(runs)


@pytest.mark.parametrize("precision,N", WALKS)
def test_turns_of_single_links_stay_in_their_plaquette(precision, N):
    """A link of 150 turns in a plaquette of 90: the other plaquettes of the same
    sites, whose links make tens of turns, keep their windings."""
    f = random_state(N, 5, th_amp=0.0)
    for z, y, x in [(5, 4, 3), (9, 15, 30), (N - 1, N - 1, N - 1)]:
        xp, yp = (x + 1) % N, (y + 1) % N
        f[5, z, y, xp] = 150 * TURN
        f[4, z, y, x] = -20 * TURN
        f[4, z, yp, x] = f[5, z, y, x] = 20 * TURN
    same_windings(N, precision, f, 6)


# phases of up to 160, 1600, 4800 and 1.6e5 turns: within and past the limit of the walks' own count
@pytest.mark.parametrize("th_amp", [1e3, 1e4, 3e4, 1e6])
@pytest.mark.parametrize("precision,N", WALKS)
def test_windings_at_many_turns(precision, N, th_amp):
    same_windings(N, precision, random_state(N, 17, th_amp=th_amp), 6)


@pytest.mark.parametrize("precision,N", [(ah.AH_FP32, 126), (ah.AH_FP32, 128), (ah.AH_FP64, 64)])
def test_many_turns_take_no_recount(precision, N):
    """Phases of up to 32 turns leave the plaquettes near a cut alone to the FP64
    list: the pass takes about as long as with phases of half a turn (a recount of
    every plaquette takes 8 times as long or more)."""
    t = [pass_time(N, precision, random_state(N, 3, th_amp=th_amp)) for th_amp in (3.0, 200.0)]
    print("\n%d^3, precision %d: %.0f us, %.0f us" % (N, precision, t[0] * 1e6, t[1] * 1e6))
    assert t[1] <= 2.0 * t[0]


@pytest.mark.parametrize("size", [1e-60, 1e60])
def test_fp64_fields_past_the_range_of_fp32(size):
    """The phase of a site does not ask for the size of phi: the same windings, in about
    the same time."""
    same_windings(33, ah.AH_FP64, random_state(33, 19), 6, size)
    f = random_state(64, 3)
    t = [pass_time(64, ah.AH_FP64, f)]
    f[0:4] *= size
    t.append(pass_time(64, ah.AH_FP64, f))
    print("\n%.0f us, %.0f us" % (t[0] * 1e6, t[1] * 1e6))
    assert t[1] <= 2.0 * t[0]
