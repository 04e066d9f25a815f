"""Weak plaquettes between large link phases (GPU): Xi is a small difference of large
phases (a gauge-rotated or long non-compact run), and its sine and 1 - cos Xi come
out as for small phases.  The reference is the phases' own exact sum in extended
precision."""
import numpy as np
import pytest

import paper_1809_00995_gb300 as ah
from test_gpu_parity import sim

pytestmark = pytest.mark.gpu


def links(N, amp, weak, seed):
    """theta of a random gauge of amplitude amp plus links of at most `weak`."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lam = rng.uniform(-amp, amp, size=(N, N, N))
    th = np.stack([np.roll(lam, -1, axis=2 - d) - lam for d in range(3)])
    return th + rng.uniform(-weak, weak, size=th.shape)


def plaquettes(th):
    """{(i, j): Xi_ij} (Eq. 3), exact to 2^-64 of the phases."""
    th = th.astype(np.longdouble)
    up = lambda a, d: np.roll(a, -1, axis=2 - d)      # noqa: E731
    return {(i, j): (th[i] - up(th[i], j)) + (up(th[j], i) - th[j]) for i, j in ((0, 1), (0, 2), (1, 2))}


# Sine of a plaquette in units of 2^-24 (FP32) or 2^-53 (FP64), |Xi| <= 0.25: phases apart by
# less than 0.78 lose half a unit in the last place of three sums (1.2 in all), the
# polynomial 0.5, larger ones less, since the sums' errors are kept.  Four of them,
# three sums of at most 1 and two products: below 12 units, 16 are allowed.  Phases past
# 2^17 (FP32) and 2^20 (FP64) go through products of four link exponentials, each good
# to 1.5 units: 10 units a sine, 64 allowed for the four.
@pytest.mark.parametrize("amp,units", [(0.3, 16), (3.0, 16), (40.0, 16), (3e3, 16), (None, 64)])
@pytest.mark.parametrize("precision,N", [(ah.AH_FP32, 64), (ah.AH_FP64, 33)])
def test_curl_of_weak_plaquettes(precision, N, amp, units):
    """phi = Pi = E = 0: after one step E = -c curl, c the step's coefficient."""
    f = np.zeros((10, N, N, N))
    if amp is None:
        amp = 3e5 if precision == ah.AH_FP32 else 3e6
    f[4:7] = links(N, amp, 0.05, 7)
    if precision == ah.AH_FP32:
        f = f.astype(np.float32).astype(np.float64)
    with sim(N, precision, ah.AH_KERNEL_FUSED) as g:
        g.set_fields(f, 30)
        g.step(1)
        e = g.fields()[7:10].astype(np.longdouble)
    s = {k: np.sin(x) for k, x in plaquettes(f[4:7]).items()}
    dn = lambda a, d: np.roll(a, 1, axis=2 - d)       # noqa: E731
    curl = np.stack([(s[0, 1] - dn(s[0, 1], 1)) + (s[0, 2] - dn(s[0, 2], 2)),
                     (dn(s[0, 1], 0) - s[0, 1]) + (s[1, 2] - dn(s[1, 2], 2)),
                     (dn(s[0, 2], 0) - s[0, 2]) + (dn(s[1, 2], 1) - s[1, 2])])
    c = -np.sum(e * curl) / np.sum(curl * curl)
    unit = 2.0 ** (-24 if precision == ah.AH_FP32 else -53)
    err = float(np.max(np.abs(e / c + curl)))
    print("\namp %g: %.2f units" % (amp, err / unit))
    assert err <= units * unit


# 1 - cos Xi = Xi^2 / 2: twice the relative error of Xi, which is that of the kept sums (3
# units), the polynomial and the coefficient (3 units), sums of positive terms
# compensated (FP32) or 200 terms deep (FP64).
@pytest.mark.parametrize("amp", [40.0, 3e3])
@pytest.mark.parametrize("precision,N,tol", [(ah.AH_FP32, 33, 2.0 ** -20), (ah.AH_FP32, 44, 2.0 ** -20),
                                             (ah.AH_FP64, 33, 2.0 ** -44), (ah.AH_FP64, 44, 2.0 ** -44)])
def test_magnetic_energy_of_a_rounded_pure_gauge(precision, N, tol, amp):
    """Every Xi is the rounding of its four phases, which the sum has to resolve; radiation
    era, s = 0, e0 = 1: B = dx^-4 sum (1 - cos Xi)."""
    f = np.zeros((10, N, N, N))
    f[0] = 1.0
    f[4:7] = links(N, amp, 0.0, 9)
    if precision == ah.AH_FP32:
        f = f.astype(np.float32).astype(np.float64)
    with sim(N, precision, ah.AH_KERNEL_FUSED) as g:
        g.set_fields(f, 6)
        got = g.observables()["sums"][7]
        dx = g.cfg.dx
    xi = plaquettes(f[4:7])
    ref = float(sum(np.sum(2 * np.sin(x / 2) ** 2) for x in xi.values())) / dx ** 4
    print("\namp %g: %.3g, relative error %.3g" % (amp, ref, got / ref - 1))
    assert abs(got - ref) <= tol * ref
