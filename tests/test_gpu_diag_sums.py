"""Precision of the whole-lattice sums of an FP32 state (GPU): the Gauss residual, and
what the sums keep of the single values."""
import numpy as np
import pytest

import paper_1809_00995_gb300 as ah
from inputs import random_state
from test_gpu_parity import sim

pytestmark = pytest.mark.gpu


def observables(N, f, flags=0):
    with sim(N, ah.AH_FP32, ah.AH_KERNEL_FUSED, flags=flags) as g:
        g.set_fields(f, 6)
        return g.observables(check_finite=False)


def cancelling_fields(N):
    """Pi = 0, E with E_3 chosen plane by plane so that div E is nothing but rounding;
    E_1, E_2 of the second half of the planes are minus those of the first."""
    rng = np.random.Generator(np.random.PCG64(4))
    f = random_state(N, 4)
    f[2:4] = 0.0
    e = np.zeros((3, N, N, N), dtype=np.float32)
    h = N // 2
    e[:2, :h] = rng.uniform(0.1, 0.3, size=(2, h, N, N)) * rng.choice([-1, 1], size=(2, h, N, N))
    e[:2, h:2 * h] = -e[:2, :h]
    e[2, N - 1] = rng.uniform(0.1, 0.3, size=(N, N))
    for z in range(N - 1):
        d = sum(e[k, z].astype(np.float64) - np.roll(e[k, z], 1, axis=1 - k) for k in range(2))
        e[2, z] = e[2, z - 1] - d
    f[7:10] = e
    return f.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("N", [33, 44])
def test_gauss_residual_of_cancelling_fields(N):
    """|G| to 2^-44 of its terms where they are small differences of large E: against
    the FP64 pass, whose differences of these values are exact."""
    f = cancelling_fields(N)
    fast, exact = observables(N, f), observables(N, f, flags=ah.AH_FLAG_EXACT_DIAG)
    print("\n%d^3: %.6g, relative error %.3g" % (N, exact["gauss_max"], fast["gauss_max"] / exact["gauss_max"] - 1))
    assert 0 < exact["gauss_max"] < 1e-5
    assert abs(fast["gauss_max"] - exact["gauss_max"]) <= 2.0 ** -44 * exact["gauss_max"]


@pytest.mark.parametrize("N", [33, 44])
def test_sums_take_every_row_by_itself(N):
    """K = 1 in even rows and 1 + 2^-23 in odd ones: every partial sum is a multiple of
    2^-23, so compensated sums are exact, and the FP64 total is to its own rounding."""
    f = np.zeros((10, N, N, N))
    f[0] = 1.0
    f[2] = 1.0
    f[3, :, 1::2] = np.float32(2.0 ** -11.5)
    got = observables(N, f)["sums"][3]
    odd = N // 2
    ref = N * N * (N + odd * 2.0 ** -23)
    print("\n%d^3: relative error %.3g" % (N, got / ref - 1))
    assert abs(got - ref) <= 2.0 ** -40 * ref
