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


def noalloc(N, f, offset=0):
    """ah_observables_noalloc on buffers that start `offset` floats into their allocation."""
    torch = pytest.importorskip("torch")
    bufs = []
    for c in range(10):
        b = torch.zeros(N ** 3 + offset, dtype=torch.float32, device="cuda")
        b[offset:] = torch.from_numpy(f[c].astype(np.float32).ravel()).cuda()
        bufs.append(b[offset:])
    out = torch.full((26,), -1, dtype=torch.int64, device="cuda")
    cfg = ah.config(N, precision=ah.AH_FP32, era=ah.AH_RADIATION, s=0.0)
    ah.ah_observables_noalloc([b.data_ptr() for b in bufs], N, cfg, 6, out.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return ah.ah_sums.from_buffer_copy(out.cpu().numpy().tobytes())


# Gauss residual and its sums in FP64, as the call promises: the FP64 pass differs by the
# order of sums of some hundreds of positive terms per thread and by contractions.
# Uniform fields, where FP32 errors add up; random ones; E of 1e12, whose squares of
# G leave the range of FP32; Pi and E of 1e-25, and E below the normal range of FP32.
# Buffers on 8 bytes only take the one-row walk.
@pytest.mark.parametrize("state", ["uniform", "random", "huge", "cancelling", "tiny", "subnormal"])
@pytest.mark.parametrize("N,offset", [(33, 0), (44, 0), (44, 2)])
def test_noalloc_gauss_sums_are_fp64(N, offset, state):
    f = cancelling_fields(N) if state == "cancelling" else random_state(N, 4)
    if state == "uniform":
        f[0], f[1], f[2], f[3] = 0.7, 0.3, 0.2, -0.9
        f[7:10] = 0.1
    if state == "huge":
        f[7:10] *= 1e12
    if state == "tiny":
        f[2:4] *= 1e-25
        f[7:10] *= 1e-25
    if state == "subnormal":
        f[2:4] = 0.0
        f[7:10] *= 1e-39
    f = f.astype(np.float32).astype(np.float64)
    got, ref = noalloc(N, f, offset), observables(N, f, flags=ah.AH_FLAG_EXACT_DIAG)
    for k in (14, 15):
        print("\n%s sums[%d] %.6g, relative error %.3g" % (state, k, ref["sums"][k], got.sums[k] / ref["sums"][k] - 1))
        assert abs(got.sums[k] - ref["sums"][k]) <= 2.0 ** -43 * ref["sums"][k]
    assert abs(got.gauss_max - ref["gauss_max"]) <= 2.0 ** -48 * ref["gauss_max"]
    assert list(got.wind_abs_plane) == list(ref["wind_abs_plane"]) and got.n_pierced == ref["n_pierced"]


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("component", [3, 7])
@pytest.mark.parametrize("N,offset", [(33, 0), (44, 0), (44, 2)])
def test_noalloc_nonfinite_site_reaches_the_gauss_sums(N, offset, component, bad):
    """A Pi or E that is no number, at a site and as a backward neighbour: the sums and
    the maximum are those of the FP64 pass."""
    f = random_state(N, 4).astype(np.float32).astype(np.float64)
    f[component, 5, 7, 31] = f[component, N - 1, N - 1, N - 1] = bad
    got, ref = noalloc(N, f, offset), observables(N, f, flags=ah.AH_FLAG_EXACT_DIAG)
    assert got.nonfinite > 0 and ref["nonfinite"] > 0
    for k in (14, 15):
        np.testing.assert_equal(got.sums[k], ref["sums"][k])
        assert not np.isfinite(got.sums[k])
    if np.isfinite(ref["gauss_max"]):
        assert abs(got.gauss_max - ref["gauss_max"]) <= 2.0 ** -48 * ref["gauss_max"]
    else:
        np.testing.assert_equal(got.gauss_max, ref["gauss_max"])


@pytest.mark.parametrize("call", ["observables", "noalloc"])
@pytest.mark.parametrize("N", [33, 44])
def test_sums_take_every_row_by_itself(N, call):
    """K = 1 in even rows and 1 + 2^-23 in odd ones: every partial sum is a multiple of
    2^-23, so compensated sums are exact, and the FP64 total is to its own rounding."""
    f = np.zeros((10, N, N, N))
    f[0] = 1.0
    f[2] = 1.0
    f[3, :, 1::2] = np.float32(2.0 ** -11.5)
    got = (noalloc(N, f).sums if call == "noalloc" else observables(N, f)["sums"])[3]
    odd = N // 2
    ref = N * N * (N + odd * 2.0 ** -23)
    print("\n%s %d^3: relative error %.3g" % (call, N, got / ref - 1))
    assert abs(got - ref) <= 2.0 ** -40 * ref
