"""FP64 kernels at the sizes where they can go wrong, against the oracle."""
import numpy as np
import pytest

from gpu_util import FP64_TOL, System, assert_parity, ensure_built, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,r_c,torques", [
    (1, 20.0, 8.0, True),          # no pair
    (2, 20.0, 10.0, True),         # r_c = L/2, three cells per side
    (33, 30.0, 6.0, True),         # one more than a warp's queue can hold of own-cell pairs
    (700, 26.0, 12.9, True),       # three cells per side: every staged chunk of 512 is split
    (700, 26.0, 6.4, False),       # four cells per side
    (1500, (60.0, 40.0, 30.0), 7.4, True),   # different cells per side
])
def test_pair_f64(n, L, r_c, torques):
    """The half-shell pair kernel: cell counts, staged chunks, queue remainders. Each coefficient is good to
    about 1e-15 of the self mobility and a sum has at most n terms, so the repository's FP64 bar holds."""
    fcm = ensure_built()
    s = System(n, L, 32, 1.4, 8, r_c, 91 + n, torques=torques, min_sep=0.0 if n > 600 else 2.2)
    U, W = run_gpu(s, fcm.FCM_FP64, stages=2, want_W=torques)
    Uo, Wo = s.oracle(fcm.FCM_FP64, stages=2)
    assert_parity(U, Uo, FP64_TOL, f"U n={n}")
    if torques:
        assert_parity(W, Wo, FP64_TOL, f"W n={n}")


@pytest.mark.parametrize("r", [0.0, 0.05, 0.2818, 0.2822, 0.5, 1.0, 2.0, 4.0, 7.999, 8.001])
def test_pair_f64_separation(r):
    """One pair at separations around the Taylor branch (r = sigma/2 = 0.2821), interval ends and the cutoff (8),
    across a periodic face; a third particle out of reach carries the rest of the mean-free loads.
    (The reference's closed form loses about 1e-16 / r^3 to cancellation, so r = 0.05 is as close as it can judge.)"""
    fcm = ensure_built()
    L = 24.0
    Y = np.array([[0.1, 5.0, 23.9], [(0.1 - r * 0.6) % L, 5.0, (23.9 + r * 0.8) % L], [12.0, 17.0, 12.0]])
    s = System(3, L, 32, 1.4, 8, 8.0, 5, Y=Y)
    U, W = run_gpu(s, fcm.FCM_FP64, stages=2)
    Uo, Wo = s.oracle(fcm.FCM_FP64, stages=2)
    assert_parity(U, Uo, FP64_TOL, f"U r={r}")
    assert_parity(W, Wo, FP64_TOL, f"W r={r}")


@pytest.mark.parametrize("M_G", [1, 2, 7, 10, 14, 16, 17, 24])
@pytest.mark.parametrize("mode", ["forces", "one_width", "two_widths"])
def test_grid_f64(M_G, mode):
    """Spread and gather over the supports: rows that fill one round of threads, several, or part of a warp; the
    kernel with one Gaussian, with the torque's folded in, and with the torque's own width; windows that wrap."""
    fcm = ensure_built()
    s = System(40, (20.0, 24.0, 16.0), (32, 27, 24), 1.4, M_G, 6.0, 17, torques=mode != "forces",
               Sigma_D=1.7 if mode == "two_widths" else 0.0)
    U, W = run_gpu(s, fcm.FCM_FP64, stages=1, want_W=mode != "forces")
    Uo, Wo = s.oracle(fcm.FCM_FP64, stages=1)
    assert_parity(U, Uo, FP64_TOL, f"U M_G={M_G} {mode}")
    if mode != "forces":
        assert_parity(W, Wo, FP64_TOL, f"W M_G={M_G} {mode}")
