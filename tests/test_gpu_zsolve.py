"""The Stokes solve's transforms along z over the lengths: every radix and number of steps, columns that do not fill a
block, lengths that go to whole-grid transforms (other prime factors, too long), against the oracle."""
import pytest

from gpu_util import FP32_TOL, FP64_TOL, System, assert_parity, ensure_built, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Mz", [6, 8, 9, 10, 12, 14, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72,
                                75, 80, 81, 90, 96, 100, 108, 120, 125, 128, 135, 144, 150, 160, 180, 192, 200, 216, 225,
                                240, 243, 250, 256, 270, 288, 300, 22, 26, 98])
def test_zsolve_lengths(Mz):
    """The oracle's own transforms are good to FP64 rounding, as are these (a step multiplies rounded factors, log2 N of
    them): far inside the repository's FP64 and FP32 bars, which a wrong factor misses by its whole value."""
    fcm = ensure_built()
    Mxy = (9, 10) if Mz % 2 else (8, 14)
    L = (9.0, 11.0, 1.1 * Mz)
    for precision, tol in ((fcm.FCM_FP64, FP64_TOL), (fcm.FCM_FP32, FP32_TOL)):
        s = System(7, L, (Mxy[0], Mxy[1], Mz), 0.9, 6, 3.0, Mz)
        U, W = run_gpu(s, precision, stages=1)
        Uo, Wo = s.oracle(precision, stages=1)
        assert_parity(U, Uo, tol, f"U {Mz}")
        assert_parity(W, Wo, tol, f"W {Mz}")
