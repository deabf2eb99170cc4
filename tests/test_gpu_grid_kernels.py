"""Spread and gather alone over the supports each kernel variant takes and the layouts where the walk over tiles can go
wrong: two particles, tiles skipped along z and x, many particles in one tile, more than 32 tiles along z, ragged grids."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, System, assert_parity, ensure_built, run_gpu

pytestmark = pytest.mark.gpu

LAYOUTS = {
    "two": ((40, 44, 48), 2),
    "sparse": ((72, 40, 96), 6),
    "cluster": ((44, 48, 40), 500),
    "long_z": ((22, 24, 300), 400),
    "ragged": ((45, 50, 37), 300),
}


def _positions(layout, n, M, seed):
    rng = np.random.default_rng(seed)
    Y = rng.random((n, 3)) * M
    if layout == "sparse":   # a few tiles apart in z and x
        Y[:, 2] = (np.arange(n) * 17.3 + 3.1) % M[2]
        Y[:, 1] = 11.2
        Y[:, 0] = (np.arange(n) // 3) * 33.0 + 5.4
    if layout == "cluster":   # two thirds in one tile, the rest all over the grid
        Y[: 2 * n // 3] = 19.5 + 4.0 * rng.random((2 * n // 3, 3))
    return Y


@pytest.mark.parametrize("torques", [True, False])
@pytest.mark.parametrize("M_G", [7, 8, 9, 10, 12, 13, 14, 16])
@pytest.mark.parametrize("layout", list(LAYOUTS))
def test_spread_and_gather(layout, M_G, torques):
    """Grid part against the oracle at the repository's FP32 bar; a misplaced window or a plane read too early or too
    late is off by its whole value."""
    fcm = ensure_built()
    M, n = LAYOUTS[layout]
    Mv = np.array(M, dtype=np.float64)
    h = 1.1
    s = System(n, tuple(h * Mv), M, h * M_G / 9.0, M_G, 4.0, 5, torques=torques,
               Y=h * _positions(layout, n, Mv, 17 * M_G + n))
    U, W = run_gpu(s, fcm.FCM_FP32, stages=1, want_W=torques)
    Uo, Wo = s.oracle(fcm.FCM_FP32, stages=1)
    assert_parity(U, Uo, FP32_TOL, f"U {layout} {M_G}")
    if torques:
        assert_parity(W, Wo, FP32_TOL, f"W {layout} {M_G}")
