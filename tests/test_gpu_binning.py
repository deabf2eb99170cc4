"""The counting sort's scan where its blocks and chunks end: products on grids and cell lists of many sizes agree
with the FP64 kernels on the same inputs (the order of the particles is what the scan decides)."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, System, assert_parity, ensure_built, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,L,r_c,n", [
    (8, 20.0, 6.0, 3),            # one tile, 27 cells
    ((64, 64, 64), 90.0, 4.3, 900),       # 2,048 tile counters: exactly one chunk of the scan
    ((72, 64, 64), 90.0, 4.3, 900),       # one tile row more: a second chunk with a remainder
    ((250, 60, 36), (250.0, 60.0, 40.0), 2.9, 2500),   # ragged tiles, thousands of cells
    ((416, 320, 160), (416.0, 320.0, 160.0), 3.0, 5000),   # 166,400 counters and 810,000 cells: chunk sums
])
def test_scan_sizes(M, L, r_c, n):
    """FP32 rounding of the product is below the repository's FP32 bar; a particle in a wrong bin loses its pairs or
    its window and is off by its whole contribution."""
    fcm = ensure_built()
    rng = np.random.default_rng(n)
    Y = rng.random((n, 3)) * np.broadcast_to(np.asarray(L, dtype=float), (3,))
    s = System(n, L, M, 1.2, 8, r_c, 3, Y=Y)
    s.Y = s.Y.astype(np.float32).astype(np.float64)
    s.F, s.T = s.F.astype(np.float32).astype(np.float64), s.T.astype(np.float32).astype(np.float64)
    U, W = run_gpu(s, fcm.FCM_FP32)
    U64, W64 = run_gpu(s, fcm.FCM_FP64)
    assert_parity(U, U64, FP32_TOL, f"U {M}")
    assert_parity(W, W64, FP32_TOL, f"W {M}")
