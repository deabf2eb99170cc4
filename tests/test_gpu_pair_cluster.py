"""The FP32 pair kernel where its cases meet: clusters of four that are not full, chunks of candidates, the near queue,
parameter sets without a polynomial fit, boxes of three cells, loads that are not finite."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, System, assert_parity, ensure_built, run_gpu

pytestmark = pytest.mark.gpu

# FP32 sums of up to a few hundred terms with coefficients good to 1e-7 of the self mobility: well inside FP32_TOL, the
# repository's bar, which a lost or doubled pair misses by orders of magnitude.


@pytest.mark.parametrize("n,L,r_c,Sigma,Sigma_D,torques", [
    (1, 30.0, 9.0, 1.5, 0.0, True),
    (5, 30.0, 9.0, 1.5, 0.0, True),        # a cluster of four and one of one
    (130, 30.0, 10.0, 1.5, 0.0, False),    # three cells per side, each at least r_c wide
    (130, 30.0, 14.9, 2.0, 0.0, True),     # three cells per side, narrower than r_c
    (900, 34.0, 11.3, 1.6, 0.0, True),     # own cell and half shell of more than one chunk of candidates
    (900, 34.0, 6.5, 1.0, 0.0, True),      # about 14 particles per cell: four warps
    (300, 60.0, 7.0, 1.1, 0.0, True),      # cells widened to eight particles: two warps
    (400, 40.0, 3.1, 0.6, 0.0, True),      # Sigma close to sigma: most pairs are near ones
    (400, 40.0, 9.0, 1.5, 1.9, True),      # Sigma_D > Sigma: no fit, every pair by the table
    (400, (50.0, 36.0, 24.0), 8.0, 1.5, 0.0, True),
])
def test_pair_cluster(n, L, r_c, Sigma, Sigma_D, torques):
    fcm = ensure_built()
    s = System(n, L, 32, Sigma, 8, r_c, 40 + n, torques=torques, Sigma_D=Sigma_D, min_sep=0.5)
    U, W = run_gpu(s, fcm.FCM_FP32, stages=2, want_W=torques)
    Uo, Wo = s.oracle(fcm.FCM_FP32, stages=2)
    assert_parity(U, Uo, FP32_TOL, "U")
    if torques:
        assert_parity(W, Wo, FP32_TOL, "W")


@pytest.mark.parametrize("bad", [np.inf, np.nan, 3e19])
def test_pair_odd_loads_stay_local(bad):
    """A load that is not finite (or huge) reaches the particles within r_c of its own and no others."""
    fcm = ensure_built()
    s = System(600, 44.0, 32, 1.5, 8, 9.5, 77)
    U0, W0 = run_gpu(s, fcm.FCM_FP32, stages=2)
    s.F[17, 1] = bad
    U, W = run_gpu(s, fcm.FCM_FP32, stages=2)
    d = s.Y - s.Y[17]
    d -= 44.0 * np.round(d / 44.0)
    far = np.linalg.norm(d, axis=1) > 9.5 * (1 + 1e-6)
    assert far.sum() > 100
    assert_parity(U[far], U0[far], FP32_TOL, "U far")
    assert_parity(W[far], W0[far], FP32_TOL, "W far")
    if not np.isfinite(bad):
        assert not np.isfinite(U[17]).all()
