"""The FP32 pair correction's radial functions one pair at a time, to the accuracy they are fitted to."""
import math

import numpy as np
import pytest

from gpu_util import System, ensure_built, run_gpu
from oracle import closed_forms as cf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Sigma,Sigma_D,r_c", [(1.6, 0.0, 11.4705), (1.41047, 0.0, 8.7628), (2.0, 0.0, 14.2752),
                                               (2.0, 1.6, 14.2752)])
def test_pair_coefficients_sweep(Sigma, Sigma_D, r_c):
    """512 isolated pairs with separations from 0.5 to the cutoff; one particle of a pair is loaded and the other's
    velocities are compared, so there is no self term. Coordinates are multiples of 2^-8 below 2^8, so all differences
    are exact. Beyond 3 Sigma every pair takes the polynomials: each function is off by at most 1e-9 of its self
    mobility (two of them act in U and in W by each load, rounded up to 2.5e-9) and by FP32 rounding, 1e-6 of the value
    by the fit's own acceptance and about twice that for exp2 of -r^2 / 4 Sigma^2 (r^2 rounded to 2^-24 of 12 units),
    taken as 4e-6 of the tensors' norms. Closer, the cubic table is good to about 1e-7 of each function's largest value."""
    fcm = ensure_built()
    rng = np.random.default_rng(int(100 * Sigma))
    ijk = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    r = np.linspace(0.5, r_c * 0.999, 512)
    d = np.abs(rng.normal(size=(512, 3)))   # into one octant, so that pairs stay r_c apart
    d *= (r / np.linalg.norm(d, axis=1))[:, None]
    A = 32.0 * ijk + np.round(256 * rng.random(3)) / 256
    d = np.round(256 * d) / 256
    Y = np.stack([A, A + d], axis=1).reshape(-1, 3)
    s = System(1024, 256.0, 32, Sigma, 8, r_c, 7, Sigma_D=Sigma_D, Y=Y)
    s.F = s.F.astype(np.float32).astype(np.float64)
    s.T = s.T.astype(np.float32).astype(np.float64)
    s.F[1::2] = 0.0
    s.T[1::2] = 0.0
    U, W = run_gpu(s, fcm.FCM_FP32, stages=2)
    x, F, T = d, s.F[::2], s.T[::2]   # from the loaded particle to the other
    vf = cf.correction_VF(x, Sigma)
    wf = cf.correction_WF(x, Sigma, Sigma_D or Sigma)
    wt = cf.correction_WT(x, Sigma, Sigma_D or Sigma)
    vt = np.swapaxes(-wf, -1, -2)
    Ue = np.einsum("pab,pb->pa", vf, F) + np.einsum("pab,pb->pa", vt, T)
    We = np.einsum("pab,pb->pa", wf, F) + np.einsum("pab,pb->pa", wt, T)
    nF, nT = np.linalg.norm(F, axis=1), np.linalg.norm(T, axis=1)
    uvf, uwt = 1 / (6 * math.pi), 1 / (8 * math.pi)
    uwf = math.sqrt(uvf * uwt)
    norm = lambda m: np.linalg.norm(m, axis=(1, 2))
    far = np.linalg.norm(d, axis=1) > 3.0 * Sigma
    assert far.sum() > 200
    fit = np.where(far, 2.5e-9, 3e-7)
    barU = fit * (uvf * nF + uwf * nT) + 4e-6 * (norm(vf) * nF + norm(vt) * nT)
    barW = fit * (uwf * nF + uwt * nT) + 4e-6 * (norm(wf) * nF + norm(wt) * nT)
    for got, exact, bar, what in ((U[1::2], Ue, barU, "U"), (W[1::2], We, barW, "W")):
        ratio = np.linalg.norm(got - exact, axis=1) / bar
        print(f"{what}: largest error over its bar: near {ratio[~far].max():.2f}, far {ratio[far].max():.2f}")
        assert ratio.max() < 1.0
