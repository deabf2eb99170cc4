"""The pair kernels' crowded cells (more than 96 particles): their parts are shared out and summed in FP64, in FP32
in launches of two and of four warps per cell, beside cells that are not crowded, and none is left from an earlier call."""
import numpy as np
import pytest

from gpu_util import (FP64_TOL, System, assert_parity, ensure_built, params_for, rel_l2, rounded, run_gpu,
                      torch_cuda)

pytestmark = pytest.mark.gpu

# A pair's term is good to a few roundings of 2^-24 and an exp2 of 2^-22, and close pairs to the cubic table's 1e-8 of the
# self mobility where their functions are a tenth of it, so it and a sum of many such terms (independent, as the terms
# are) have an rms error below sqrt(2^-44 + 1e-14) = 2.6e-7 of their rms, whatever their number: 3e-7. Plain FP32 sums over
# the 10,000 neighbours of the first two cases add more than that by themselves.
BAR = 3e-7
CROWD = 96


def _cells(s, max_n):
    """Particles per pair cell and the mean over the cells, as the library divides the box."""
    V = float(np.prod(np.broadcast_to(np.asarray(s.L, float), (3,))))
    side = max(s.r_c, (8.0 * V / max_n) ** (1.0 / 3.0))
    m = [max(3, int(e / side)) for e in np.broadcast_to(np.asarray(s.L, float), (3,))]
    c = [np.minimum((s.Y[:, d] % e * m[d] / e).astype(int), m[d] - 1)
         for d, e in enumerate(np.broadcast_to(np.asarray(s.L, float), (3,)))]
    count = np.bincount(c[0] + m[0] * (c[1] + m[1] * c[2]), minlength=m[0] * m[1] * m[2])
    return count, s.n / count.size


def _corner(n, L, corner, seed):
    return np.random.default_rng(seed).random((n, 3)) * corner + 0.01


@pytest.mark.parametrize("n,L,corner,r_c,torques,two_warps", [
    (24000, 300.0, 21.3, 11.47, True, True),    # one cell of 24,000: 750 parts, 38 chunks each
    (24000, 300.0, 21.3, 11.47, False, True),
    (20000, 60.0, 60.0, 11.9, True, False),     # every cell crowded, four per CTA slot or more
    (3000, 34.0, 34.0, 14.9, True, False),      # three cells per side, narrower than the cutoff: images by distance
    (2500, 60.0, 25.0, 11.5, False, False),     # crowded cells among empty and ordinary ones
])
def test_crowded_cells(n, L, corner, r_c, torques, two_warps):
    fcm = ensure_built()
    s = System(n, L, 32, 1.6, 8, r_c, 3, torques=torques, Y=_corner(n, L, corner, n))
    s.Y, s.F, s.T = (rounded(a, fcm.FCM_FP32) for a in (s.Y, s.F, s.T))
    count, mean = _cells(s, n)
    assert count.max() > CROWD and (mean < 10) == two_warps
    U, W = run_gpu(s, fcm.FCM_FP32, stages=2, want_W=torques)
    U64, W64 = run_gpu(s, fcm.FCM_FP64, stages=2, want_W=torques)
    print(f"largest cell {count.max()}, U {rel_l2(U, U64):.3e}", f"W {rel_l2(W, W64):.3e}" if torques else "")
    assert rel_l2(U, U64) < BAR
    if torques:
        assert rel_l2(W, W64) < BAR


@pytest.mark.parametrize("k", [96, 97, 128, 129])
def test_edge_of_a_crowded_cell(k):
    """One cell at and past the limit, the rest of the box thin."""
    fcm = ensure_built()
    rng = np.random.default_rng(k)
    Y = np.concatenate([rng.random((k, 3)) * 9.0 + 0.3, 26.0 + rng.random((500, 3)) * 70.0])
    s = System(k + 500, 100.0, 32, 1.2, 8, 8.6, 5, Y=Y)
    s.Y, s.F, s.T = (rounded(a, fcm.FCM_FP32) for a in (s.Y, s.F, s.T))
    count, _ = _cells(s, s.n)
    assert count[0] == k
    U, W = run_gpu(s, fcm.FCM_FP32, stages=2)
    U64, W64 = run_gpu(s, fcm.FCM_FP64, stages=2)
    assert rel_l2(U, U64) < BAR and rel_l2(W, W64) < BAR


def test_calls_and_systems_do_not_share_crowds():
    """A call after a crowded one, on the same handle, and a batch in which one system is crowded."""
    torch = torch_cuda()
    fcm = ensure_built()
    n, L = 3000, 120.0
    crowd = System(n, L, 32, 1.6, 8, 11.4, 8, Y=_corner(n, L, 25.0, 1))
    thin = System(n, L, 32, 1.6, 8, 11.4, 9, Y=np.random.default_rng(2).random((n, 3)) * L)
    alone = [run_gpu(s, fcm.FCM_FP32, stages=2) for s in (crowd, thin)]
    with fcm.Handle(params_for(fcm, crowd, fcm.FCM_FP32, max_n=2 * n), 0, 2) as h:
        for s, ref in ((crowd, alone[0]), (thin, alone[1]), (crowd, alone[0])):
            for got, want in zip(run_gpu(s, fcm.FCM_FP32, stages=2, handle=h), ref):
                assert rel_l2(got, want) < 1e-6   # the order of FP32 sums is free, the handle's cells are others
        to = lambda a: torch.as_tensor(np.concatenate(a), dtype=torch.float32, device="cuda:0")
        for pair, ref in (((thin, crowd), (alone[1], alone[0])), ((crowd, thin), (alone[0], alone[1]))):
            pos, F, T = (to([getattr(s, k) for s in pair]) for k in "YFT")
            U, W = torch.empty_like(F), torch.empty_like(F)
            h.batch_apply([0, n, 2 * n], pos, F, T, U, W, torch.cuda.current_stream().cuda_stream, fcm.STAGE_PAIR)
            assert h.check() == 0
            for k in range(2):
                rows = slice(k * n, (k + 1) * n)
                assert rel_l2(U[rows].double().cpu().numpy(), ref[k][0]) < 1e-6
                assert rel_l2(W[rows].double().cpu().numpy(), ref[k][1]) < 1e-6


def test_crowded_cells_without_allocation():
    torch = torch_cuda()
    fcm = ensure_built()
    n, L = 12000, 200.0
    s = System(n, L, 32, 1.6, 8, 11.47, 4, Y=_corner(n, L, 22.0, 7))
    s.Y, s.F, s.T = (rounded(a, fcm.FCM_FP32) for a in (s.Y, s.F, s.T))
    U64, W64 = run_gpu(s, fcm.FCM_FP64, stages=2)
    to = lambda a: torch.as_tensor(a, dtype=torch.float32, device="cuda:0")
    pos, F, T = to(s.Y), to(s.F), to(s.T)
    U, W = torch.empty_like(F), torch.empty_like(F)
    for _ in range(2):
        fcm.pair_correction_noalloc(params_for(fcm, s, fcm.FCM_FP32), n, pos, F, T, U, W,
                                    torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert rel_l2(U.double().cpu().numpy(), U64) < BAR and rel_l2(W.double().cpu().numpy(), W64) < BAR


@pytest.mark.parametrize("n,L,corner,r_c,torques", [
    (1500, 100.0, 19.9, 9.9, True),     # one cell of 1,500
    (1500, 100.0, 19.9, 9.9, False),
    (3000, 34.0, 34.0, 11.3, True),     # every cell crowded
    (700, 100.0, 24.0, 9.9, True),      # crowded cells among empty and ordinary ones
])
def test_crowded_cells_fp64(n, L, corner, r_c, torques):
    """The same sharing out in FP64, against the oracle."""
    fcm = ensure_built()
    s = System(n, L, 32, 1.6, 8, r_c, 3, torques=torques, Y=_corner(n, L, corner, n))
    count, _ = _cells(s, n)
    assert count.max() > CROWD
    U, W = run_gpu(s, fcm.FCM_FP64, stages=2, want_W=torques)
    Uo, Wo = s.oracle(fcm.FCM_FP64, stages=2)
    assert_parity(U, Uo, FP64_TOL, "U")
    if torques:
        assert_parity(W, Wo, FP64_TOL, "W")
