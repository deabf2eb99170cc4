"""The pair kernels' chunks of candidates and two-warp launches, and the binning's scan over many chunks of counters, at
sizes that are checked to reach them, against references that do not use the binning."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, FP64_TOL, System, assert_parity, ensure_built, params_for, rounded, run_gpu, torch_cuda
from oracle import grid_fcm as og

pytestmark = pytest.mark.gpu

CHUNK32, CHUNK64 = 640, 512   # staged candidates per pass of the FP32 and the FP64 pair kernel
CROWD = 96                    # particles above which a cell of the FP32 kernel goes another way
SCAN_CHUNK, SUMS_ABOVE = 2048, 32   # counters per block of the scan; chunks above which it uses their sums


def _cells(Y, L, r_c, max_n, systems=1):
    """Pair cells per dimension and the particles of each cell, as the library divides the box."""
    L = np.broadcast_to(np.asarray(L, dtype=float), (3,))
    side = max(r_c, (8.0 * float(np.prod(L)) * systems / max_n) ** (1.0 / 3.0))
    m = np.maximum((L / side).astype(int), 3)
    c = np.minimum((np.mod(Y, L) * m / L).astype(int), m - 1)
    return m, np.bincount(c[:, 0] + m[0] * (c[:, 1] + m[1] * c[:, 2]), minlength=int(m.prod())).reshape(m[::-1])


def _half_shell(count):
    """Candidates of every cell: its own and those of 13 neighbours."""
    tot = count.copy()
    for dz, dy, dx in [(0, 0, 1)] + [(0, 1, d) for d in (-1, 0, 1)] + [(1, e, d) for e in (-1, 0, 1) for d in (-1, 0, 1)]:
        tot = tot + np.roll(count, (-dz, -dy, -dx), axis=(0, 1, 2))
    return tot


def _check(fcm, s, precision, tol, torques):
    U, W = run_gpu(s, precision, stages=2, want_W=torques)
    Uo, Wo = s.oracle(precision, stages=2)
    assert_parity(U, Uo, tol, "U")
    if torques:
        assert_parity(W, Wo, tol, "W")


@pytest.mark.parametrize("torques", [True, False])
@pytest.mark.parametrize("n,L,r_c,chunks", [
    (1620, 34.0, 11.3, 2),    # three cells per side at the cutoff
    (1620, 34.0, 14.9, 2),    # three narrower ones: nearest images
    (4300, 50.0, 12.4, 2),    # four per side
])
def test_fp32_chunks(n, L, r_c, chunks, torques):
    """Candidates of a later chunk, which the clusters meet again, in cells that are not crowded."""
    fcm = ensure_built()
    rng = np.random.default_rng(n)
    s = System(n, L, 32, 1.6, 8, r_c, 12, torques=torques, Y=rng.random((n, 3)) * L)
    _, count = _cells(rounded(s.Y, fcm.FCM_FP32), L, r_c, n)
    tot = _half_shell(count)
    assert count.max() <= CROWD and np.mean(tot > CHUNK32) > 0.9 and -(-tot.max() // CHUNK32) == chunks
    _check(fcm, s, fcm.FCM_FP32, FP32_TOL, torques)


@pytest.mark.parametrize("torques", [True, False])
def test_fp32_two_warps(torques):
    """Cells of eight particles, four shifted images and more per dimension, pairs in every one."""
    fcm = ensure_built()
    n, L, r_c = 4096, 64.0, 7.9
    rng = np.random.default_rng(1)
    s = System(n, L, 32, 1.1, 8, r_c, 12, torques=torques, Y=rng.random((n, 3)) * L)
    m, count = _cells(s.Y, L, r_c, n)
    assert n < 10 * count.size and m.min() >= 4 and count.max() <= CROWD
    _check(fcm, s, fcm.FCM_FP32, FP32_TOL, torques)


def test_fp64_chunks():
    fcm = ensure_built()
    n, L, r_c = 1300, 26.0, 8.6
    s = System(n, L, 32, 1.4, 8, r_c, 12, Y=np.random.default_rng(2).random((n, 3)) * L)
    _, count = _cells(s.Y, L, r_c, n)
    assert np.mean(_half_shell(count) > CHUNK64) > 0.9
    _check(fcm, s, fcm.FCM_FP64, FP64_TOL, True)


@pytest.mark.parametrize("systems", [1, 2])
def test_scan_many_cells(systems):
    """More than 32 chunks of cell counters per system: starts from the chunks' sums, in the first and a later system."""
    torch = torch_cuda()
    fcm = ensure_built()
    n, L, r_c, Sigma = 80000, 200.0, 6.0, 1.0
    rng = np.random.default_rng(5)
    Y = [rounded(rng.random((n, 3)) * L, fcm.FCM_FP32) for _ in range(systems)]
    F, T = ([rounded(rng.normal(size=(n, 3)), fcm.FCM_FP32) for _ in range(systems)] for _ in range(2))
    m, _ = _cells(Y[0], L, r_c, n * systems, systems)
    assert 8 * int(m.prod()) > SUMS_ABOVE * SCAN_CHUNK
    s = System(n * systems, L, 32, Sigma, 8, r_c, 1, Y=np.concatenate(Y))
    to = lambda a: torch.as_tensor(np.concatenate(a), dtype=torch.float32, device="cuda:0")
    pos, Fd, Td = to(Y), to(F), to(T)
    U, W = torch.empty_like(Fd), torch.empty_like(Fd)
    with fcm.Handle(params_for(fcm, s, fcm.FCM_FP32), 0, systems) as h:
        h.batch_apply([n * k for k in range(systems + 1)], pos, Fd, Td, U, W, torch.cuda.current_stream().cuda_stream,
                      fcm.STAGE_PAIR)
        assert h.check() == 0
    for k in range(systems):
        rows = np.sort(rng.choice(n, 200, replace=False))
        Uo, Wo = og.pair_correction_subset(Y[k], F[k], T[k], L, r_c, Sigma, Sigma, rows)
        assert_parity(U[n * k + rows].double().cpu().numpy(), Uo, FP32_TOL, f"U system {k}")
        assert_parity(W[n * k + rows].double().cpu().numpy(), Wo, FP32_TOL, f"W system {k}")


def test_scan_many_tiles():
    """More than 32 chunks of tile counters in each of two systems, the last one part-full, against the FP64 kernels,
    which take particles one by one whatever their order."""
    torch = torch_cuda()
    fcm = ensure_built()
    n, M = 3000, (264, 264, 256)
    L = tuple(1.1 * e for e in M)
    tiles = (M[0] // 8) * (M[1] // 8) * (M[2] // 8)
    assert 2 * tiles > SUMS_ABOVE * SCAN_CHUNK and 2 * tiles % SCAN_CHUNK
    rng = np.random.default_rng(6)
    Y = [rounded(rng.random((n, 3)) * L, fcm.FCM_FP32) for _ in range(2)]
    s = System(2 * n, L, M, 1.0, 8, 3.0, 2, Y=np.concatenate(Y))
    s.F, s.T = rounded(s.F, fcm.FCM_FP32), rounded(s.T, fcm.FCM_FP32)
    to = lambda a: torch.as_tensor(a, dtype=torch.float32, device="cuda:0")
    pos, Fd, Td = to(s.Y), to(s.F), to(s.T)
    U, W = torch.empty_like(Fd), torch.empty_like(Fd)
    with fcm.Handle(params_for(fcm, s, fcm.FCM_FP32), 0, 2) as h:
        h.batch_apply([0, n, 2 * n], pos, Fd, Td, U, W, torch.cuda.current_stream().cuda_stream, fcm.STAGE_GRID)
        assert h.check() == 0
    for k in range(2):
        rows = slice(n * k, n * (k + 1))
        one = System(n, L, M, 1.0, 8, 3.0, 2, Y=Y[k])
        one.F, one.T = s.F[rows], s.T[rows]
        U64, W64 = run_gpu(one, fcm.FCM_FP64, stages=1)
        assert_parity(U[rows].double().cpu().numpy(), U64, FP32_TOL, f"U system {k}")
        assert_parity(W[rows].double().cpu().numpy(), W64, FP32_TOL, f"W system {k}")
