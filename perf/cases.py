"""What a user of this package has it compute, as cases that can be timed and compared.

A case is a dict of plain numbers: a periodic system (box, grid, kernel width, support, cutoff), the
call made on it and its precision. ``prepare`` makes what a program holds before the call (device
arrays, the handle, the server), ``run`` makes one call through the public binding and returns its
outputs, and ``exact`` computes the same product with torch in 64 bits straight from the formulas of
the fast force-coupling method.

Kinds of calls:

* ``apply``: one system, one mobility product (simulation steps, one product of an iterative solver);
* ``batch``: many systems of one parameter set in one pass (ensembles, parameter studies);
* ``brownian``: a Brownian velocity increment (grid part and Lanczos pair part);
* ``rigid``: the velocities of rigid rods under given loads (Broyden iterations on the device);
* ``serve``: requests in host memory through the request server.

Positions are random, non-overlapping suspensions (a random subset of the sites of a fine lattice, each
moved at random inside its site) or, where a case says ``rods``, rods of 64 touching spheres in random
directions that may cross. Loads are independent normal numbers.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2310_12651_gb300 import fcm, inputs

SIGMA = 1.0 / math.sqrt(math.pi)   # kernel width of standard FCM for spheres of radius 1
PER_ROD = 64
ROD_BOND = 2.2


# ---------------------------------------------------------------- the cases

def _system(kind, n, box, grid, Sigma, M_G, r_c, torques=True, double=False, systems=1, ragged=False, rods=False):
    Lx, Ly, Lz = box if isinstance(box, tuple) else (box, box, box)
    Mx, My, Mz = grid if isinstance(grid, tuple) else (grid, grid, grid)
    return {"kind": kind, "n": int(n), "Lx": float(Lx), "Ly": float(Ly), "Lz": float(Lz), "Mx": int(Mx), "My": int(My),
            "Mz": int(Mz), "Sigma": float(Sigma), "M_G": int(M_G), "r_c": float(r_c), "torques": bool(torques),
            "double": bool(double), "systems": int(systems), "ragged": bool(ragged), "rods": bool(rods)}


def listed():
    cases = []

    def add(name, case):
        cases.append(dict(case, name=name))

    # The smallest call: a small suspension stepped one product at a time, where launches and latency count.
    add("one_small", _system("apply", 2000, 55.1339, 32, 1.6, 10, 11.4705))
    # A thousand spheres in double precision at the 1e-8 rule, forces only: the accuracy reference of a study.
    add("one_double_dilute", _system("apply", 1000, 100.0, 64, 2.0, 12, 16.901, torques=False, double=True))
    # Double precision with torques at 5%: a solver or a test that needs more than single precision.
    add("one_double", _system("apply", 8192, 88.207, 64, 2.0, 14, 14.2752, double=True))
    # One suspension of ordinary size at 5%, forces and torques: a step of a single simulation.
    add("one_suspension", _system("apply", 65536, 176.4139, 128, 1.5, 12, 10.7606))
    # Settings of the paper's timing study (box of 400 radii, forces only, tolerance 1e-4) at 0.8%: sedimentation.
    add("one_dilute_forces", _system("apply", 122231, 400.0, 216, 3.4 * SIGMA, 10, 18.6 * SIGMA, torques=False))
    # A million spheres at 10%, forces and torques: the largest single system.
    add("one_million", _system("apply", 1048576, 352.83, 256, 1.69257, 14, 12.3934))
    # Thirty-two suspensions of 65,536 spheres in one pass: the throughput workload, and the largest case.
    add("batch_suspensions", _system("batch", 65536, 176.4139, 128, 2.0, 14, 14.2752, systems=32))
    # Eight suspensions of rods: clustered particles, uneven work per tile and per cell.
    add("batch_rods", _system("batch", 65536, 176.4139, 128, 2.5 * SIGMA, 12, 8.7628, systems=8, rods=True))
    # Small systems of uneven sizes (one of them empty) in a box with three different edges: a parameter study.
    add("batch_ragged", _system("batch", 4999, (118.0, 96.0, 71.0), (90, 72, 54), 2.5 * SIGMA, 12, 8.7628, systems=13,
                                ragged=True))
    # A Brownian velocity increment of a suspension: noise on the grid and the square root of the pair part.
    add("brownian_step", dict(_system("brownian", 32768, 140.02, 108, 1.41047, 12, 8.7628)))
    # Rigid rods of 22 particles in a flat box, the paper's Section 6.1 suspension of 2,304 rods: one velocity solve.
    add("rigid_rods", dict(_system("rigid", 2304 * 22, (960.0, 960.0, 60.0), (240, 240, 16), 4.08643, 12, 25.3378,
                                   torques=False), tol=1e-4, precond=0))
    # Requests of three box sizes in host memory, all queued at once: the request server.
    add("serve_requests", dict(_system("serve", 6000, 102.866, 80, 2.5 * SIGMA, 12, 8.7628), requests=24))
    return cases


def _smooth_above(v):
    """The smallest even 2^a 3^b 5^c at or above v."""
    m = max(2, int(math.ceil(v - 1e-9)))
    m += m & 1
    while True:
        r = m
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            return m
        m += 2


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _drawn_system(rng, n, torques, stretch, max_grid=256):
    """Box, grid, width, support and cutoff for n spheres: a volume fraction, a tolerance and a number of
    neighbours are drawn, the rest follows from the paper's rules (resolution, window and cutoff over the width)."""
    phi = math.exp(rng.uniform(math.log(0.004), math.log(0.2)))
    tight = rng.random() < 0.35
    ratio, trunc, slope = (1.3, 4.8, 7.14) if tight else (1.05, 4.6, 6.2)
    L = inputs.box_edge(n, phi)
    box = (L, L, L)
    if stretch:
        a, b = rng.uniform(0.75, 1.35), rng.uniform(0.75, 1.35)
        box = (L * a, L * b, L / (a * b))
    short = min(box)
    neighbours = rng.uniform(25.0, 150.0)
    r_c = min((neighbours / phi) ** (1.0 / 3.0), 0.45 * short)
    Sigma = max(r_c / slope, 1.3 * SIGMA)
    grid = tuple(max(32, _smooth_above(e * ratio / Sigma)) for e in box)
    if max(grid) > max_grid:   # a wider kernel on the largest grid
        Sigma = max(e * ratio / max_grid for e in box)
        grid = tuple(max(32, min(max_grid, _smooth_above(e * ratio / Sigma))) for e in box)
    h = min(e / m for e, m in zip(box, grid))
    M_G = min(16, 2 * int(math.ceil(trunc * Sigma / h - 1e-9)), min(grid))
    r_c = min(slope * Sigma, 0.5 * short)
    return [round(e, 4) for e in box], grid, round(Sigma, 5), M_G, round(min(r_c, 0.4999 * short), 4)


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm, odd ones among them."""
    kind = rng.choices(("apply", "batch", "double", "brownian", "rigid", "serve"), (40, 25, 15, 8, 6, 6))[0]
    if kind == "rigid":
        rods = _log_int(rng, 200, 2304)
        L = round(960.0 * math.sqrt(rods / 2304.0), 3)
        M = _smooth_above(L / 4.0)
        return dict(_system("rigid", rods * 22, (L, L, 60.0), (M, M, 16), 4.08643, 12, 25.3378, torques=False),
                    tol=1e-4, precond=rng.randrange(2))
    if kind == "serve":
        return dict(_system("serve", _log_int(rng, 2000, 9000), 102.866, 80, 2.5 * SIGMA, 12, 8.7628),
                    requests=rng.randint(8, 30))
    torques = rng.random() < 0.7
    if kind == "double":
        n = _log_int(rng, 400, 8192)
        box, grid, Sigma, M_G, r_c = _drawn_system(rng, n, torques, rng.random() < 0.3, 64)
        return _system("apply", n, tuple(box), grid, Sigma, M_G, r_c, torques, double=True)
    if kind == "brownian":
        n = _log_int(rng, 1500, 50000)
        box, grid, Sigma, M_G, r_c = _drawn_system(rng, n, False, False, 128)
        return _system("brownian", n, tuple(box), grid, Sigma, M_G, r_c)
    if kind == "batch":
        systems = _log_int(rng, 2, 48)
        n = _log_int(rng, 700, max(800, 600000 // systems))
        box, grid, Sigma, M_G, r_c = _drawn_system(rng, n, torques, rng.random() < 0.4, 128)
        return _system("batch", n, tuple(box), grid, Sigma, M_G, r_c, torques, systems=systems,
                       ragged=rng.random() < 0.6, rods=rng.random() < 0.25)
    n = _log_int(rng, 500, 1000000)
    box, grid, Sigma, M_G, r_c = _drawn_system(rng, n, torques, rng.random() < 0.3)
    return _system("apply", n, tuple(box), grid, Sigma, M_G, r_c, torques, rods=rng.random() < 0.2)


# ---------------------------------------------------------------- inputs

def _counts(case):
    """Particles of each system: equal, or (ragged) uneven with one empty system in the middle."""
    if not case["ragged"]:
        return [case["n"]] * case["systems"]
    rng = random.Random(case["n"] * 1009 + case["systems"])
    c = [max(1, int(case["n"] * math.exp(rng.uniform(-1.4, 0.6)))) for _ in range(case["systems"])]
    if case["systems"] > 2:
        c[case["systems"] // 2] = 0
    return c


def _suspension(n, box, gen):
    """n centres at least about 2 apart: random sites of a lattice, each centre moved at random inside its site."""
    dev = gen.device
    L = torch.tensor(box, dtype=torch.float64, device=dev)
    step = max(2.05, 0.72 * (box[0] * box[1] * box[2] / max(n, 1)) ** (1.0 / 3.0))
    m = [max(1, int(e / step)) for e in box]
    while m[0] * m[1] * m[2] < n:
        k = min(range(3), key=lambda d: m[d] / box[d])
        m[k] += 1
    site = torch.randperm(m[0] * m[1] * m[2], generator=gen, device=dev)[:n]
    ijk = torch.stack([site % m[0], (site // m[0]) % m[1], site // (m[0] * m[1])], dim=1).double()
    edge = L / torch.tensor(m, dtype=torch.float64, device=dev)
    play = (edge - 2.0).clamp_min(0.0)
    u = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=gen) - 0.5
    shift = torch.rand(3, dtype=torch.float64, device=dev, generator=gen)
    return torch.remainder((ijk + 0.5 + shift) * edge + u * play, L)


def _rods(n, box, gen):
    """n spheres in rods of 64 with centres and directions at random (the last rod shorter)."""
    dev = gen.device
    L = torch.tensor(box, dtype=torch.float64, device=dev)
    k = -(-n // PER_ROD)
    c = torch.rand((k, 3), dtype=torch.float64, device=dev, generator=gen) * L
    v = torch.randn((k, 3), dtype=torch.float64, device=dev, generator=gen)
    v = v / v.norm(dim=1, keepdim=True)
    s = (torch.arange(PER_ROD, dtype=torch.float64, device=dev) - 0.5 * (PER_ROD - 1)) * ROD_BOND
    return torch.remainder((c[:, None, :] + s[None, :, None] * v[:, None, :]).reshape(-1, 3)[:n], L)


def _arrays(case, counts, seed):
    """Positions, forces and torques (None without) of all systems, stacked, in the case's precision."""
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    box = (case["Lx"], case["Ly"], case["Lz"])
    make = _rods if case["rods"] else _suspension
    pos = torch.cat([make(n, box, gen) for n in counts])
    dt = torch.float64 if case["double"] else torch.float32
    F = torch.randn(pos.shape, dtype=dt, device=dev, generator=gen)
    T = torch.randn(pos.shape, dtype=dt, device=dev, generator=gen) if case["torques"] else None
    return pos.to(dt).contiguous(), F, T


def _params(case, n):
    return fcm.make_params((case["Lx"], case["Ly"], case["Lz"]), (case["Mx"], case["My"], case["Mz"]), case["Sigma"],
                           case["r_c"], case["M_G"], n, fcm.FCM_FP64 if case["double"] else fcm.FCM_FP32)


def _requests(case, seed):
    """Requests of the serving case: three box sizes at one grid spacing, sizes spread around n."""
    sizes = random.Random(case["n"] * 31 + case["requests"])
    out = []
    for k in range(case["requests"]):
        edge, grid = ((71.6275, 54), (102.866, 80), (147.7283, 108))[k % 3]
        n = max(16, int(case["n"] * (edge / 102.866) ** 3 * math.exp(sizes.uniform(-0.7, 0.7))))
        c = dict(case, n=n, Lx=edge, Ly=edge, Lz=edge, Mx=grid, My=grid, Mz=grid, rods=k % 2 == 1)
        out.append((c, _arrays(c, [n], seed * 64 + k)))
    return out


def _noise(case, seed):
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(int(seed) + 7919)
    dt = torch.float64 if case["double"] else torch.float32
    xi = torch.randn(3 * case["Mx"] * case["My"] * case["Mz"], dtype=dt, device="cuda:0", generator=gen)
    z = torch.randn((case["n"], 3), dtype=dt, device="cuda:0", generator=gen)
    return xi, z


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "kind": kind}
    if kind == "serve":
        reqs = []
        for c, arrays in _requests(case, seed):
            reqs.append((_params(c, c["n"]), [a.cpu().numpy() for a in arrays]))
        return dict(state, server=fcm.Server(0, 8 << 30, 64), requests=reqs)
    if kind == "rigid":
        rods = case["n"] // 22
        Y, off, X = inputs.doublet_rods(rods, case["Lx"], case["Lz"], seed)
        ft = inputs.rod_loads(rods, seed + 1, scale=0.1)
        to = lambda a, dt=torch.float32: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda:0")
        return dict(state, handle=fcm.Handle(_params(case, case["n"])), pos=to(Y), off=to(off, torch.int32), X=to(X),
                    ft=to(ft), F=to(np.zeros_like(Y)), UG=to(np.zeros((rods, 6))))
    counts = _counts(case)
    pos, F, T = _arrays(case, counts, seed)
    state = dict(state, pos=pos, F=F, T=T, handle=fcm.Handle(_params(case, max(1, sum(counts))), 0, len(counts)))
    if kind == "batch":
        state["offsets"] = [sum(counts[:k]) for k in range(len(counts) + 1)]
        state["U"] = torch.empty_like(F)
        state["W"] = torch.empty_like(F) if T is not None else None
    if kind == "brownian":
        state["xi"], state["z"] = _noise(case, seed)
        state["U"], state["W"] = torch.empty_like(F), torch.empty_like(F)
    return state


# ---------------------------------------------------------------- one call

def run(state):
    kind = state["kind"]
    if kind == "serve":
        tickets = [state["server"].submit(p, *arrays) for p, arrays in state["requests"]]
        for t in tickets:
            if not state["server"].wait(t, 60.0) or t.status != fcm.FCM_OK:
                raise RuntimeError("request failed with status %s" % t.status)
        return {"U": [t.U for t in tickets], "W": [t.W for t in tickets]}
    h = state["handle"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "apply":
        U, W = fcm.apply_tensors(h, state["pos"], state["F"], state["T"], want_W=state["T"] is not None)
        return {"U": U} if W is None else {"U": U, "W": W}
    if kind == "batch":
        h.batch_apply(state["offsets"], state["pos"], state["F"], state["T"], state["U"], state["W"], stream)
        return {"U": state["U"]} if state["W"] is None else {"U": state["U"], "W": state["W"]}
    if kind == "brownian":
        h.brownian(state["pos"].shape[0], state["pos"], 1.0, state["xi"], state["z"], state["U"], state["W"],
                   max_iter=40, tol=1e-6, stream=stream)
        return {"U": state["U"], "W": state["W"]}
    h.rigid_solve(state["pos"].shape[0], state["pos"], state["ft"].shape[0], state["off"], state["X"], state["ft"],
                  state["F"], state["UG"], max_iter=256, tol=state["case"]["tol"], stream=stream,
                  precond=state["case"]["precond"])
    return {"F": state["F"], "UG": state["UG"]}


# ---------------------------------------------------------------- work of one call

def _product_flops(case, n, torques, stages=3):
    """Window points (22 operations per point and side with torques, 8 without), grid transforms and pairs
    (250 or 100 operations per ordered pair) of one product on n particles."""
    M = case["Mx"] * case["My"] * case["Mz"]
    V = case["Lx"] * case["Ly"] * case["Lz"]
    grid = 2.0 * n * case["M_G"] ** 3 * (22.0 if torques else 8.0) + 6 * 2.5 * M * math.log2(M) + 15.0 * M
    pair = n * n / V * 4.0 / 3.0 * math.pi * case["r_c"] ** 3 * (250.0 if torques else 100.0)
    return (grid if stages & 1 else 0.0) + (pair if stages & 2 else 0.0)


def work(case):
    size = 8 if case["double"] else 4
    kind = case["kind"]
    if kind == "serve":
        per = [(c, a[0].shape[0]) for c, a in _requests(case, 0)]
        return {"bytes": sum(15.0 * size * n for _, n in per), "flops": sum(_product_flops(c, n, True) for c, n in per)}
    if kind == "rigid":   # about two dozen products from the diagonal start, half a dozen from the bodies' own mobility
        its = 6 if case["precond"] else 23
        return {"bytes": size * (6.0 * case["n"] + 15.0 * case["n"] / 22), "flops": its * _product_flops(case, case["n"], False)}
    if kind == "brownian":   # one grid pass (half of a product's points) and about nine pair products
        M = 3.0 * case["Mx"] * case["My"] * case["Mz"]
        return {"bytes": size * (M + 12.0 * case["n"]),
                "flops": 0.5 * _product_flops(case, case["n"], True, 1) + 9 * _product_flops(case, case["n"], False, 2)}
    counts = _counts(case)
    vectors = 15.0 if case["torques"] else 9.0
    return {"bytes": vectors * size * sum(counts), "flops": sum(_product_flops(case, n, case["torques"]) for n in counts)}


# ---------------------------------------------------------------- the same in 64 bits

class _Exact:
    """The mobility product of one system in 64 bits: windows as the case's precision places them."""

    def __init__(self, case, pos):
        self.c = case
        self.dev = pos.device
        self.L = torch.tensor([case["Lx"], case["Ly"], case["Lz"]], dtype=torch.float64, device=self.dev)
        self.M = [case["Mx"], case["My"], case["Mz"]]
        self.h = self.L / torch.tensor(self.M, dtype=torch.float64, device=self.dev)
        self.S = case["Sigma"]
        self.dd = SIGMA ** 2 - self.S ** 2
        self.Y = pos.double()
        MG = case["M_G"]
        inv = torch.tensor([m / float(l) for m, l in zip(self.M, self.L)], dtype=pos.dtype, device=self.dev)
        s = pos * inv if pos.dtype == torch.float32 else pos / self.h
        self.i0 = torch.floor(s - 0.5 * MG).long() + 1

    def _windows(self, a, b):
        """Flat grid index and the three 1-D displacements and Gaussians of particles a .. b."""
        MG = self.c["M_G"]
        j = torch.arange(MG, device=self.dev)
        idx, d, g = [], [], []
        for k in range(3):
            i = self.i0[a:b, k, None] + j
            dk = i.double() * self.h[k] - self.Y[a:b, k, None]
            idx.append(torch.remainder(i, self.M[k]))
            d.append(dk)
            g.append(torch.exp(-dk * dk / (2 * self.S ** 2)))
        flat = (idx[2][:, :, None, None] * self.M[1] + idx[1][:, None, :, None]) * self.M[0] + idx[0][:, None, None, :]
        return flat, [d[2][:, :, None, None], d[1][:, None, :, None], d[0][:, None, None, :]], \
            g[2][:, :, None, None] * g[1][:, None, :, None] * g[0][:, None, None, :]

    def _weights(self, d, g):
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        norm = (2 * math.pi * self.S ** 2) ** -1.5
        S2 = self.S ** 2
        return norm * g * (1 - 1.5 * self.dd / S2 + 0.5 * self.dd / S2 ** 2 * r2), norm * g / (2 * S2)

    def _parts(self):
        n = self.Y.shape[0]
        step = max(1, 40_000_000 // self.c["M_G"] ** 3)
        return [(a, min(n, a + step)) for a in range(0, n, step)]

    def spread(self, F, T):
        size = self.M[0] * self.M[1] * self.M[2]
        f = torch.zeros((3, size), dtype=torch.float64, device=self.dev)
        for a, b in self._parts():
            flat, (dz, dy, dx), g = self._windows(a, b)
            w, wt = self._weights((dz, dy, dx), g)
            d = (dx, dy, dz)
            flat = flat.reshape(-1)
            for c in range(3):
                v = F[a:b, c].double()[:, None, None, None] * w
                if T is not None:
                    p, q = (c + 1) % 3, (c + 2) % 3
                    v = v + wt * (T[a:b, p].double()[:, None, None, None] * d[q] - T[a:b, q].double()[:, None, None, None] * d[p])
                f[c].index_add_(0, flat, v.reshape(-1))
        return f.reshape(3, self.M[2], self.M[1], self.M[0])

    def solve(self, f, half=False):
        fh = torch.fft.rfftn(f, dim=(1, 2, 3))
        ks, keep = [], torch.ones(fh.shape[1:], dtype=torch.bool, device=self.dev)
        for axis, (k, m) in enumerate(((2, self.M[2]), (1, self.M[1]), (0, self.M[0]))):
            i = torch.arange(fh.shape[1 + axis], device=self.dev)
            i = torch.where(i <= m // 2, i, i - m)
            shape = [1, 1, 1]
            shape[axis] = -1
            if m % 2 == 0:
                keep &= (i.abs() != m // 2).reshape(shape)
            ks.append((2 * math.pi / self.L[k] * i).reshape(shape))
        kz, ky, kx = ks
        k2 = kx * kx + ky * ky + kz * kz
        keep &= k2 > 0
        inv = torch.where(keep, 1.0 / torch.where(keep, k2, 1.0), 0.0)
        along = (kx * fh[0] + ky * fh[1] + kz * fh[2]) * inv
        scale = torch.sqrt(inv) if half else inv
        u = torch.stack([(fh[c] - k * along) * scale for c, k in enumerate((kx, ky, kz))])
        return torch.fft.irfftn(u, s=(self.M[2], self.M[1], self.M[0]), dim=(1, 2, 3))

    def gather(self, u, torques):
        n = self.Y.shape[0]
        U = torch.zeros((n, 3), dtype=torch.float64, device=self.dev)
        W = torch.zeros_like(U)
        uf = u.reshape(3, -1)
        h3 = float(self.h.prod())
        for a, b in self._parts():
            flat, (dz, dy, dx), g = self._windows(a, b)
            w, wt = self._weights((dz, dy, dx), g)
            d = (dx, dy, dz)
            for c in range(3):
                uc = uf[c][flat]
                U[a:b, c] = h3 * (w * uc).sum((1, 2, 3))
                if torques:   # (d x u): component q gains d_p u_c with (q, p, c) cyclic, and loses it otherwise
                    p, q = (c + 1) % 3, (c + 2) % 3
                    W[a:b, p] += h3 * (wt * d[q] * uc).sum((1, 2, 3))
                    W[a:b, q] -= h3 * (wt * d[p] * uc).sum((1, 2, 3))
        return U, W

    def neighbours(self):
        """Ordered pairs (i, j) closer than r_c and their separations, part by part."""
        m = [max(int(float(e) / self.c["r_c"]), 3) for e in self.L]
        n = self.Y.shape[0]
        cell = [torch.clamp((self.Y[:, k] * (m[k] / float(self.L[k]))).long(), 0, m[k] - 1) for k in range(3)]
        key = cell[0] + m[0] * (cell[1] + m[1] * cell[2])
        order = torch.argsort(key)
        count = torch.bincount(key, minlength=m[0] * m[1] * m[2])
        start = torch.cumsum(count, 0) - count
        cap = int(count.max())
        table = torch.full((m[0] * m[1] * m[2], cap), -1, dtype=torch.long, device=self.dev)
        ks = key[order]
        table[ks, torch.arange(n, device=self.dev) - start[ks]] = order
        all_cells = torch.nonzero(count).reshape(-1)
        step = max(1, 30_000_000 // (27 * cap * cap))
        for a in range(0, all_cells.numel(), step):
            cc = all_cells[a:a + step]
            x, y, z = cc % m[0], (cc // m[0]) % m[1], cc // (m[0] * m[1])
            near = []
            for dz in (-1, 0, 1):
                for dy in (-1, 0, 1):
                    for dx in (-1, 0, 1):
                        near.append((x + dx) % m[0] + m[0] * ((y + dy) % m[1] + m[1] * ((z + dz) % m[2])))
            J = table[torch.stack(near, 1)].reshape(cc.numel(), 1, 27 * cap)
            I = table[cc][:, :, None]
            d = self.Y[I.clamp_min(0)] - self.Y[J.clamp_min(0)]
            d = d - self.L * torch.round(d / self.L)
            ok = ((d * d).sum(-1) < self.c["r_c"] ** 2) & (I >= 0) & (J >= 0) & (I != J)
            at = torch.nonzero(ok.reshape(-1)).reshape(-1)
            yield I.expand_as(ok).reshape(-1)[at], J.expand_as(ok).reshape(-1)[at], d.reshape(-1, 3)[at]

    def coefficients(self, x, torques):
        """The correction blocks as functions of the separation: al I + bt x x (forces), cr (cross products)
        and gm I + dl x x (torques), each the difference between the true kernels and the wide ones."""
        r2 = (x * x).sum(1)
        r = torch.sqrt(r2)
        s2, S2, dd, pi = SIGMA ** 2, self.S ** 2, self.dd, math.pi
        gauss = lambda v: (2 * pi * v) ** -1.5 * torch.exp(-r2 / (2 * v))   # normalised Gaussian of variance v
        e = torch.erfc(r / (2 * self.S)) - torch.erfc(r / (2 * SIGMA))
        gs, gS = gauss(2 * s2), gauss(2 * S2)
        t1, t2 = e / (8 * pi * r), e * s2 / (4 * pi * r ** 3)
        s3 = (s2 * s2 * gs - S2 * S2 * gS) / r2
        q, tt, rho = dd * gS, dd * dd * gS / (8 * S2), r2 / (2 * S2)
        al = t1 + t2 - 2 * s3 + q * (1 + 2 * S2 / r2) - tt * (2 - rho)
        bt = (t1 - 3 * t2 + 6 * s3 - q * (1 + 6 * S2 / r2) - tt * rho) / r2
        if not torques:
            return al, bt, None, None, None
        sd = 1.0 / (6.0 * math.sqrt(pi)) ** (1.0 / 3.0)
        v1, v2 = s2 + sd * sd, S2 + S2
        ef = torch.erfc(r / math.sqrt(2 * v2)) - torch.erfc(r / math.sqrt(2 * v1))
        g1, g2 = gauss(v1), gauss(v2)
        cr = (ef - 4 * pi * r * (v1 * g1 - v2 * g2)) / (8 * pi * r ** 3) + 0.25 * dd * g2 / v2
        et = torch.erfc(r / (2 * self.S)) - torch.erfc(r / (2 * sd))
        ga, gb = gauss(2 * sd * sd), gS
        w1, w2 = et / (8 * pi * r ** 3), 0.5 / r2
        gm = 0.5 * (-w1 + ((2 * sd * sd + r2) * ga - (2 * S2 + r2) * gb) * w2)
        dl = 0.5 * (3 * w1 - ((6 * sd * sd + r2) * ga - (6 * S2 + r2) * gb) * w2) / r2
        return al, bt, cr, gm, dl

    def self_terms(self):
        S, dd, pi = self.S, self.dd, math.pi
        sp = S * math.sqrt(pi)
        vf = 1 / (6 * pi) - 1 / (6 * pi * sp) + dd / (12 * sp ** 3) - dd * dd / (32 * S ** 5 * pi ** 1.5)
        return vf, 1 / (8 * pi) - 1 / (48 * sp ** 3)

    def pairs(self, F, T):
        vf, wt = self.self_terms()
        U = vf * F.double()
        W = wt * T.double() if T is not None else torch.zeros_like(U)
        for i, j, x in self.neighbours():
            al, bt, cr, gm, dl = (None if v is None else v[:, None] for v in self.coefficients(x, T is not None))
            Fj = F[j].double()
            u = al * Fj + bt * (x * Fj).sum(1, keepdim=True) * x
            if T is not None:
                Tj = T[j].double()
                u = u + cr * torch.linalg.cross(Tj, x)
                W.index_add_(0, i, cr * torch.linalg.cross(Fj, x) + gm * Tj + dl * (x * Tj).sum(1, keepdim=True) * x)
            U.index_add_(0, i, u)
        return U, W

    def product(self, F, T):
        U, W = self.gather(self.solve(self.spread(F, T)), T is not None)
        Up, Wp = self.pairs(F, T)
        return U + Up, (W + Wp if T is not None else None)

    def increment(self, xi, z):
        """Grid part and Lanczos square root of the pair part's force block, to convergence."""
        noise = xi.double().reshape(3, self.M[2], self.M[1], self.M[0])
        U, W = self.gather(self.solve(noise, half=True), True)
        amp = math.sqrt(2.0 / float(self.h.prod()))
        parts = []
        for i, j, x in self.neighbours():
            al, bt = self.coefficients(x, False)[:2]
            parts.append((i, j, x, al[:, None], bt[:, None]))
        vf = self.self_terms()[0]

        def times(v):
            out = vf * v
            for i, j, x, al, bt in parts:
                vj = v[j]
                out.index_add_(0, i, al * vj + bt * (x * vj).sum(1, keepdim=True) * x)
            return out

        norm = float(z.double().norm())
        V, alpha, beta = [z.double() / norm], [], []
        root = None
        for k in range(40):
            w = times(V[k])
            alpha.append(float((w * V[k]).sum()))
            for v in V:   # full orthogonalisation
                w = w - (w * v).sum() * v
            t = np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1)
            val, vec = np.linalg.eigh(t)
            new = vec @ (np.sqrt(val) * vec[0])
            if root is not None and np.linalg.norm(new - np.append(root, 0.0)) < 1e-13 * np.linalg.norm(new):
                break
            root = new
            beta.append(float(w.norm()))
            V.append(w / beta[-1])
        U = amp * U
        for c, v in zip(math.sqrt(2.0) * norm * new, V):
            U = U + float(c) * v
        return U, amp * W


def exact(case, seed):
    kind = case["kind"]
    if kind == "rigid":   # the converged solve takes minutes in 64 bits
        return None
    if kind == "serve":
        out = [_Exact(c, a[0]).product(a[1], a[2]) for c, a in _requests(case, seed)]
        return {"U": [u for u, _ in out], "W": [w for _, w in out]}
    counts = _counts(case)
    pos, F, T = _arrays(case, counts, seed)
    if kind == "brownian":
        U, W = _Exact(case, pos).increment(*_noise(case, seed))
        return {"U": U, "W": W}
    Us, Ws, a = [], [], 0
    for n in counts:
        if n:
            U, W = _Exact(case, pos[a:a + n]).product(F[a:a + n], None if T is None else T[a:a + n])
            Us.append(U)
            Ws.append(W)
        a += n
    return {"U": torch.cat(Us)} if T is None else {"U": torch.cat(Us), "W": torch.cat(Ws)}
