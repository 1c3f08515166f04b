"""Performance cases: what a user of this framework has it do.

An evolution case is the whole public call sequence of a host application that
owns its data: upload the state of every level from page-locked memory, advance
a number of coarse steps, download the state of every level.  The others are
the moving-box loop, the request server and the allocation-free constraint
monitor.  ``exact`` is an independent dense-array torch implementation of the
same method in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_09629_gb300 as sc
from paper_2503_09629_gb300 import workloads as W


def listed():
    return [
        # the smallest request of the serving mix: one coarse step of a 2-level wave, launch- and latency-bound
        {"name": "wave2_16", "kind": "wave", "nx": 16, "ny": 16, "nz": 16, "levels": 2, "fd": 4, "rk": 4, "steps": 1},
        # an ordinary wave run on a domain with odd, unequal extents and a ragged refined box
        {"name": "wave2_ragged", "kind": "wave", "nx": 61, "ny": 37, "nz": 45, "levels": 2, "fd": 4, "rk": 4, "steps": 4},
        # the Gaussian-pulse parity run: three levels, every level a union of uneven boxes
        {"name": "wave3_64_uneven", "kind": "uneven", "n": 64, "layout": 0, "steps": 2},
        # the largest convergence run of the same workload: arrays far larger than the L2 cache
        {"name": "wave3_256_uneven", "kind": "uneven", "n": 256, "layout": 0, "steps": 4},
        # 8th-order differences and third-order Runge-Kutta, the options of the wave path
        {"name": "wave2_40_fd8_rk3", "kind": "wave", "nx": 40, "ny": 40, "nz": 40, "levels": 2, "fd": 8, "rk": 3, "steps": 4},
        # the smallest black-hole hierarchy that nests: one coarse step
        {"name": "z4c3_20", "kind": "z4c", "n": 20, "levels": 3, "fd": 4, "rk": 4, "steps": 1},
        # an ordinary black-hole request of the serving mix
        {"name": "z4c3_48", "kind": "z4c", "n": 48, "levels": 3, "fd": 4, "rk": 4, "steps": 4},
        # the headline workload: binary black-hole data on seven nested levels, one coarse step
        {"name": "z4c7_64", "kind": "bl7", "steps": 1},
        # the paper's production discretisation: 8th-order differences
        {"name": "z4c3_64_fd8", "kind": "z4c", "n": 64, "levels": 3, "fd": 8, "rk": 4, "steps": 2},
        # a tracked binary: interpolate the shift, step, move the box stacks, twice
        {"name": "z4c_moving_32", "kind": "moving", "n": 32, "steps": 2},
        # an ensemble served on one GPU: a burst of mixed wave and black-hole requests, read back as they finish
        {"name": "serve_mixed_12", "kind": "serve", "requests": 12, "layout": 3},
        # the constraint monitor of a host application that owns all device memory, on a ragged box
        {"name": "constraints_ragged", "kind": "constraints", "nx": 26, "ny": 17, "nz": 25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["wave", "wave", "z4c", "z4c", "uneven", "constraints"])
    if kind == "wave":
        fd = rng.choice([4, 4, 8])
        n = [_log_int(rng, 20, 200) for _ in range(3)]
        return {"kind": "wave", "nx": n[0], "ny": n[1], "nz": n[2], "levels": rng.choice([1, 2, 3]), "fd": fd,
                "rk": rng.choice([4, 4, 3, 2]), "steps": rng.randint(1, 4)}
    if kind == "z4c":
        return {"kind": "z4c", "n": rng.randint(20, 64), "levels": rng.choice([2, 3, 4]), "fd": rng.choice([4, 4, 8]),
                "rk": rng.choice([4, 4, 4, 3]), "steps": rng.randint(1, 2)}
    if kind == "uneven":
        return {"kind": "uneven", "n": rng.choice([64, 128, 192]), "layout": rng.randint(1, 999), "steps": rng.randint(1, 4)}
    return {"kind": "constraints", "nx": rng.randint(5, 26), "ny": rng.randint(5, 26), "nz": rng.randint(5, 26)}


# ---- hierarchies ----------------------------------------------------------

def _nested(extents, levels):
    """Nested boxes: each finer box covers the central part of its parent, a quarter left free on every side."""
    boxes = [[((0, 0, 0), tuple(n - 1 for n in extents))]]
    lo, n = [0, 0, 0], list(extents)
    for _ in range(levels - 1):
        q = [max(v // 4, 5) if v >= 20 else v // 4 for v in n]
        lo = [2 * (lo[d] + q[d]) for d in range(3)]
        n = [2 * (n[d] - 2 * q[d]) for d in range(3)]
        boxes.append([(tuple(lo), tuple(lo[d] + n[d] - 1 for d in range(3)))])
    return boxes


def _hierarchy(case):
    k = case["kind"]
    if k == "uneven":
        return W.gaussian_3level(case["n"], case["layout"])
    if k == "bl7":
        return W.bl_7level()
    if k == "wave":
        ext = (case["nx"], case["ny"], case["nz"])
        return W.Hierarchy(system=W.WAVE, boxes=_nested(ext, case["levels"]), ncells0=ext, origin=(0.0, 0.0, 0.0),
                           h0=1.0 / max(ext), fd_order=case["fd"], rk_order=case["rk"])
    n = case["n"]
    return W.Hierarchy(system=W.Z4C, boxes=_nested((n, n, n), case["levels"]), ncells0=(n, n, n), origin=(-8.0, -8.0, -8.0),
                       h0=16.0 / n, bc=W.BC_RADIATIVE, fd_order=case["fd"], rk_order=case["rk"])


# ---- inputs ---------------------------------------------------------------

def _modes(rng, period, count, amplitude):
    """Smooth random field: a few plane waves of whole periods per domain length."""
    k = 2 * np.pi * rng.integers(1, 5, size=(count, 3)) / np.asarray(period)
    a = rng.uniform(-1, 1, count)
    return k, amplitude * a / np.abs(a).sum(), rng.uniform(0, 2 * np.pi, count)


def _fields(h, rng, punctures=None):
    """A function (x, y, z) -> (F, nz, ny, nx) of the initial data on coordinate axes (torch, float64)."""
    period = [n * h.h0 for n in h.ncells0]
    if h.system == W.WAVE:
        amp, width = rng.uniform(0.5, 1.5), 0.05 * max(period) * rng.uniform(0.8, 1.5)
        centre = [h.origin[d] + period[d] * rng.uniform(0.45, 0.55) for d in range(3)]
        noise = [_modes(rng, period, 8, 1e-3) for _ in range(2)]
    else:
        hf = h.h0 / 2 ** (h.nlevels - 1)
        if punctures is None:
            sep = 2.0 if h.nlevels == 7 else min(2.0, 0.1 * period[0])
            punctures = [(0.0, 0.0, s * sep / 2) for s in (1, -1)]
        # a quarter of the finest spacing off its corners: no cell centre of any level comes near a puncture
        centres = [[h.origin[d] + hf * (round((p[d] + rng.uniform(-3, 3) * hf - h.origin[d]) / hf) + 0.25) for d in range(3)]
                   for p in punctures]
        masses = rng.uniform(0.3, 0.7, 2)
        noise = [_modes(rng, period, 4, 1e-3) for _ in range(22)]

    def smooth(m, X, Y, Z):
        out = torch.zeros_like(X + Y + Z)
        for k, a, p in zip(*m):
            out += a * torch.sin(k[0] * X + k[1] * Y + k[2] * Z + p)
        return out

    def fn(x, y, z):
        X, Y, Z = x[None, None, :], y[None, :, None], z[:, None, None]
        if h.system == W.WAVE:
            r2 = (X - centre[0]) ** 2 + (Y - centre[1]) ** 2 + (Z - centre[2]) ** 2
            return torch.stack([amp * torch.exp(-r2 / (2 * width ** 2)) + smooth(noise[0], X, Y, Z), smooth(noise[1], X, Y, Z)])
        psi = torch.ones_like(X + Y + Z)
        for m, c in zip(masses, centres):
            psi += m / (2 * torch.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2))
        lapse = psi ** -2
        out = torch.stack([lapse * smooth(m, X, Y, Z) for m in noise])  # every field non-zero, regular at the punctures
        out[0] += lapse
        for f in (1, 4, 6):
            out[f] += 1.0
        out[18] += lapse
        return out

    return fn


def _axes(h, level, lo, hi, g, device):
    hl = h.h0 / 2 ** level
    return [h.origin[d] + (torch.arange(lo[d] - g, hi[d] + 1 + g, dtype=torch.float64, device=device) + 0.5) * hl for d in range(3)]


def _packed(h, fn, device):
    """The packed state: level by level, box by box, all fields; with the outer ghost shell on a radiative level 0."""
    parts = []
    for l, boxes in enumerate(h.boxes):
        g = h.ghost if l == 0 and h.bc == W.BC_RADIATIVE else 0
        for lo, hi in boxes:
            parts.append(fn(*_axes(h, l, lo, hi, g, device)).reshape(-1))
    return torch.cat(parts)


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    return out.copy_(t)


def _requests(case, seed):
    """The serving mix of the case's layout with wave numbers, masses and separations of the seed."""
    rng = np.random.default_rng(seed)
    out = []
    for _, h, steps in W.serving_requests(case["requests"], seed=case["layout"], burst=True):
        if h.system == W.WAVE:
            h.id_params = [float(rng.uniform(0.5, 1.5))] + [float(v) for v in rng.integers(1, 5, size=3)]
        else:
            s = float(rng.uniform(2.0, 6.0))
            m = rng.uniform(0.3, 0.7, 2)
            h.id_params = [float(m[0]), 0.0, 0.0, s / 2, float(m[1]), 0.0, 0.0, -s / 2]
        out.append((h, min(steps, 16)))
    return out


# off the symmetry planes and cell faces, so that the first steps of any inputs leave the boxes the same extents
MOVING = [(-1.65, 0.03, 0.05), (1.65, 0.03, 0.05)]


def _moving(case):
    h, _, radii, first = W.moving_bl(case["n"])
    h.boxes = W.moving_layout(h, MOVING, radii, first)
    return h, radii, first


class State:
    pass


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    s = State()
    s.case = case
    kind = case["kind"]
    if kind == "serve":
        s.requests = _requests(case, seed)
        s.server = sc.Server(32 << 30, max_active=8, depth=2)
        return s
    if kind == "constraints":
        s.n, s.h = (case["nx"], case["ny"], case["nz"]), 0.125
        s.data = _constraint_data(case, seed)
        s.out = torch.empty((7,) + s.n[::-1], dtype=torch.float64, device="cuda")
        return s
    if kind == "moving":
        h, s.radii, s.first = _moving(case)
        s.positions = MOVING
        fn = _fields(h, rng, punctures=s.positions)
    else:
        h = _hierarchy(case)
        fn = _fields(h, rng)
    s.h = h
    s.ghosted = h.bc == W.BC_RADIATIVE
    s.src = _pinned(_packed(h, fn, "cuda"))
    s.ctx = sc.Context(h)
    s.dst = torch.empty(s.src.shape, dtype=torch.float64, pin_memory=True)
    return s


def run(state):
    kind = state.case["kind"]
    if kind == "serve":
        out = {}
        tickets = [state.server.sc_server_submit(h, n) for h, n in state.requests]

        def finished(t):
            h = state.server.hier[t]
            fields = [state.server.sc_server_read(t, l, 0, f) for l in range(h.nlevels) for f in range(h.nfields())]
            out["request%d" % tickets.index(t)] = np.concatenate([a.reshape(-1) for a in fields])
            state.server.sc_server_release(t)

        state.server.run_until_done(tickets, on_done=finished)
        return out
    if kind == "constraints":
        sc.sc_z4c_constraints_noalloc(state.data.data_ptr(), state.out.data_ptr(), state.n, state.h,
                                      torch.cuda.current_stream().cuda_stream)
        return state.out
    ctx, steps = state.ctx, state.case["steps"]
    if kind == "moving":
        ctx.sc_regrid(state.h.boxes)  # a restart: back to the layout that the state belongs to
        ctx.sc_set_state(state.src.data_ptr(), True)
        positions = state.positions
        for _ in range(steps):
            moved = W.track_punctures(ctx, positions, state.h.cfl * state.h.h0)
            ctx.sc_advance(1)
            positions = moved
            ctx.sc_regrid(W.moving_layout(state.h, positions, state.radii, state.first))
        return ctx.sc_get_state(None, True)
    ctx.sc_set_state(state.src.data_ptr(), state.ghosted)
    ctx.sc_advance(steps)
    ctx.sc_get_state(state.dst.data_ptr(), state.ghosted)
    return state.dst


# ---- work -----------------------------------------------------------------

def _flops_per_update(h):
    """Floating-point operations of one cell and Runge-Kutta step: right-hand side, dissipation and stage update."""
    if h.system == W.WAVE:
        return (20 if h.fd_order == 4 else 34) * h.rk_order
    return (3151 if h.fd_order == 4 else 3976) * h.rk_order


def work(case):
    if case["kind"] == "constraints":
        n = case["nx"] * case["ny"] * case["nz"]
        g = (case["nx"] + 6) * (case["ny"] + 6) * (case["nz"] + 6)
        return {"bytes": 8.0 * (22 * g + 7 * n), "flops": 3151.0 * n}
    if case["kind"] == "serve":
        runs = _requests(case, 0)
    elif case["kind"] == "moving":
        runs = [(_moving(case)[0], case["steps"])]
    else:
        runs = [(_hierarchy(case), case["steps"])]
    bytes_, flops = 0.0, 0.0
    for h, steps in runs:
        cells = sum(h.interior_cells(l) for l in range(h.nlevels))
        bytes_ += 8.0 * cells * h.nfields() * (1 if case["kind"] == "serve" else 2)  # a served request starts from parameters
        flops += steps * h.zone_updates_per_coarse_step()[1] * _flops_per_update(h)
    return {"bytes": bytes_, "flops": flops}


# ---- the method in plain torch --------------------------------------------

SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))


def _lagrange(nodes, p):
    return [math.prod((p - b) / (a - b) for b in nodes if b != a) for a in nodes]


def _shift(u, d, m):
    """u at m cells further along x, y or z (d = 0, 1, 2; the last axis is x)."""
    return torch.roll(u, -m, dims=u.dim() - 1 - d)


def _d1(u, d, h, order):
    w = (8.0, -1.0) if order == 4 else (672.0, -168.0, 32.0, -3.0)
    return sum(c * (_shift(u, d, m) - _shift(u, d, -m)) for m, c in enumerate(w, 1)) / ((12.0 if order == 4 else 840.0) * h)


def _d2(u, d, h, order):
    w = (-30.0, 16.0, -1.0) if order == 4 else (-14350.0, 8064.0, -1008.0, 128.0, -9.0)
    s = w[0] * u + sum(c * (_shift(u, d, m) + _shift(u, d, -m)) for m, c in enumerate(w[1:], 1))
    return s / ((12.0 if order == 4 else 5040.0) * h * h)


def _ko(u):
    out = -60.0 * u
    for d in range(3):
        for m, c in ((1, 15.0), (2, -6.0), (3, 1.0)):
            out = out + c * (_shift(u, d, m) + _shift(u, d, -m))
    return out


def _full(u):
    """Six symmetric components to (3, 3, ...)."""
    return torch.stack([torch.stack([u[SYM[i][j]] for j in range(3)]) for i in range(3)])


def _geometry(U, h, order):
    """The quantities that the right-hand side and the constraints share."""
    e = torch.einsum
    D = lambda u: torch.stack([_d1(u, d, h, order) for d in range(3)])  # noqa: E731
    first = torch.stack([D(U[f]) for f in range(22)])  # [f][d]

    def hess(f):
        pure = [_d2(U[f], d, h, order) for d in range(3)]
        mixed = {(a, b): _d1(first[f][a], b, h, order) for a, b in ((0, 1), (0, 2), (1, 2))}
        return torch.stack([torch.stack([pure[i] if i == j else mixed[(min(i, j), max(i, j))] for j in range(3)]) for i in range(3)])

    q = {"g": _full(U[1:7]), "A": _full(U[8:14]), "first": first}
    g = q["g"]
    adj = torch.stack([torch.stack([g[(j + 1) % 3][(i + 1) % 3] * g[(j + 2) % 3][(i + 2) % 3]
                                    - g[(j + 1) % 3][(i + 2) % 3] * g[(j + 2) % 3][(i + 1) % 3] for j in range(3)]) for i in range(3)])
    gu = q["gu"] = adj / (g[0] * adj[:, 0]).sum(0)
    dg = torch.stack([_full(first[1:7, d]) for d in range(3)])  # [k][i][j] = d_k g_ij
    Gl = q["Gl"] = 0.5 * (dg.permute(1, 2, 0, 3, 4, 5) + dg.permute(1, 0, 2, 3, 4, 5) - dg)  # [k][i][j]
    Gu = q["Gu"] = e("kl...,lij...->kij...", gu, Gl)
    q["Gd"] = e("jk...,ijk...->i...", gu, Gu)
    ddg = torch.stack([hess(1 + s) for s in range(6)])  # [s][l][m]
    Wf, dW = U[0], first[0]
    DDW = hess(0) - e("kij...,k...->ij...", Gu, dW)
    trDDW, dWdW = e("lm...,lm...", gu, DDW), e("lm...,l...,m...", gu, dW, dW)
    lap = e("lm...,slm...->s...", gu, ddg)
    dGam = first[14:17]
    rt = -0.5 * _full(lap)
    t = e("ki...,kj...->ij...", g, dGam)
    rt = rt + 0.5 * (t + t.transpose(0, 1))
    t = e("k...,ijk...->ij...", q["Gd"], Gl)
    rt = rt + 0.5 * (t + t.transpose(0, 1))
    up = e("lm...,jkm...->jkl...", gu, Gl)
    t = e("kli...,jkl...->ij...", Gu, up)
    rt = rt + t + t.transpose(0, 1) + e("kim...,kjm...->ij...", Gu, e("lm...,klj...->kjm...", gu, Gl))
    q["R"] = rt + (DDW + g * trDDW) / Wf - 2.0 * g * dWdW / Wf ** 2
    q["Rsc"] = Wf ** 2 * e("ij...,ij...", gu, q["R"])
    q["Am"] = e("ik...,kj...->ij...", gu, q["A"])
    q["Auu"] = e("ik...,kj...->ij...", q["Am"], gu)
    q["AA"] = e("ij...,ij...", q["A"], q["Auu"])
    q["hess"] = hess
    return q


def _z4c_rhs(U, h, H):
    e = torch.einsum
    q = _geometry(U, h, H.fd_order)
    g, A, gu, Gu, Gd, R, Am, Auu, AA, first, hess = (q[k] for k in ("g", "A", "gu", "Gu", "Gd", "R", "Am", "Auu", "AA", "first", "hess"))
    Wf, Kh, Th, al, Gam, be = U[0], U[7], U[17], U[18], U[14:17], U[19:22]
    dW, dal, dbe = first[0], first[18], first[19:22]
    Gp = e("kij...,k...->ij...", Gu, dal)
    wa = e("i...,j...->ij...", dal, dW)
    Gp = Gp - (wa + wa.transpose(0, 1) - g * e("kl...,l...,k...", gu, dW, dal)) / Wf
    DDal = hess(18) - Gp
    divb, Kt = dbe[0, 0] + dbe[1, 1] + dbe[2, 2], Kh + 2.0 * Th
    adv = e("d...,fd...->f...", be, first)
    out = adv.clone()
    out[0] += Wf * (al * Kt - divb) / 3.0
    X = al * R - DDal
    trX = e("ij...,ij...", gu, X)
    lie = lambda T: e("ki...,kj...->ij...", T, dbe) + e("kj...,ki...->ij...", T, dbe)  # noqa: E731
    dtg = -2.0 * al * A - (2.0 / 3.0) * g * divb + lie(g)
    dtA = Wf ** 2 * (X - g * trX / 3.0) + al * Kt * A - (2.0 / 3.0) * A * divb + lie(A) - 2.0 * al * e("ki...,kj...->ij...", Am, A)
    for s, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        out[1 + s] += dtg[i, j]
        out[8 + s] += dtA[i, j]
    out[7] += -Wf ** 2 * e("ij...,ij...", gu, DDal) + al * (AA + Kt ** 2 / 3.0) + al * H.kappa1 * (1.0 - H.kappa2) * Th
    ddbe = torch.stack([hess(19 + i) for i in range(3)])
    br = e("ijk...,jk...->i...", Gu, Auu) - 3.0 * e("ij...,j...->i...", Auu, dW) / Wf
    br = br - e("ij...,j...->i...", gu, 2.0 * first[7] + first[17]) / 3.0
    out[14:17] += (-2.0 * e("ij...,j...->i...", Auu, dal) + 2.0 * al * br + e("jk...,ijk...->i...", gu, ddbe)
                   + e("ij...,kjk...->i...", gu, ddbe) / 3.0 - e("j...,ij...->i...", Gd, dbe) + (2.0 / 3.0) * Gd * divb
                   - 2.0 * H.kappa1 * al * (Gam - Gd))
    out[17] += 0.5 * al * (q["Rsc"] - AA + (2.0 / 3.0) * Kt ** 2) - al * H.kappa1 * (2.0 + H.kappa2) * Th
    out[18] += -2.0 * al * Kh
    out[19:22] += 0.75 * Gam - H.eta * be
    return out + H.ko_sigma / (64.0 * h) * _ko(U)


class _Level:
    def __init__(self, H, l, dev):
        g, bx = H.ghost, H.boxes[l]
        self.h = H.h0 / 2 ** l
        self.org = [min(b[0][d] for b in bx) - g for d in range(3)]
        self.ext = [max(b[1][d] for b in bx) + g + 1 - self.org[d] for d in range(3)]
        self.inside = torch.zeros(self.ext[::-1], dtype=torch.bool, device=dev)
        shell = torch.zeros_like(self.inside)
        for lo, hi in bx:
            self.inside[self.cut(lo, hi, 0)] = True
            shell[self.cut(lo, hi, g)] = True
        self.ghosts = shell & ~self.inside

    def cut(self, lo, hi, g):
        return tuple(slice(lo[d] - g - self.org[d], hi[d] + g + 1 - self.org[d]) for d in (2, 1, 0))

    def matrices(self, other, dev, restrict):
        """Per axis the interpolation matrix from `other`'s array onto this one's (rows without a stencil are zero)."""
        out = []
        for d in range(3):
            M = torch.zeros(self.ext[d], other.ext[d], dtype=torch.float64)
            for r in range(self.ext[d]):
                i = r + self.org[d]
                first = 2 * i - 2 if restrict else i // 2 - 3 + (i & 1)
                w = _lagrange([m - 2.5 for m in range(6)], 0.0) if restrict else _lagrange([first + m - i // 2 for m in range(6)], 0.25 if i & 1 else -0.25)
                a = first - other.org[d]
                if a >= 0 and a + 6 <= other.ext[d]:
                    M[r, a:a + 6] = torch.tensor(w, dtype=torch.float64)
            out.append(M.to(dev))
        return out


def _apply(M, u):
    u = torch.matmul(u, M[0].T)
    u = torch.matmul(M[1], u)
    return torch.einsum("ab,fbyx->fayx", M[2], u)


def _dense(rk, t, m):
    """m-th derivative in t of the dense-output weights of the stage vectors."""
    P = {4: [(0, 1, -1.5, 2 / 3), (0, 0, 1, -2 / 3), (0, 0, 1, -2 / 3), (0, 0, -0.5, 2 / 3)],
         3: [(0, 1, -1.25, 0.5), (0, 0, 0, 0), (0, 0, 2.25, -1.5), (0, 0, -1, 1)],
         2: [(0, 1, -1, 0), (0, 0, 1, 0), (0, 0, 0, 0), (0, 0, 0, 0)]}[rk]
    return np.array([np.polyval(np.polyder(np.array(p[::-1], dtype=float), m) if m else np.array(p[::-1], dtype=float), t) for p in P])


def _ghost_weights(rk, H, t, which):
    """Coefficients of the parent's k1..k4 in a fine ghost value: stage input `which`, or the end of the substep (0)."""
    if which == 0:
        return H * _dense(rk, t + 0.5, 0)
    h, y0, y1, y2 = 0.5 * H, H * _dense(rk, t, 0), _dense(rk, t, 1), _dense(rk, t, 2) / H
    if which == 1:
        return y0
    if rk == 4:
        y3, fy = _dense(4, t, 3) / H ** 2, np.array([0.0, -4.0, 4.0, 0.0]) / H ** 2
        if which == 2:
            return y0 + 0.5 * h * y1
        if which == 3:
            return y0 + 0.5 * h * y1 + 0.25 * h * h * y2 + h ** 3 / 16 * (y3 - fy)
        return y0 + h * y1 + 0.5 * h * h * y2 + h ** 3 / 8 * (y3 + fy)
    if rk == 3:
        return y0 + h / 3 * y1 if which == 2 else y0 + 2 * h / 3 * y1 + 2 * h * h / 9 * y2
    return y0 + 0.5 * h * y1


class _Evolution:
    """Subcycled evolution on dense level arrays."""

    def __init__(self, H, fn, dev):
        self.H, self.dev = H, dev
        self.lev = [_Level(H, l, dev) for l in range(H.nlevels)]
        self.radiative = H.bc == W.BC_RADIATIVE
        for l, L in enumerate(self.lev):
            hi = [L.org[d] + L.ext[d] - 1 for d in range(3)]
            L.y = fn(*_axes(H, l, L.org, hi, 0, dev))
            L.evolved = torch.ones_like(L.inside) if l == 0 and self.radiative else L.inside
            if l:
                P = self.lev[l - 1]
                L.prolong, L.restrict = L.matrices(P, dev, False), P.matrices(L, dev, True)
                kids = torch.zeros_like(P.inside)
                z = [2 * P.org[d] - L.org[d] for d in range(3)]
                pad = torch.zeros([2 * n for n in P.ext[::-1]], dtype=torch.bool, device=dev)  # fine cells below the parent array
                src = [slice(max(0, z[d]), min(L.ext[d], z[d] + 2 * P.ext[d])) for d in range(3)]
                dst = [slice(src[d].start - z[d], src[d].stop - z[d]) for d in range(3)]
                pad[dst[2], dst[1], dst[0]] = L.inside[src[2], src[1], src[0]]
                kids = pad.reshape(P.ext[2], 2, P.ext[1], 2, P.ext[0], 2).all(5).all(3).all(1)
                L.covered = kids & P.inside
            elif not self.radiative:
                n = H.ncells0
                L.wrap = [(torch.arange(L.ext[d], device=dev) + L.org[d]) % n[d] - L.org[d] for d in range(3)]

    def rhs(self, l, Y):
        L = self.lev[l]
        if self.H.system == W.WAVE:
            return torch.stack([Y[1], sum(_d2(Y[0], d, L.h, self.H.fd_order) for d in range(3))])
        out = _z4c_rhs(Y, L.h, self.H)
        if l == 0 and self.radiative:
            x = _axes(self.H, 0, L.org, [L.org[d] + L.ext[d] - 1 for d in range(3)], 0, self.dev)
            X = (x[0][None, None, :], x[1][None, :, None], x[2][:, None, None])
            r = torch.sqrt(X[0] ** 2 + X[1] ** 2 + X[2] ** 2)
            inf = torch.zeros(22, 1, 1, 1, dtype=torch.float64, device=self.dev)
            inf[[0, 1, 4, 6, 18]] = 1.0
            k = -(Y - inf) / r
            for d in range(3):
                der = (_shift(Y, d, 1) - _shift(Y, d, -1)) / (2 * L.h)
                ax = 3 - d
                s = lambda i: Y.select(ax, i)  # noqa: E731
                der.select(ax, 0).copy_((-3 * s(0) + 4 * s(1) - s(2)) / (2 * L.h))
                der.select(ax, L.ext[d] - 1).copy_((3 * s(-1) - 4 * s(-2) + s(-3)) / (2 * L.h))
                k -= X[d] / r * der
            out = torch.where(L.inside, out, k)
        return out

    def fill(self, l, Y, which, theta):
        L = self.lev[l]
        if l == 0:
            if not self.radiative:
                Y.copy_(Y[:, L.wrap[2]][:, :, L.wrap[1]][:, :, :, L.wrap[0]])
            return
        c = _ghost_weights(self.H.rk_order, self.H.cfl * self.lev[l - 1].h, theta, which)
        v = L.pv[0] + sum(float(cj) * p for cj, p in zip(c, L.pv[1:]) if cj)
        Y[:, L.ghosts] = v[:, L.ghosts]

    def step(self, l, theta):
        L, rk = self.lev[l], self.H.rk_order
        dt = self.H.cfl * L.h
        mult = {4: (0.5, 0.5, 1.0), 3: (1 / 3, 2 / 3), 2: (0.5,)}[rk]
        Y, L.k = L.y, []
        L.yn = L.y
        for s in range(rk):
            self.fill(l, Y, s + 1, theta)
            k = torch.where(L.evolved, self.rhs(l, Y), 0.0)
            L.k.append(k)
            if s + 1 < rk:
                Y = L.yn + mult[s] * dt * k
        k = L.k
        inc = {4: lambda: (k[0] + 2 * k[1] + 2 * k[2] + k[3]) / 6, 3: lambda: (k[0] + 3 * k[2]) / 4, 2: lambda: k[1]}[rk]()
        L.y = L.yn + dt * inc
        if l or rk == 3:
            self.fill(l, L.y, 0, theta)
        if rk == 3 and l + 1 < len(self.lev):
            L.k.append(torch.where(L.evolved, self.rhs(l, L.y), 0.0))

    def children(self, l):
        L, F = self.lev[l], self.lev[l + 1]
        F.pv = [_apply(F.prolong, v) for v in [L.yn] + L.k]
        F.pv += [torch.zeros_like(F.pv[0])] * (5 - len(F.pv))
        for s in range(2):
            self.step(l + 1, 0.5 * s)
            if l + 2 < len(self.lev):
                self.children(l + 1)
        r = _apply(F.restrict, F.y)
        L.y = torch.where(F.covered, r, L.y)

    def advance(self, n):
        for _ in range(n):
            self.step(0, 0.0)
            if len(self.lev) > 1:
                self.children(0)

    def packed(self):
        parts = []
        for l, L in enumerate(self.lev):
            g = self.H.ghost if l == 0 and self.radiative else 0
            parts += [L.y[(slice(None),) + L.cut(lo, hi, g)].reshape(-1) for lo, hi in self.H.boxes[l]]
        return torch.cat(parts)


def _constraint_data(case, seed):
    """One ghosted box of black-hole data, spacing 0.125, the punctures off its centre."""
    n = (case["nx"], case["ny"], case["nz"])
    h = W.Hierarchy(system=W.Z4C, boxes=[[((0, 0, 0), tuple(v - 1 for v in n))]], ncells0=n,
                    origin=tuple(-0.0625 * v for v in n), h0=0.125, bc=W.BC_RADIATIVE)
    fn = _fields(h, np.random.default_rng(seed), punctures=[(0.5, 0.0, 0.25), (-0.5, 0.0, -0.25)])
    return fn(*_axes(h, 0, (0, 0, 0), tuple(v - 1 for v in n), 3, "cuda" if torch.cuda.is_available() else "cpu")).contiguous()


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "constraints":
        U, h, e = _constraint_data(case, seed), 0.125, torch.einsum
        q = _geometry(U, h, 4)
        gu, Auu, first = q["gu"], q["Auu"], q["first"]
        Kt = U[7] + 2.0 * U[17]
        dg = torch.stack([_full(first[1:7, d]) for d in range(3)])
        dA = torch.stack([_full(first[8:14, d]) for d in range(3)])
        dgu = -e("ac...,bd...,mcd...->mab...", gu, gu, dg)
        M = (e("jam...,jp...,mp...->a...", dgu, gu, q["A"]) + e("am...,jjp...,mp...->a...", gu, dgu, q["A"])
             + e("am...,jp...,jmp...->a...", gu, gu, dA) + e("abc...,bc...->a...", q["Gu"], Auu)
             - 3.0 * e("ab...,b...->a...", Auu, first[0]) / U[0] - (2.0 / 3.0) * e("ab...,b...->a...", gu, first[7] + 2.0 * first[17]))
        out = torch.cat([(q["Rsc"] + (2.0 / 3.0) * Kt ** 2 - q["AA"])[None], M, U[14:17] - q["Gd"]])
        return out[:, 3:-3, 3:-3, 3:-3].contiguous()
    if kind in ("serve", "moving"):
        return None  # many runs, or layouts that move between steps
    h = _hierarchy(case)
    if kind == "bl7" or sum(h.interior_cells(l) for l in range(h.nlevels)) > (1 << 21):
        return None  # over 20 seconds, or too large for this plain form
    ev = _Evolution(h, _fields(h, np.random.default_rng(seed)), dev)
    ev.advance(case["steps"])
    return ev.packed()
