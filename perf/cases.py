"""The work that users of this library have it do, as cases that can be timed and checked.

Every case goes through the public entry points (`solver.Block`, `solver.Batch`, `solver.Pipe`):
a residual, a Runge-Kutta step, a time step with its CFL bound, the steps of many blocks at once
(device states, host states, linked blocks).  Grids and flows are those of `inputs.py` (the wavy
periodic box, the cylinder O-grid, the C-grid around a wing, the randomised grid of the shock
tests), with sizes from the tests and the benchmark or drawn from the same ranges.

`exact` evaluates the same scheme in 64 bits with plain torch operations: metrics, reference-state
differences, characteristic reconstruction and Runge-Kutta stages, written here from the formulas
of the paper, on the nodes and the (float or double) state that the call gets.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_05886_gb300 import inputs as I

WENO5, LINEAR, WENO7, WENOCU6 = 0, 1, 2, 3
F64, F32 = 0, 1
# floating-point operations a point needs in one direction pass: projections and differences of
# the stencil, reconstruction, eigensystem, reference state, face flux, residual
PASS_FLOPS = {WENO5: 2000, LINEAR: 700, WENO7: 2900, WENOCU6: 2600}
DEVICE = "cuda"
BOX = 10.0          # side of the periodic wavy box


# --------------------------------------------------------------------------- the cases
def listed():
    d = dict(nk=1, order=6, scheme=WENO5, precision=F32, characteristic=1, global_lf=0)
    return [
        # the free-stream check of a small 2-D grid: one residual, for an outside time integrator
        dict(d, name="rhs_2d_33_f64", kind="rhs", grid="wavy2d", ni=33, nj=33, precision=F64),
        # an accuracy study: the 2-D vortex with linear upwind in double precision
        dict(d, name="step_2d_128_f64_linear", kind="step", grid="wavy2d", ni=128, nj=128, scheme=LINEAR, precision=F64),
        # a shock on a randomised grid with global Lax-Friedrichs speeds, as in the paper's shock tests
        dict(d, name="step_shock_200_f64", kind="step", grid="shock2d", ni=200, nj=200, precision=F64, global_lf=1),
        # one small block of a cylinder mesh with a slip wall, stepped by itself
        dict(d, name="step_ogrid_48x37x29", kind="step", grid="ogrid_wall", ni=48, nj=37, nk=29),
        # the loop of a simulation: the CFL bound, then a step of that size, on a ragged O-grid
        dict(d, name="advance_ogrid_181x97x61", kind="advance", grid="ogrid_wall", ni=181, nj=97, nk=61),
        # a large single block in the mixed precision, the scheme of the paper
        dict(d, name="step_wavy_256", kind="step", grid="wavy", ni=256, nj=256, nk=256),
        # the residual of the seventh-order scheme with eighth-order metrics
        dict(d, name="rhs_wavy_150_weno7", kind="rhs", grid="wavy", ni=150, nj=141, nk=133, order=8, scheme=WENO7),
        # a double-precision production block
        dict(d, name="step_wavy_96_f64", kind="step", grid="wavy", ni=96, nj=96, nk=96, precision=F64),
        # the multi-block benchmark: 64 uneven blocks advanced together (Mach 3, half O-grids, half wavy boxes)
        dict(d, name="batch_64", kind="batch", grid="mixed", blocks=64, lo=32, hi=128, ni=0, nj=0, nk=0),
        # fewer and smaller blocks with the cheaper linear scheme
        dict(d, name="batch_20_linear", kind="batch", grid="mixed", blocks=20, lo=32, hi=96, ni=0, nj=0, nk=0, scheme=LINEAR),
        # blocks whose states live in host memory: copied in, advanced and copied back every step
        dict(d, name="pipe_16", kind="pipe", grid="mixed", blocks=16, lo=32, hi=128, ni=0, nj=0, nk=0),
        # the C-grid around a wing (slip wall, wake cut, far field), split into linked blocks of one batch
        dict(d, name="linked_wing_192x96x80", kind="linked", grid="wing", ni=192, nj=96, nk=80, parts=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c = dict(nk=1, order=6, scheme=WENO5, precision=F32, characteristic=1, global_lf=0)
    kind = rng.choice(["2d", "2d", "shock", "rhs", "step", "step", "advance", "batch", "pipe", "linked"])
    c["order"] = rng.choice([2, 4, 6, 6, 6, 8])
    c["scheme"] = rng.choice([WENO5, WENO5, LINEAR, LINEAR, WENO7, WENOCU6])
    if kind == "2d":
        c.update(kind=rng.choice(["rhs", "step"]), grid="wavy2d", ni=_log(rng, 20, 512), nj=_log(rng, 20, 512),
                 precision=rng.choice([F64, F64, F32]), characteristic=rng.choice([1, 1, 1, 0]))
    elif kind == "shock":
        n = _log(rng, 48, 400)
        c.update(kind="step", grid="shock2d", ni=n, nj=n, scheme=WENO5,
                 precision=rng.choice([F64, F32]), global_lf=1)
    elif kind in ("rhs", "step", "advance"):
        c["precision"] = rng.choice([F32, F32, F32, F64])
        top = 190 if c["precision"] == F32 else 80
        c.update(kind=kind, grid="wavy" if kind == "rhs" else rng.choice(["wavy", "ogrid_wall", "wing"]),
                 ni=_log(rng, 20, top), nj=_log(rng, 20, top), nk=_log(rng, 20, top),
                 characteristic=rng.choice([1, 1, 1, 0]))
        if c["grid"] == "wing":
            c.update(ni=2 * max(c["ni"] // 2, 32), nj=max(c["nj"], 40), scheme=rng.choice([WENO5, LINEAR]))
    elif kind == "linked":
        c.update(kind=kind, grid=rng.choice(["wing", "wavy"]), ni=2 * _log(rng, 32, 100), nj=_log(rng, 40, 110),
                 nk=_log(rng, 40, 110), parts=rng.randint(2, 8), scheme=rng.choice([WENO5, LINEAR]))
    else:
        lo = _log(rng, 20, 40)
        c.update(kind=kind, grid="mixed", blocks=_log(rng, 2, 32), lo=lo, hi=_log(rng, lo + 8, 110), ni=0, nj=0, nk=0)
    return c


# --------------------------------------------------------------------------- grids and flows
def _ghost(c):
    return max(4 if c["scheme"] == WENO7 else 3, c["order"] // 2)


def _node_ghost(c):
    return _ghost(c) + 3 * (c["order"] // 2)


def _axis(n, gn):
    return torch.arange(-gn, n + gn, dtype=torch.float64, device=DEVICE)


def _wavy(n, gn, amp):
    """The periodic wavy box, x_a = L (xi_a + amp sin sin sin), nodes made on the GPU."""
    dims = 2 if n[2] == 1 else 3
    ax = [_axis(n[a], gn) / n[a] for a in range(dims)]
    s = torch.full((), amp, dtype=torch.float64, device=DEVICE)
    pos = []
    for a in range(dims):
        shape = [1] * dims
        shape[dims - 1 - a] = -1
        pos.append(ax[a].reshape(shape))
        s = s * torch.sin(2 * math.pi * pos[a])
    nodes = torch.stack([BOX * (p + s) for p in pos])
    per = (I.BC_PERIODIC, I.BC_PERIODIC)
    return I.Grid(dims, tuple(n), gn, nodes.cpu().numpy(), (per, per, per), "wavy")


def _ogrid(n, gn, span, wall):
    """The cylinder O-grid: i around, j radial with a tanh stretch, k along the span."""
    ni, nj, nk = n
    th = (2 * math.pi / ni * _axis(ni, gn)).reshape(1, 1, -1)
    j = _axis(nj, gn).reshape(1, -1, 1)
    e = (j + 0.5) / (nj - 0.5) if wall else j / (nj - 1)
    r = 0.5 + 19.5 * (1.0 - torch.tanh(3.0 * (1.0 - e)) / math.tanh(3.0))
    z = (span / nk * _axis(nk, gn)).reshape(-1, 1, 1)
    one = torch.ones((nk + 2 * gn, nj + 2 * gn, ni + 2 * gn), dtype=torch.float64, device=DEVICE)
    nodes = torch.stack([r * torch.cos(th) * one, r * torch.sin(th) * one, z * one])
    per = (I.BC_PERIODIC, I.BC_PERIODIC)
    inner = I.BC_SLIP_WALL if wall else I.BC_EXTRAP
    return I.Grid(3, tuple(n), gn, nodes.cpu().numpy(), (per, (inner, I.BC_FARFIELD), per), "ogrid")


def _one_grid(c, rng):
    n, gn = (c["ni"], c["nj"], c["nk"]), _node_ghost(c)
    if c["grid"] in ("wavy", "wavy2d"):
        return _wavy(n, gn, rng.uniform(0.06, 0.09))
    if c["grid"] == "ogrid_wall":
        return _ogrid(n, gn, rng.uniform(1.0, 8.0), True)
    if c["grid"] == "shock2d":
        return I.random_grid_2d(c["ni"], L=1.0, frac=0.1, seed=int(rng.integers(1 << 30)), Gn=gn)
    return I.cgrid_wing(n, first_cell=1e-3, Gn=gn)


def _perturbed(q, n, rng, amp):
    """Smooth seeded Fourier modes in index space on top of a state."""
    ni, nj, nk = n
    ax = [torch.arange(m, dtype=torch.float64, device=DEVICE) / m for m in (ni, nj, nk)]
    for v in range(5):
        f = torch.zeros((nk, nj, ni), dtype=torch.float64, device=DEVICE)
        for _ in range(2):
            k = rng.integers(1, 3, size=3)
            ph = rng.uniform(0, 2 * math.pi, size=3)
            w = [torch.sin(2 * math.pi * int(k[a]) * ax[a] + float(ph[a])) for a in range(3)]
            f += w[0].reshape(1, 1, -1) * w[1].reshape(1, -1, 1) * w[2].reshape(-1, 1, 1)
        q[v] = q[v] * (1 + 0.3 * amp * f) if v in (0, 4) else (q[v] + amp * f if v < 3 or nk > 1 else q[v])
    return q


def _flow(c, grid, rng):
    """(q_inf, state): the flow a block of this grid starts from, float64 on the GPU."""
    n = tuple(int(v) for v in grid.n)
    if c["grid"] == "shock2d":
        qinf = I.uniform_qinf(0.0)
        q = torch.as_tensor(I.normal_shock_state(grid, rng.uniform(0.2, 0.6), mach=2.0)).to(DEVICE)
        return qinf, q
    if c["grid"] == "mixed":
        qinf, amp = I.uniform_qinf(3.0), 1e-3
    elif c["grid"] in ("wavy", "wavy2d"):
        qinf, amp = I.uniform_qinf(0.8, rho=1.0, p=1.0), 1e-2
    else:
        qinf, amp = I.uniform_qinf(0.5, 3.0), 1e-2
    q = torch.as_tensor(qinf, device=DEVICE).reshape(5, 1, 1, 1).repeat(1, n[2], n[1], n[0])
    if c["grid"] in ("wavy", "wavy2d"):
        g = grid.Gn
        xy = grid.nodes[:2, g:-g, g:-g][:, None] if grid.dims == 2 else grid.nodes[:2, g:-g, g:-g, g:-g]
        x, y = (torch.as_tensor(np.ascontiguousarray(a)).to(DEVICE) for a in xy)
        dx, dy = x - 0.5 * BOX, y - 0.5 * BOX
        u0, r2 = 0.8 * math.sqrt(1.4), dx * dx + dy * dy
        f = 5.0 / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
        t = 1.0 - 0.4 * 25.0 / (8 * 1.4 * math.pi ** 2) * torch.exp(1 - r2)
        rho = t ** 2.5
        u, v = u0 - f * dy, f * dx
        q = torch.stack([rho, rho * u, rho * v, 0 * rho, rho * t / 0.4 + 0.5 * rho * (u * u + v * v)])
    return qinf, _perturbed(q, n, rng, amp)


def _blocks(c, seed):
    """The case's (grid, q_inf, state in the case's precision) blocks; the linked case's unsplit one."""
    rng = np.random.default_rng([seed, 2101])
    dt = torch.float32 if c["precision"] == F32 else torch.float64
    out = []
    if c["grid"] == "mixed":
        sizes = I.batched_block_sizes(c["blocks"], c["lo"], c["hi"], seed=4)   # the mesh; the flow is the seed's
        grids = [_ogrid(n, _node_ghost(c), rng.uniform(1.0, 8.0), False) if b < c["blocks"] // 2
                 else _wavy(n, _node_ghost(c), rng.uniform(0.06, 0.09)) for b, n in enumerate(sizes)]
    else:
        grids = [_one_grid(c, rng)]
    for g in grids:
        qinf, q = _flow(c, g, rng)
        out.append((g, qinf, q.to(dt).contiguous()))
    return out


def _parts(c):
    k, n = c["parts"], c["nk"]
    return [n // k + (1 if b < n % k else 0) for b in range(k)]


# --------------------------------------------------------------------------- the calls
def prepare(case, seed):
    from paper_2101_05886_gb300.solver import Batch, Block, Pipe

    c = case
    blocks = _blocks(c, seed)
    links = ()
    if c["kind"] == "linked":        # the block split along k, every part with its neighbours' nodes
        g, qinf, q = blocks[0]
        sizes = _parts(c)
        grids, links = I.split_grid(g, 2, sizes)
        blocks = [(p, qinf, s.contiguous()) for p, s in zip(grids, torch.split(q, sizes, dim=1))]
    objs = [Block(g, metric_order=c["order"], scheme=c["scheme"], precision=c["precision"],
                  characteristic=c["characteristic"], q_inf=qinf, global_lf=c["global_lf"]) for g, qinf, _ in blocks]
    states = [q for _, _, q in blocks]
    s = {"case": c, "blocks": objs, "states": states}
    s["dt"] = min(b.cfl_dt(q, 0.4) for b, q in zip(objs, states))
    if c["kind"] == "rhs":
        s["out"] = torch.empty_like(states[0])
    elif c["kind"] in ("batch", "linked"):
        s["batch"] = Batch(objs, states, links=links)
    elif c["kind"] == "pipe":
        s["states"] = [q.cpu().pin_memory() for q in states]
        s["pipe"] = Pipe(objs, s["states"], groups=4)
    return s


def run(state):
    kind, b, q = state["case"]["kind"], state["blocks"][0], state["states"][0]
    if kind == "rhs":
        return b.rhs(q, state["out"])
    if kind == "step":
        return b.rk3_step(q, state["dt"])
    if kind == "advance":
        dt = b.cfl_dt(q, 0.4)
        return b.rk3_step(q, dt), dt
    if kind == "pipe":
        state["pipe"].rk3_step(state["dt"])
        return state["states"]
    state["batch"].rk3_step(state["dt"])
    return state["states"]


def work(case):
    c = case
    if c["grid"] == "mixed":
        pts = sum(a * b * d for a, b, d in I.batched_block_sizes(c["blocks"], c["lo"], c["hi"], seed=4))
    else:
        pts = c["ni"] * c["nj"] * c["nk"]
    dims = 3 if c["nk"] != 1 else 2
    stages = 1 if c["kind"] == "rhs" else 3
    flops = PASS_FLOPS[c["scheme"]] * dims * stages * pts
    # the state in and out, the metric vectors and the cell volume
    values = 5 + 5 + dims * dims + 1
    return {"bytes": float(values * (4 if c["precision"] == F32 else 8) * pts), "flops": float(flops)}


# --------------------------------------------------------------------------- the same in 64 bits
def _weights(order):
    w = {2: [1, 1], 4: [-1, 7, 7, -1], 6: [1, -8, 37, 37, -8, 1], 8: [-3, 29, -139, 533, 533, -139, 29, -3]}[order]
    return [x / sum(w) for x in w]


class _Geometry:
    """Symmetric conservative metrics and Jacobian of a block, with its ghost layers."""

    def __init__(self, c, grid):
        self.dims, self.order, self.g = grid.dims, c["order"], _ghost(c)
        h, m = self.order // 2, self.order
        w = _weights(m)
        self.w = w
        dc = [(w[t + h - 1] if t > -h else 0.0) - (w[t + h] if t < h else 0.0) for t in range(-h, h + 1)]
        self.n = n = tuple(int(v) for v in grid.n)
        x = torch.as_tensor(np.ascontiguousarray(grid.nodes)).to(DEVICE)
        if self.dims == 2:
            x = x[:, None]
        gn, g1, g2, g3 = grid.Gn, self.g + m, self.g + h, self.g

        def win(a, have, want, d=None, t=0):
            """The box with `want` ghost layers out of one with `have`, moved by t along d."""
            for e in range(self.dims):
                o = have - want + (t if e == d else 0)
                a = a.narrow(a.dim() - 1 - e, o, n[e] + 2 * want)
            return a

        def ddx(f, have, want, d):
            f0 = win(f, have, want)
            return sum(dc[t + h] * (win(f, have, want, d, t) - f0) for t in range(-h, h + 1) if t)

        d1 = [[ddx(x[b], gn, g1, e) for e in range(self.dims)] for b in range(self.dims)]
        met = [None] * 9
        if self.dims == 2:
            y_e, x_e, y_x, x_x = (win(a, g1, g2) for a in (d1[1][1], d1[0][1], d1[1][0], d1[0][0]))
            z = torch.zeros_like(y_e)
            met = [y_e, -x_e, z, -y_x, x_x, z, z, z, z]
        else:
            for d in range(3):
                e, f = (d + 1) % 3, (d + 2) % 3
                for a in range(3):
                    b, k = (a + 1) % 3, (a + 2) % 3
                    b0, k0 = win(x[b], gn, g2), win(x[k], gn, g2)
                    s = 0.0
                    for t in range(-h, h + 1):
                        if not t:
                            continue
                        s = s + dc[t + h] * (win(d1[b][e], g1, g2, f, t) * (win(x[k], gn, g2, f, t) - k0)
                                             - (win(x[b], gn, g2, f, t) - b0) * win(d1[k][e], g1, g2, f, t)
                                             + (win(x[b], gn, g2, e, t) - b0) * win(d1[k][f], g1, g2, e, t)
                                             - win(d1[b][f], g1, g2, e, t) * (win(x[k], gn, g2, e, t) - k0))
                    met[3 * d + a] = 0.5 * s
        inv = 0.0
        for d in range(self.dims):
            for t in range(-h, h + 1):
                if not t:
                    continue
                p = sum((win(x[a], gn, g3, d, t) - win(x[a], gn, g3)) * win(met[3 * d + a], g2, g3, d, t)
                        for a in range(self.dims))
                inv = inv + dc[t + h] * p
        self.inv = inv / self.dims
        self.k = [win(a, g2, g3) for a in met]

    def line(self, a, d):
        """A ghosted array as (t2, t1, along d): ghosts kept along d only."""
        for e in range(self.dims):
            if e != d:
                a = a.narrow(2 - e, self.g, self.n[e])
        return a.movedim(2 - d, 2)

    def interior(self, a):
        for e in range(self.dims):
            a = a.narrow(2 - e, self.g, self.n[e])
        return a


def _ghosted(c, grid, geo, q, qinf, d):
    """The state with its ghost cells along d: (5, t2, t1, n_d + 2 g)."""
    g, n = geo.g, q.shape[3 - d]
    s = q.movedim(3 - d, 3)
    ends = []
    for side in (0, 1):
        bc = grid.bc[d][side]
        if bc == I.BC_PERIODIC:
            ends.append(s[..., n - g:] if side == 0 else s[..., :g])
        elif bc == I.BC_FARFIELD:
            ends.append(qinf.reshape(5, 1, 1, 1).expand(*s.shape[:3], g))
        elif bc == I.BC_EXTRAP:
            ends.append((s[..., :1] if side == 0 else s[..., -1:]).expand(*s.shape[:3], g))
        else:
            m = (s[..., :g] if side == 0 else s[..., n - g:]).flip(3)      # the mirror cells
            h = geo.order // 2
            f = g - h if side == 0 else g + n - h                          # first cell of the boundary face's formula
            k = torch.stack([sum(w * geo.line(geo.k[3 * d + a], d)[..., f + j] for j, w in enumerate(geo.w))
                             for a in range(3)])
            k = (k / k.square().sum(0).sqrt())[..., None]
            w = m.clone()
            w[1:4] -= 2 * (m[1:4] * k).sum(0) * k
            if bc == I.BC_CUT:                                             # wake cells meet across the cut
                nt = s.shape[2]
                t = torch.arange(nt, device=s.device)
                cut = ((t < grid.cut) | (t >= nt - grid.cut)).reshape(1, 1, nt, 1)
                w = torch.where(cut, m.flip(2), w)
            ends.append(w)
    return torch.cat([ends[0], s, ends[1]], dim=3)


def _flux(q, k, gamma=1.4):
    u = (q[1] * k[0] + q[2] * k[1] + q[3] * k[2]) / q[0]
    p = (gamma - 1) * (q[4] - 0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0])
    return [q[0] * u, q[1] * u + p * k[0], q[2] * u + p * k[1], q[3] * u + p * k[2], (q[4] + p) * u]


def _reconstruct(scheme, v):
    """The face value from the upwind-biased stencil v (paper's Sec. 2.2.2 and Remark 2)."""
    if scheme == LINEAR:
        return (2 * v[0] - 13 * v[1] + 47 * v[2] + 27 * v[3] - 3 * v[4]) / 60
    if scheme == WENO7:
        qs = [(-3 * v[0] + 13 * v[1] - 23 * v[2] + 25 * v[3]) / 12, (v[1] - 5 * v[2] + 13 * v[3] + 3 * v[4]) / 12,
              (-v[2] + 7 * v[3] + 7 * v[4] - v[5]) / 12, (3 * v[3] + 13 * v[4] - 5 * v[5] + v[6]) / 12]
        form = [(547, -3882, 4642, -1854, 7043, -17246, 7042, 11003, -9402, 2107),
                (267, -1642, 1602, -494, 2843, -5966, 1922, 3443, -2522, 547),
                (547, -2522, 1922, -494, 3443, -5966, 1602, 2843, -1642, 267),
                (2107, -9402, 7042, -1854, 11003, -17246, 4642, 7043, -3882, 547)]
        al = []
        for r, cw in enumerate((1, 12, 18, 4)):
            a, b, e, f = v[r:r + 4]
            m = form[r]
            beta = (a * (m[0] * a + m[1] * b + m[2] * e + m[3] * f) + b * (m[4] * b + m[5] * e + m[6] * f)
                    + e * (m[7] * e + m[8] * f) + m[9] * f * f) / 240
            al.append(cw / 35 / (beta + 1e-6) ** 2)
    else:
        qs = [v[0] / 3 - 7 * v[1] / 6 + 11 * v[2] / 6, -v[1] / 6 + 5 * v[2] / 6 + v[3] / 3, v[2] / 3 + 5 * v[3] / 6 - v[4] / 6]
        beta = [13 / 12 * (v[0] - 2 * v[1] + v[2]) ** 2 + 0.25 * (v[0] - 4 * v[1] + 3 * v[2]) ** 2,
                13 / 12 * (v[1] - 2 * v[2] + v[3]) ** 2 + 0.25 * (v[1] - v[3]) ** 2,
                13 / 12 * (v[2] - 2 * v[3] + v[4]) ** 2 + 0.25 * (3 * v[2] - 4 * v[3] + v[4]) ** 2]
        if scheme == WENO5:
            al = [cw / (b + 1e-6) ** 2 for cw, b in zip((0.1, 0.6, 0.3), beta)]
        else:
            qs.append((11 * v[3] - 7 * v[4] + 2 * v[5]) / 6)
            a, b, e, f, g = (v[t + 1] - v[t] for t in range(5))            # beta6 in the first differences
            b6 = (a * (271779 * a - 1837242 * b + 2249110 * e - 1213142 * f + 245620 * g)
                  + b * (3544296 * b - 9252940 * e + 5189840 * f - 1079386 * g)
                  + e * (6713736 * e - 7947412 * f + 1713274 * g) + f * (2534504 * f - 1150710 * g) + 139633 * g * g) / 120960
            tau = (b6 - (beta[0] + 4 * beta[1] + beta[2]) / 6).abs()
            al = [cw * (20 + tau / (b_ + 1e-40)) ** 2 for cw, b_ in zip((0.05, 0.45, 0.45, 0.05), beta + [b6])]
    total = sum(al)
    return sum(a * q for a, q in zip(al, qs)) / total


def _speeds(q, k, inv, gamma=1.4):
    p = (gamma - 1) * (q[4] - 0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0])
    u = (q[1] * k[0] + q[2] * k[1] + q[3] * k[2]) / q[0] / inv
    a = (gamma * p / q[0]).sqrt() * (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).sqrt() / inv.abs()
    return [(u - a).abs(), u.abs(), (u + a).abs()]


def _direction(c, grid, geo, q, qinf, d, gamma=1.4):
    """Face flux differences of direction d, in the state's layout."""
    g, n = geo.g, q.shape[3 - d]
    Q = _ghosted(c, grid, geo, q, qinf, d)
    K = [geo.line(geo.k[3 * d + a], d) for a in range(3)]
    V = geo.line(geo.inv, d)
    at = lambda a, m: a[..., g - 1 + m: g + n + m]        # noqa: E731  cell f + m of every face f = -1 .. n-1
    first = 1 - geo.order // 2
    face = lambda a: sum(w * at(a, first + j) for j, w in enumerate(geo.w))     # noqa: E731
    kf = [face(a) for a in K]
    vf = face(V)
    Qs = [face(Q[v] * V) / vf for v in range(5)]
    taps = range(-3, 5) if c["scheme"] == WENO7 else range(-2, 4)
    char = c["characteristic"]
    if c["global_lf"]:
        lam = [a.max() for a in _speeds(q.movedim(3 - d, 3), [a[..., g:g + n] for a in K], V[..., g:g + n])]
    else:
        lam = [torch.stack([at(s, m) for m in taps]).amax(0) for s in _speeds(Q, K, V)]
    l0, l1, l2 = lam
    lam = [l0, l1, l1, l1, l2] if char else [torch.maximum(l0, l2)] * 5
    if char:
        ql, qr = [at(Q[v], 0) for v in range(5)], [at(Q[v], 1) for v in range(5)]
        rl, rr = ql[0].sqrt(), qr[0].sqrt()
        pr = lambda s: (gamma - 1) * (s[4] - 0.5 * (s[1] ** 2 + s[2] ** 2 + s[3] ** 2) / s[0])      # noqa: E731
        u = [(rl * ql[1 + a] / ql[0] + rr * qr[1 + a] / qr[0]) / (rl + rr) for a in range(3)]
        H = (rl * (ql[4] + pr(ql)) / ql[0] + rr * (qr[4] + pr(qr)) / qr[0]) / (rl + rr)
        q2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        cs = ((gamma - 1) * (H - 0.5 * q2)).sqrt()
        kn = (kf[0] ** 2 + kf[1] ** 2 + kf[2] ** 2).sqrt()
        nn = [a / kn for a in kf]
        low, z = nn[2] ** 2 <= 0.5, torch.zeros_like(kn)
        s = torch.where(low, nn[0] ** 2 + nn[1] ** 2, nn[1] ** 2 + nn[2] ** 2).sqrt()
        t1 = [torch.where(low, -nn[1] / s, z), torch.where(low, nn[0], nn[2]) / s, torch.where(low, z, -nn[1] / s)]
        t2 = [nn[1] * t1[2] - nn[2] * t1[1], nn[2] * t1[0] - nn[0] * t1[2], nn[0] * t1[1] - nn[1] * t1[0]]
        dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]          # noqa: E731
        un, b = dot(u, nn), (gamma - 1) / cs ** 2

        def left(x):
            m = x[1:4]
            e = 0.5 * b * (0.5 * q2 * x[0] - dot(u, m) + x[4])
            w = 0.5 * (un * x[0] - dot(nn, m)) / cs
            return [e + w, x[0] - 2 * e, dot(t1, m) - dot(t1, u) * x[0], dot(t2, m) - dot(t2, u) * x[0], e - w]

        def right(h):
            s0, s1 = h[0] + h[1] + h[4], h[4] - h[0]
            out = [s0] + [u[a] * s0 + cs * nn[a] * s1 + t1[a] * h[2] + t2[a] * h[3] for a in range(3)]
            return out + [H * (h[0] + h[4]) + cs * un * s1 + 0.5 * q2 * h[1] + dot(t1, u) * h[2] + dot(t2, u) * h[3]]
    else:
        left = right = lambda x: list(x)                  # noqa: E731
    plus, minus = [[] for _ in range(5)], [[] for _ in range(5)]
    for m in taps:
        qm, km = [at(Q[v], m) for v in range(5)], [at(a, m) for a in K]
        F = [a - b_ for a, b_ in zip(_flux(qm, km), _flux(Qs, km))]
        D = [(a - b_) * at(V, m) for a, b_ in zip(qm, Qs)]
        for v, (a, b_) in enumerate(zip(left(F), left(D))):
            plus[v].append(0.5 * (a + lam[v] * b_))
            minus[v].append(0.5 * (a - lam[v] * b_))
        del qm, km, F, D
    h = []
    for v in range(5):
        h.append(_reconstruct(c["scheme"], plus[v]) + _reconstruct(c["scheme"], minus[v][::-1]))
        plus[v] = minus[v] = None
    flux = torch.stack([a + b_ for a, b_ in zip(right(h), _flux(Qs, kf))])
    return (flux[..., 1:] - flux[..., :-1]).movedim(3, 3 - d)


def _residual(c, grid, geo, q, qinf):
    r = _direction(c, grid, geo, q, qinf, 0)
    for d in range(1, geo.dims):
        r += _direction(c, grid, geo, q, qinf, d)
    return -r / geo.interior(geo.inv)


def _bound(geo, q, cfl):
    s, inv = 0.0, geo.interior(geo.inv)
    for d in range(geo.dims):
        a, _, b = _speeds(q, [geo.interior(geo.k[3 * d + e]) for e in range(3)], inv)
        s = s + torch.maximum(a, b)
    return cfl / s.max().item()


def exact(case, seed):
    c = case
    blocks = _blocks(c, seed)
    # q_inf is used in the state's precision
    rounded = lambda x: torch.as_tensor(x).to(torch.float32 if c["precision"] == F32 else torch.float64).double().to(DEVICE)  # noqa: E731
    dts, out = [], []
    for g, _, q in blocks:
        if c["kind"] != "rhs":
            dts.append(_bound(_Geometry(c, g), q.double(), 0.4))
    for g, qinf, q in blocks:
        geo, q0, qi = _Geometry(c, g), q.double(), rounded(qinf)
        if c["kind"] == "rhs":
            return _residual(c, g, geo, q0, qi)
        dt = min(dts)
        q1 = q0 + dt * _residual(c, g, geo, q0, qi)
        q2 = 0.75 * q0 + 0.25 * (q1 + dt * _residual(c, g, geo, q1, qi))
        del q1
        out.append(q0 / 3 + 2 / 3 * (q2 + dt * _residual(c, g, geo, q2, qi)))
        del geo, q2
    if c["kind"] == "step":
        return out[0]
    if c["kind"] == "advance":
        return out[0], dts[0]
    if c["kind"] == "linked":
        return [s.contiguous() for s in torch.split(out[0], _parts(c), dim=1)]
    return out
