"""Performance cases of the GB300 NUMA hot path: what a user of the framework
has it do, through its public entry points (paper_1511_01561_gb300.numa).

  rhs    one evaluation of R = dq/dt at a device state (Solver.rhs): what a
         caller with a time integrator of its own asks for;
  run    a forecast segment: hand the state over, advance it some steps, fetch
         the new state (Solver.set_state, Solver.run, Solver.get_state);
  host   states that arrive in pinned host memory, advanced one step each and
         returned to the host, pipelined (HostStepper);
  serve  an ensemble of forecast requests of mixed size, order and precision
         through the continuous-batching scheduler (Scheduler).

Meshes, constants and time steps follow paper_1511_01561_gb300.inputs: the
rising bubble in a box, the thin box and the cubed-sphere shell.  exact()
restates the method in plain FP64 torch.
"""
import math
import random

import numpy as np
import torch

from paper_1511_01561_gb300 import inputs, numa

DEV = "cuda:0"
F64 = torch.float64


# ---- the cases ----------------------------------------------------------------

def _box(name, call, N, ne, precision, steps=1, **over):
    c = dict(name=name, call=call, mesh="box", N=N, nex=ne[0], ney=ne[1], nez=ne[2], Lx=1000.0, Ly=1000.0, Lz=1000.0,
             periodic=False, warp=0.0, npanel=0, nlayer=0, precision=precision, scheme="ssp3", filter=0, storage="cg",
             steps=steps)
    c.update(over)
    return c


def _shell(name, call, N, npanel, nlayer, precision, steps=1, **over):
    return _box(name, call, N, (0, 0, 0), precision, steps, mesh="shell", npanel=npanel, nlayer=nlayer, **over)


def listed():
    return [
        # the smallest workload (inputs.WORKLOADS "bubble_4x4x4_N4"), one right-hand side: launches and latency
        _box("rhs_box_4_N4_fp64", "rhs", 4, (4, 4, 4), "fp64"),
        # the smallest member of the serving stream (8 elements an edge) on its own: short kernels back to back
        _box("run_box_8_N4_fp64", "run", 4, (8, 8, 8), "fp64", 20),
        # the headline workload, the rising bubble at 32^3 elements, in each precision it is offered in
        _box("run_bubble_32_N4_fp64", "run", 4, (32, 32, 32), "fp64", 10),
        _box("run_bubble_32_N4_fp32_mixed", "run", 4, (32, 32, 32), "fp32_mixed", 20),
        _box("run_bubble_32_N4_fp64_pairs", "run", 4, (32, 32, 32), "fp64_pairs", 10),
        # a higher order of the serving stream on an uneven element count per axis
        _box("run_box_19x23x17_N6_fp64", "run", 6, (19, 23, 17), "fp64", 6),
        # curved elements of low order, periodic in x and y, five-stage low-storage scheme with the filter every
        # second step: terrain-like meshes with the paper's stage count and stabilisation
        _box("run_warped_21x17x13_N3_ls54_filter", "run", 3, (21, 17, 13), "fp64", 8, periodic=True, warp=0.03,
             scheme="ls54", filter=2),
        # the deep-atmosphere shell at its full size (baroclinic-wave stand-in): the largest FP64 work
        _shell("run_shell_30x8_N4_fp64", "run", 4, 30, 8, "fp64", 4),
        _shell("run_shell_30x8_N4_fp32_mixed", "run", 4, 30, 8, "fp32_mixed", 10),
        # the thin box with implicit vertical columns ("thin_64x64x8_N4"): the long-time-step production scheme
        _box("run_thin_64x64x8_N4_imex", "run", 4, (64, 64, 8), "fp64", 10, Lx=1024e3, Ly=1024e3, Lz=8e3,
             scheme="imex"),
        # states streamed from and to host memory, as an ensemble driver or a data-assimilation loop does
        _box("host_bubble_32_N4_fp64", "host", 4, (32, 32, 32), "fp64", 1),
        # six requests of the serving stream's lower half, mixed orders and precisions, until all results are in
        dict(name="serve_6_mixed", call="serve", members=6, edge_lo=8, edge_hi=14, steps_lo=100, steps_hi=150,
             mix=1511),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """Another case of the same ranges: element nodes from 8 thousand to 2.5 million, every order, precision,
    mesh kind and integrator."""
    N = rng.choice((2, 3, 3, 4, 4, 4, 5, 6, 6, 7, 8))
    nodes = math.exp(rng.uniform(math.log(8e3), math.log(2.5e6)))
    elems = nodes / (N + 1) ** 3
    precision = rng.choice(("fp64", "fp64", "fp64", "fp32_mixed", "fp32_mixed", "fp64_pairs"))
    call = rng.choice(("run", "run", "run", "rhs"))
    steps = rng.randint(3, 10) if call == "run" else 1
    kind = rng.random()
    if kind < 0.3:
        npanel = max(2, int(round((elems / 6 / 4) ** (1.0 / 3.0) * rng.uniform(0.9, 1.8))))
        nlayer = max(2, min(12, int(round(elems / (6 * npanel * npanel)))))
        c = _shell("", call, N, npanel, nlayer, precision, steps)
    else:
        edge = elems ** (1.0 / 3.0)
        ne = [max(2, int(round(edge * rng.uniform(0.7, 1.4)))) for _ in range(3)]
        c = _box("", call, N, ne, precision, steps, periodic=rng.random() < 0.25,
                 warp=round(rng.uniform(0.01, 0.04), 4) if kind > 0.8 else 0.0,
                 storage="dg" if rng.random() < 0.1 else "cg")
    if call == "run":
        c["scheme"] = rng.choice(("ssp3", "ssp3", "ssp3", "ls54"))
        if c["mesh"] == "box" and c["warp"] == 0.0 and c["storage"] == "cg" and precision == "fp64" and rng.random() < 0.3:
            ne_h = max(2, c["nex"])
            c.update(scheme="imex", nex=ne_h, Lx=16e3 * ne_h, Ly=16e3 * c["ney"], Lz=1e3 * c["nez"])
            if c["nez"] > 12:
                c.update(nez=12, Lz=12e3)
        elif rng.random() < 0.25:
            c["filter"] = rng.randint(1, 3)
    del c["name"]
    return c


# ---- configurations, inputs ---------------------------------------------------

FILTER_P, FILTER_MU = 12.0, 1.0  # every application: first damped mode N - 1, as the benchmark's


def _cfg(c):
    if c["mesh"] == "shell":
        return inputs.shell(c["npanel"], c["nlayer"], c["N"], storage=c["storage"])
    p = int(c["periodic"])
    return inputs.box((c["nex"], c["ney"], c["nez"]), c["N"], L=(c["Lx"], c["Ly"], c["Lz"]), periodic=(p, p, 0),
                      warp=c["warp"], storage=c["storage"])


def _dt(c):
    """Acoustic Courant number 0.3 on the closest node pair (the column scheme: on the closest horizontal one)."""
    end = 0.5 * (1.0 - math.cos(math.pi / c["N"]))
    if c["mesh"] == "shell":
        h = min(0.5 * math.pi * inputs.EARTH_RADIUS / c["npanel"] * 0.7, 30e3 / c["nlayer"])
    else:
        h = min(c["Lx"] / c["nex"], c["Ly"] / c["ney"])
        if c["scheme"] == "imex":
            return 0.2 * h * end / 350.0
        h = min(h, c["Lz"] / c["nez"]) * (1.0 - 4.0 * c["warp"])
    return 0.3 * h * end / 350.0


def _lobatto(N):
    """Lobatto points, weights and the derivative matrix of order N."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    x = 0.5 * (x - x[::-1])
    for _ in range(3):  # Newton on (1 - x^2) P_N'
        x[1:-1] -= (P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1]))
    x = 0.5 * (x - x[::-1])
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    lam = np.array([1.0 / np.prod([x[j] - x[k] for k in range(N + 1) if k != j]) for j in range(N + 1)])
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = lam[j] / lam[i] / (x[i] - x[j])
        D[i, i] = -D[i].sum()
    return x, w, D


PANELS = ([[0, 1, 0], [0, 0, 1], [1, 0, 0]], [[-1, 0, 0], [0, 0, 1], [0, 1, 0]], [[0, -1, 0], [0, 0, 1], [-1, 0, 0]],
          [[1, 0, 0], [0, 0, 1], [0, -1, 0]], [[0, 1, 0], [-1, 0, 0], [0, 0, 1]], [[0, 1, 0], [1, 0, 0], [0, 0, -1]])


class _Mesh:
    """Element-node coordinates X [3][Ne, P, P, P] (k, j, i), the element-to-global map, global coordinates, wall
    normals and reference state of one configuration, in FP64 torch."""

    def __init__(self, cfg):
        self.cfg = cfg
        N = self.N = cfg["N"]
        P = self.P = N + 1
        xi, w, D = _lobatto(N)
        self.xi, self.w = xi, w
        self.D = torch.tensor(D, dtype=F64, device=DEV)
        t01 = 0.5 * (1.0 + xi)
        if cfg["kind"] == "box":
            ne, L, per = cfg["ne"], cfg["L"], cfg["periodic"]
            ax, ix, n = [], [], []
            for d in range(3):
                a = (np.arange(ne[d])[:, None] + t01[None, :]) / ne[d]
                n.append(ne[d] * N + (0 if per[d] else 1))
                ax.append(torch.tensor(a, dtype=F64, device=DEV))
                ix.append(torch.tensor((np.arange(ne[d])[:, None] * N + np.arange(P)) % n[d], device=DEV))
            shape = (ne[2], ne[1], ne[0], P, P, P)
            u = ax[0].view(1, 1, ne[0], 1, 1, P).expand(shape).reshape(-1, P, P, P)
            v = ax[1].view(1, ne[1], 1, 1, P, 1).expand(shape).reshape(-1, P, P, P)
            t = ax[2].view(ne[2], 1, 1, P, 1, 1).expand(shape).reshape(-1, P, P, P)
            pi, wp = math.pi, cfg["warp"]
            if wp:
                su, sv, st = torch.sin(pi * u), torch.sin(pi * v), torch.sin(pi * t)
                self.X = [L[0] * (u + wp * su * sv * st), L[1] * (v + wp * torch.sin(2 * pi * u) * sv * st),
                          L[2] * (t + wp * su * torch.sin(2 * pi * v) * st)]
            else:
                self.X = [L[0] * u, L[1] * v, L[2] * t]
            g = (ix[0].view(1, 1, ne[0], 1, 1, P) + n[0] * (ix[1].view(1, ne[1], 1, 1, P, 1)
                                                            + n[1] * ix[2].view(ne[2], 1, 1, P, 1, 1)))
            self.l2g = g.expand(shape).reshape(-1)
            self.Ng = n[0] * n[1] * n[2]
            self.ncol, self.nz = n[0] * n[1], n[2]
            self.fixed = []  # per direction: the global nodes on walls normal to it
            lat = torch.arange(self.Ng, device=DEV)
            lat = (lat % n[0], (lat // n[0]) % n[1], lat // (n[0] * n[1]))
            for d in range(3):
                self.fixed.append(None if per[d] else (lat[d] == 0) | (lat[d] == n[d] - 1))
            self.height = None
        else:
            npn, nl = cfg["npanel"], cfg["nlayer"]
            K = npn * N
            al = (-0.25 * math.pi + (np.arange(npn)[:, None] + t01) * (0.5 * math.pi / npn))  # [ia][i]
            dR = (cfg["r_outer"] - cfg["r_inner"]) / nl
            hk = (np.arange(nl)[:, None] + t01) * dR  # [il][k]
            lat = 2 * (np.arange(npn)[:, None] * N + np.arange(P)) - K
            dirs, keys = [], []
            for fr in np.array(PANELS):
                ta, tb = np.tan(al)[None, :, None, :], np.tan(al)[:, None, :, None]  # [ib][ia][j][i]
                vec = fr[2][:, None, None, None, None] + fr[0][:, None, None, None, None] * ta \
                    + fr[1][:, None, None, None, None] * tb
                dirs.append(vec / np.sqrt((vec ** 2).sum(0)))
                la, lb = lat[None, :, None, :], lat[:, None, :, None]
                pt = [K * fr[2][d] + la * fr[0][d] + lb * fr[1][d] + K for d in range(3)]
                keys.append((pt[0] * (2 * K + 1) + pt[1]) * (2 * K + 1) + pt[2])
            dirs = np.stack(dirs, 1).reshape(3, -1, P, P)  # [3][column of elements][j][i]
            keys = np.stack(keys).reshape(-1)
            _, at, inv = np.unique(keys, return_index=True, return_inverse=True)
            rank = np.empty(len(at), dtype=np.int64)
            rank[np.argsort(at)] = np.arange(len(at))  # columns by first appearance
            col = torch.tensor(rank[inv.reshape(-1)].reshape(-1, 1, 1, P, P), device=DEV)
            self.ncol, self.nz = len(at), nl * N + 1
            self.Ng = self.ncol * self.nz
            lev = torch.tensor(np.arange(nl)[:, None] * N + np.arange(P), device=DEV).view(1, nl, P, 1, 1)
            self.l2g = (col + self.ncol * lev).reshape(-1)
            h = torch.tensor(hk, dtype=F64, device=DEV).view(1, nl, P, 1, 1)
            r = cfg["r_inner"] + h
            vec = torch.tensor(dirs, dtype=F64, device=DEV)
            self.X = [(r * vec[d].view(-1, 1, 1, P, P)).reshape(-1, P, P, P) for d in range(3)]
            self.height = torch.full((self.Ng,), math.inf, dtype=F64, device=DEV).scatter_reduce(
                0, self.l2g, h.expand(vec.shape[1], nl, P, P, P).reshape(-1), "amin")
            self.fixed = None
        # a node's coordinates are the least of its element nodes' (they differ by rounding, or by the period)
        self.x = torch.full((3, self.Ng), math.inf, dtype=F64, device=DEV)
        for d in range(3):
            self.x[d].scatter_reduce_(0, self.l2g, self.X[d].reshape(-1), "amin")
        self._reference()

    def _reference(self):
        c = self.cfg
        if self.height is None:
            phi = c["g"] * self.x[2]
            self.up = None
        else:
            a, r = c["r_inner"], self.x.norm(dim=0)
            phi = c["g"] * a * self.height / (a + self.height)
            self.up = self.x / r
            self.gr = c["g"] * (a / r) ** 2
        if c["ref"] == "isentropic":
            ex = 1.0 - phi / (c["cp"] * c["theta0"])
            self.p0 = c["P00"] * ex ** (c["cp"] / c["Rd"])
            self.Th0 = self.p0 / (c["Rd"] * ex)
            self.rho0 = self.Th0 / c["theta0"]
        else:
            self.p0 = c["P00"] * torch.exp(-phi / (c["Rd"] * c["T0"]))
            self.rho0 = self.p0 / (c["Rd"] * c["T0"])
            self.Th0 = (c["P00"] / c["Rd"]) * (self.p0 / c["P00"]) ** (c["cv"] / c["cp"])


def _initial(m, seed):
    """A developing flow: the box's warm bubble (0.3 to 1 K, no pressure perturbation of its own) or the shell's zonal
    jet, under smooth random motion of a few m/s (along the walls at the walls) with its density and rho*theta."""
    c = m.cfg
    rng = np.random.default_rng(seed)
    q = torch.zeros((5, m.Ng), dtype=F64, device=DEV)
    if m.up is None:
        L = c["L"]
        s = [m.x[d] / L[d] for d in range(3)]
        rc = 0.25 * min(L) if max(L) < 10 * min(L) else 0.03 * max(L)
        dist2 = sum((m.x[d] - L[d] * (rng.uniform(0.35, 0.65) if d < 2 else rng.uniform(0.3, 0.5))) ** 2
                    for d in range(3))
        r = dist2.sqrt() / rc
        dth = torch.where(r <= 1.0, 0.5 * rng.uniform(0.3, 1.0) * (1.0 + torch.cos(math.pi * r)), torch.zeros_like(r))
        q[0] = m.Th0 / (m.Th0 / m.rho0 + dth) - m.rho0

        def mode(d):  # zero at the walls normal to d (d < 0: no condition)
            f = rng.uniform(0.5, 1.0)
            for e in range(3):
                if c["periodic"][e]:
                    f = f * torch.sin(2 * math.pi * (rng.integers(1, 3) * s[e] + rng.uniform()))
                elif e == d:
                    f = f * torch.sin(math.pi * rng.integers(1, 3) * s[e])
                else:
                    f = f * torch.cos(math.pi * rng.integers(0, 3) * s[e])
            return f
        flat = min(L) / max(L)
        for d in range(3):
            q[1 + d] = 4.0 * (flat if d == 2 else 1.0) * m.rho0 * mode(d)
        q[0] += 2e-4 * m.rho0 * mode(-1)
        q[4] = 1e-4 * m.Th0 * mode(-1)
    else:
        lat, lon = torch.asin(m.up[2]), torch.atan2(m.up[1], m.up[0])
        lc, pc = rng.uniform(0.0, 2 * math.pi), rng.uniform(0.5, 1.0)
        cd = math.sin(pc) * torch.sin(lat) + math.cos(pc) * torch.cos(lat) * torch.cos(lon - lc)
        u = rng.uniform(30.0, 40.0) * torch.sin(2 * lat) ** 2
        u = u + torch.exp(-(torch.acos(cd.clamp(-1, 1)) / 0.1) ** 2)
        q[1], q[2] = -m.rho0 * u * torch.sin(lon), m.rho0 * u * torch.cos(lon)
        k = rng.integers(1, 4, 3)
        wave = torch.sin(k[0] * m.up[0] + rng.uniform(0, 6)) * torch.cos(k[1] * m.up[1] + k[2] * m.up[2])
        q[0], q[4] = 2e-4 * m.rho0 * wave, 1e-4 * m.Th0 * wave
    return q


def _members(c, seed):
    """The requests of a serving case: sizes, orders, precisions and step counts from the case, amplitudes and centres
    from the seed (as in inputs.serving_stream)."""
    shape, val = random.Random(c["mix"]), random.Random(seed)
    out = []
    for k in range(c["members"]):
        ne, N = shape.randint(c["edge_lo"], c["edge_hi"]), (3, 4, 6)[k % 3]
        steps = shape.randint(c["steps_lo"], c["steps_hi"])
        dx = (1000.0 / ne) * 0.5 * (1.0 - math.cos(math.pi / N))
        params = (val.uniform(0.1, 2.0), 250.0) + tuple(val.uniform(250.0, 750.0) for _ in range(3))
        out.append(dict(cfg=inputs.box(ne, N), params=params, dt=min(0.01, 0.5 * dx / 350.0), nsteps=steps,
                        precision="fp64" if k % 2 == 0 else "fp32_mixed"))
    return out


# ---- prepare, run -------------------------------------------------------------

def prepare(case, seed):
    if case["call"] == "serve":
        return dict(case=case, sched=numa.Scheduler(1 << 30, DEV), requests=_members(case, seed))
    cfg = _cfg(case)
    m = _Mesh(cfg)
    s = numa.Solver(cfg, case["precision"], DEV)
    s.set_time_scheme(case["scheme"])
    if case["filter"]:
        s.set_filter(case["filter"], max(1, case["N"] - 1), FILTER_P, FILTER_MU)
    st = dict(case=case, solver=s, dt=_dt(case))
    if case["call"] == "host":
        st["q"] = [_initial(m, seed * 16 + k).cpu().pin_memory() for k in range(3)]
        st["out"] = [torch.empty((5, m.Ng), dtype=F64).pin_memory() for _ in range(3)]
        st["stepper"] = numa.HostStepper(s)
        return st
    q = _initial(m, seed)
    if case["storage"] == "dg":
        q = q[:, m.l2g].contiguous()
    st.update(q=q, out=torch.empty_like(q))
    st["rows"] = list(st["out"].unbind(0))  # the five variables of the result
    return st


def run(st):
    c = st["case"]
    if c["call"] == "serve":
        s = st["sched"]
        ids = [s.submit(r["cfg"], "bubble", r["params"], r["dt"], r["nsteps"], r["precision"]) for r in st["requests"]]
        while True:
            active, waiting = s.step()
            if not active and not waiting and all(s.poll(i)[0] in ("done", "failed") for i in ids):
                return [s.result(i) for i in ids]
    s = st["solver"]
    if c["call"] == "rhs":
        s.rhs(st["q"], st["out"])
        return st["rows"]
    if c["call"] == "host":
        for q, out in zip(st["q"], st["out"]):
            st["stepper"].submit(q, out, st["dt"], c["steps"])
        st["stepper"].synchronize()
        return st["out"]
    s.set_state(st["q"])
    s.run(st["dt"], c["steps"])
    s.get_state(st["out"])
    return st["rows"]


# ---- work ---------------------------------------------------------------------

def _counts(cfg):
    P, N = cfg["N"] + 1, cfg["N"]
    if cfg["kind"] == "box":
        ne, per = cfg["ne"], cfg["periodic"]
        Ng = math.prod(ne[d] * N + (0 if per[d] else 1) for d in range(3))
        return math.prod(ne), math.prod(ne) * P ** 3, Ng
    K, nl = cfg["npanel"] * N, cfg["nlayer"]
    Ne = 6 * cfg["npanel"] ** 2 * nl
    return Ne, Ne * P ** 3, (6 * K * K + 2) * (nl * N + 1)


def _stage(cfg, precision):
    """Bytes and flops of one right-hand side: the state in, its tendency or successor out, the reference state and,
    on curved elements, the metric terms; 15 contractions per node on box elements, 36 and the chain rule on curved."""
    Ne, Nl, Ng = _counts(cfg)
    N = cfg["N"]
    w = 4 if precision == "fp32_mixed" else 8
    curved = cfg["kind"] == "shell" or cfg["warp"] != 0.0
    nodes = Nl if cfg.get("storage", "cg") == "dg" else Ng
    by = nodes * (40 + 40 + 24 + (24 if cfg["kind"] == "shell" else 0)) + (Nl * 10 * w if curved else Ne * 3 * w)
    fl = Nl * ((36 if curved else 15) * 2 * (N + 1) + (90 if curved else 0)) + nodes * 60
    return by, fl


def work(case):
    if case["call"] == "serve":
        by = fl = 0
        for r in _members(case, 0):
            b, f = _stage(r["cfg"], r["precision"])
            by, fl = by + 3 * r["nsteps"] * b, fl + 3 * r["nsteps"] * f
        return {"bytes": by, "flops": fl}
    by, fl = _stage(_cfg(case), case["precision"])
    stages = {"ssp3": 3, "ls54": 5, "imex": 1}[case["scheme"]] * case["steps"] if case["call"] != "rhs" else 1
    k = 3 if case["call"] == "host" else 1
    return {"bytes": k * stages * by, "flops": k * stages * fl}


# ---- exact: the method in plain FP64 torch -------------------------------------

class _Exact(_Mesh):
    def __init__(self, cfg):
        super().__init__(cfg)
        A = [[self._d(x, d) for d in range(3)] for x in self.X]  # dx_c / dxi_d
        cof = lambda a, b, c, d: a * d - b * c  # noqa: E731
        C = [[cof(A[(c + 1) % 3][(d + 1) % 3], A[(c + 1) % 3][(d + 2) % 3], A[(c + 2) % 3][(d + 1) % 3],
                  A[(c + 2) % 3][(d + 2) % 3]) for d in range(3)] for c in range(3)]
        J = sum(A[0][d] * C[0][d] for d in range(3))
        self.B = [[C[c][d] / J for c in range(3)] for d in range(3)]  # dxi_d / dx_c
        w = torch.tensor(self.w, dtype=F64, device=DEV)
        self.Jw = J * (w[:, None, None] * w[None, :, None] * w[None, None, :])
        self.M = self._dss(self.Jw)

    def _dss(self, x):
        return torch.zeros(self.Ng, dtype=F64, device=DEV).index_add_(0, self.l2g, x.reshape(-1))

    def _d(self, x, d):
        """Derivative along direction d of x [Ne, P, P, P], taken relative to the first node of each line."""
        x = x - x.narrow(3 - d, 0, 1)
        return self._apply(self.D, x, d)

    def _apply(self, Mx, x, d):
        return torch.einsum(("im,ekjm->ekji", "jm,ekmi->ekji", "km,emji->ekji")[d], Mx, x)

    def rhs(self, q):
        c, P = self.cfg, self.P
        gam = c["cp"] / c["cv"]
        rho, Th = self.rho0 + q[0], self.Th0 + q[4]
        p = self.p0 * torch.expm1(gam * torch.log1p(q[4] / self.Th0))
        u = q[1:4] / rho
        at = lambda f: f[self.l2g].view(-1, P, P, P)  # noqa: E731

        def div(fl):
            out = 0.0
            for cc in range(3):
                f = at(fl[cc])
                for d in range(3):
                    out = out + self.B[d][cc] * self._d(f, d)
            return -self._dss(self.Jw * out) / self.M
        R = torch.empty_like(q)
        R[0] = div(q[1:4])
        for v in range(3):
            R[1 + v] = div([q[1 + v] * u[cc] + (p if cc == v else 0.0) for cc in range(3)])
        R[4] = div([Th * u[cc] for cc in range(3)])
        if self.up is None:
            R[3] -= c["g"] * q[0]
            for d in range(3):
                if self.fixed[d] is not None:
                    R[1 + d][self.fixed[d]] = 0.0
        else:
            R[1:4] -= q[0] * self.gr * self.up
            R[1] += 2 * c["Omega"] * q[2]
            R[2] -= 2 * c["Omega"] * q[1]
            e = torch.cat([torch.arange(self.ncol, device=DEV), torch.arange(self.Ng - self.ncol, self.Ng, device=DEV)])
            R[1:4, e] -= (R[1:4, e] * self.up[:, e]).sum(0) * self.up[:, e]
        return R

    def filtered(self, q, s):
        N, P = self.N, self.P
        V = np.polynomial.legendre.legvander(self.xi, N)
        sig = np.ones(P)
        for k in range(s, P):
            th = 1.0 if s >= N else (k - s) / (N - s)
            o = th - 0.5
            x = 0.0 if th >= 1 else 1.0 if th <= 0 else 0.5 if o == 0 else 0.5 * math.erfc(
                2 * math.sqrt(FILTER_P) * math.sqrt(-math.log(1 - 4 * o * o) / (4 * o * o)) * o)
            sig[k] = 1 - FILTER_MU * (1 - x)
        F = torch.tensor(V @ np.diag(sig) @ np.linalg.inv(V), dtype=F64, device=DEV)
        out = torch.empty_like(q)
        for v in range(5):
            x = q[v][self.l2g].view(-1, P, P, P)
            for d in range(3):
                x = self._apply(F, x, d)
            out[v] = self._dss(self.Jw * x) / self.M
        if self.up is None:
            for d in range(3):
                if self.fixed[d] is not None:
                    out[1 + d][self.fixed[d]] = q[1 + d][self.fixed[d]]
        else:
            e = torch.cat([torch.arange(self.ncol, device=DEV), torch.arange(self.Ng - self.ncol, self.Ng, device=DEV)])
            ch = out[1:4, e] - q[1:4, e]
            out[1:4, e] -= (ch * self.up[:, e]).sum(0) * self.up[:, e]
        return out

    def imex(self, q, dt, steps, nu=0.05):
        """Leapfrog with the implicit vertical operator L (rho', W, Theta' along the z-columns of the box)."""
        c, nz, N = self.cfg, self.nz, self.N
        h = c["L"][2] / c["ne"][2]
        G, mass, D = np.zeros((nz, nz)), np.zeros(nz), self.D.cpu().numpy()
        for e in range(c["ne"][2]):
            at = slice(e * N, e * N + N + 1)
            G[at, at] += self.w[:, None] * D
            mass[at] += 0.5 * h * self.w
        G /= mass[:, None]
        lev = slice(0, self.Ng, self.ncol)
        p0, Th0, rho0 = (t[lev].cpu().numpy() for t in (self.p0, self.Th0, self.rho0))
        c2, th0 = c["cp"] / c["cv"] * p0 / Th0, Th0 / rho0
        Lm = np.zeros((3 * nz, 3 * nz))
        Lm[:nz, nz:2 * nz] = -G
        Lm[nz:2 * nz, :nz] = -c["g"] * np.eye(nz)
        Lm[nz:2 * nz, 2 * nz:] = -G * c2[None, :]
        Lm[[nz, 2 * nz - 1]] = 0.0
        Lm[2 * nz:, nz:2 * nz] = -G * th0[None, :]
        L = torch.tensor(Lm, dtype=F64, device=DEV)
        inv = [torch.tensor(np.linalg.inv(np.eye(3 * nz) - t * Lm), dtype=F64, device=DEV) for t in (dt, 0.5 * dt)]
        rows = [0, 3, 4]

        def solve(f, tau, qst, sv):
            b = qst[rows].reshape(3 * nz, self.ncol) - tau * (L @ sv[rows].reshape(3 * nz, self.ncol))
            x = qst.clone()
            x[rows] = (inv[f] @ b).reshape(3, -1)
            return x
        new = solve(1, 0.5 * dt, q + dt * self.rhs(q), q)
        prev, q = q, new
        for _ in range(steps - 1):
            new = solve(0, dt, prev + 2 * dt * self.rhs(q), 2 * q - prev)
            prev, q = q + nu * (prev - 2 * q + new), new
        return q

    def advance(self, q, dt, steps, scheme="ssp3", every=0):
        if scheme == "imex" and not every:
            return self.imex(q, dt, steps)
        A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
             -1275806237668 / 842570457699)
        B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
             3134564353537 / 4481467310338, 2277821191437 / 14882151754819)
        for k in range(steps):
            if scheme == "ls54":
                dq = torch.zeros_like(q)
                for a, b in zip(A, B):
                    dq = a * dq + dt * self.rhs(q)
                    q = q + b * dq
            else:
                q1 = q + dt * self.rhs(q)
                q2 = 0.75 * q + 0.25 * (q1 + dt * self.rhs(q1))
                q = q / 3.0 + (2.0 / 3.0) * (q2 + dt * self.rhs(q2))
            if every and (k + 1) % every == 0:
                q = self.filtered(q, max(1, self.N - 1))
        return q

    def bubble(self, params):
        A, rc, *ctr = params
        r = sum((self.x[d] - ctr[d]) ** 2 for d in range(3)).sqrt()
        dth = torch.where(r <= rc, 0.5 * A * (1.0 + torch.cos(math.pi * r / rc)), torch.zeros_like(r))
        q = torch.zeros((5, self.Ng), dtype=F64, device=DEV)
        q[0] = self.Th0 / (self.Th0 / self.rho0 + dth) - self.rho0
        return q


def exact(case, seed):
    if case["call"] == "serve":
        out = []
        for r in _members(case, seed):
            m = _Exact(r["cfg"])
            out.append(m.advance(m.bubble(r["params"]), r["dt"], r["nsteps"]).cpu().numpy())
        return out
    m = _Exact(_cfg(case))
    if case["call"] == "host":
        return [m.advance(_initial(m, seed * 16 + k), _dt(case), case["steps"]).cpu() for k in range(3)]
    q = _initial(m, seed)
    q = m.rhs(q) if case["call"] == "rhs" else m.advance(q, _dt(case), case["steps"], case["scheme"], case["filter"])
    if case["storage"] == "dg":
        q = q[:, m.l2g]
    return list(q.unbind(0))
