"""Measured cases: what a user of the operator library has it compute, over the range it is used in.

Workloads are those of the package's own configurations (Taylor--Green vortex boxes, the stretched
turbulent channel, the sine-deformed periodic box, the discrete adjoint of the vortex), through the
public entry points of `paper_1806_03095_gb300.api.DGCNS`, in FP64 and in the mixed form.

`exact` evaluates the same weak form in plain torch FP64: dense 1D matrices, one face at a time,
the adjoint by torch's reverse mode.
"""
import math

import numpy as np
import torch

from paper_1806_03095_gb300 import api

TWO_PI = 2.0 * math.pi
GAMMA, PR, GAS_R, RHO0 = 1.4, 0.71, 287.0, 1.0
# the 5-stage fourth-order 2N scheme of Carpenter & Kennedy (1994)
RK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
RK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0, 1720146321549.0 / 2090206949498.0,
        3134564353537.0 / 4481467310338.0, 2277821191437.0 / 14882151754819.0)


def _case(name, call, mesh, cells, k, precision, geometry="affine", steps=1):
    return {"name": name, "call": call, "mesh": mesh, "nx": cells[0], "ny": cells[1], "nz": cells[2], "k": k,
            "precision": precision, "geometry": geometry, "steps": steps}


def listed():
    return [
        # the smallest run: 10 time steps of a 8^3 vortex, 50 operator evaluations of 164 k DoFs, launch-bound
        _case("tgv8_k3_fp64_10steps", "steps", "tgv", (8, 8, 8), 3, "fp64", steps=10),
        # one evaluation of the same box in the mixed form: latency of a single call
        _case("tgv8_k3_mixed_apply", "apply", "tgv", (8, 8, 8), 3, "mixed"),
        # the production vortex: a time step of 64^3 cells (84 M DoFs)
        _case("tgv64_k3_fp64_step", "steps", "tgv", (64, 64, 64), 3, "fp64"),
        # the same vortex in the mixed form, one Runge--Kutta stage: what a user's own time loop calls
        _case("tgv64_k3_mixed_stage", "stage", "tgv", (64, 64, 64), 3, "mixed"),
        # the operator alone at k = 4 on a box of odd extents, mixed form
        _case("tgv_odd_k4_mixed_apply", "apply", "tgv", (37, 29, 41), 4, "mixed"),
        # high order: the 40^3 vortex at k = 5 (69 M DoFs) in both precisions
        _case("tgv40_k5_fp64_apply", "apply", "tgv", (40, 40, 40), 5, "fp64"),
        _case("tgv40_k5_mixed_stage", "stage", "tgv", (40, 40, 40), 5, "mixed"),
        # the channel: walls, body force, Jacobians stored per quadrature point, mixed form
        _case("channel32_k3_mixed_stage", "stage", "channel", (32, 32, 32), 3, "mixed", "stored"),
        # a curved mesh of odd, ragged extents at k = 2, FP64
        _case("sine_odd_k2_fp64_apply", "apply", "sine", (29, 23, 31), 2, "fp64", "stored"),
        # the backward direction: vector-Jacobian product of the 24^3 vortex at k = 4, both precisions
        _case("adjoint24_k4_fp64", "adjoint", "tgv", (24, 24, 24), 4, "fp64"),
        _case("adjoint24_k4_mixed", "adjoint", "tgv", (24, 24, 24), 4, "mixed"),
        # the inverse mass operator alone, the memory-bound end of the path
        _case("mass64_k3_mixed", "inverse_mass", "tgv", (64, 64, 64), 3, "mixed"),
    ]


def draw(rng):
    """Another case of the same ranges: vortex, channel or curved box, k = 2..5, up to the listed node counts."""
    kind = rng.choice(["steps", "apply", "apply", "stage", "adjoint", "inverse_mass", "stored", "stored"])
    precision = rng.choice(["fp64", "mixed"])
    mesh, geometry, steps = "tgv", "affine", 1
    if kind == "stored":
        kind = rng.choice(["apply", "stage"])
        mesh = rng.choice(["channel", "sine"])
        geometry = "stored"
        k = rng.choice([2, 3, 5] if precision == "fp64" else [3, 5])
        low, high = 9, (32 if k <= 3 else 20)
    elif kind == "adjoint":
        k = rng.choice([2, 3, 4] if precision == "fp64" else [3, 4])
        low, high = 5, 24
    else:
        k = rng.choice([2, 3, 4, 5] if precision == "fp64" else [3, 4, 5])
        low, high = 5, {2: 80, 3: 60, 4: 46, 5: 38}[k]
        if kind == "steps" and precision == "mixed":
            kind = "stage"  # whole steps are compared in FP64
    m = math.exp(rng.uniform(math.log(low), math.log(high)))
    cells = [max(3, min(high, int(round(m * math.exp(rng.uniform(-0.25, 0.25)))))) for _ in range(3)]
    if kind == "steps":
        steps = max(1, min(10, int(20000 * 64 / (cells[0] * cells[1] * cells[2] * (k + 1) ** 3))))
    c = _case("", kind, mesh, cells, k, precision, geometry, steps)
    del c["name"]
    return c


def _setup(case):
    k = int(case["k"])
    if case["mesh"] == "channel":
        box = dict(lo=(0.0, -1.0, 0.0), hi=(TWO_PI, 1.0, math.pi), periodic=(1, 0, 1), mapping=api.MAP_CHANNEL,
                   map_param=1.8, Re=180.0, u_max=18.3, u_mach=18.3, body_force=(1.0, 0.0, 0.0))
    else:
        sine = case["mesh"] == "sine"
        box = dict(lo=(-math.pi,) * 3, hi=(math.pi,) * 3, periodic=(1, 1, 1),
                   mapping=api.MAP_SINE if sine else api.MAP_AFFINE, map_param=0.05 if sine else 0.0, Re=1600.0,
                   u_max=1.0, u_mach=0.0, body_force=(0.0, 0.0, 0.0))
    box.update(cells=(int(case["nx"]), int(case["ny"]), int(case["nz"])), k=k, nq_conv=(3 * k) // 2 + 1, nq_visc=k + 1,
               affine=case["mesh"] == "tgv", Ma=0.1, precision=api.MIXED if case["precision"] == "mixed" else api.FP64)
    h = [(box["hi"][d] - box["lo"][d]) / box["cells"][d] for d in range(3)]
    if case["mesh"] == "channel":
        c = 1.8
        h[1] = 1.0 - math.tanh(c * (1.0 - 2.0 / box["cells"][1])) / math.tanh(c)
    h_min = min(h) * (0.6 if case["mesh"] == "sine" else 1.0)
    # whole steps at the stability limit of the scheme; a single stage at a twentieth of it, as in a run that
    # resolves the start-up transient in time
    Cr = 0.02 if case["call"] == "stage" else 0.4
    box["dt"] = api.cfl_dt(k, h_min, box["u_max"], box["Ma"], Cr=Cr, D=0.02, nu=1.0 / box["Re"])
    # the adjoint integrates backwards along smooth trajectories, the others start from a rough field
    box["noise"] = 0.002 if case["call"] == "adjoint" else 0.05
    return box


# -- inputs ------------------------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _lgl(k):
    """k+1 Gauss--Lobatto--Legendre points on [0, 1]."""
    p = np.polynomial.legendre.Legendre.basis(k)
    d1, d2 = p.deriv(1), p.deriv(2)
    r = np.sort(np.real(d1.roots())) if k > 1 else np.zeros(0)
    for _ in range(3):
        r = r - d1(r) / d2(r) if r.size else r
    return 0.5 * (np.concatenate([[-1.0], r, [1.0]]) + 1.0)


def _node_coords(s):
    """[nz, ny, nx, 3, n, n, n]: the mesh mapping at the Lobatto nodes of every cell."""
    dev = _device()
    xi = torch.tensor(_lgl(s["k"]), dtype=torch.float64, device=dev)
    ax = []
    for d in range(3):
        n = s["cells"][d]
        h = (s["hi"][d] - s["lo"][d]) / n
        c = torch.arange(n, dtype=torch.float64, device=dev)
        shape = [1] * 6
        shape[2 - d], shape[5 - d] = n, len(xi)
        ax.append((s["lo"][d] + (c[:, None] + xi[None, :]) * h).reshape(shape))
    full = [s["cells"][2], s["cells"][1], s["cells"][0]] + [len(xi)] * 3
    x = [a.expand(full) for a in ax]
    if s["mapping"] == api.MAP_CHANNEL:
        c = s["map_param"]
        x[1] = torch.tanh(c * (2.0 * (x[1] + 1.0) / 2.0 - 1.0)) / math.tanh(c)
    elif s["mapping"] == api.MAP_SINE:
        X = [(x[d] - s["lo"][d]) / TWO_PI for d in range(3)]
        y = []
        for a in range(3):
            f = 1.0
            for b in range(3):
                f = f * torch.sin(TWO_PI * X[b] + 0.5 * a * (b + 1))
            y.append(x[a] + s["map_param"] * TWO_PI * f)
        x = y
    return torch.stack(x, 3)


def _state(s, seed):
    """The closed-form Taylor--Green state or the laminar channel profile at the nodes, with a seeded uniform
    perturbation of every velocity component by `noise` (5 %, the adjoint 0.2 %) of the reference velocity and of
    the pressure by the same share of rho u^2: [cells, 5, n^3]."""
    g = torch.Generator(device=_device())
    g.manual_seed(1806 + int(seed))
    xyz = _node_coords(s)
    x, y, z = xyz[:, :, :, 0], xyz[:, :, :, 1], xyz[:, :, :, 2]
    um = s["u_max"]
    T0 = (um / s["Ma"]) ** 2 / (GAMMA * GAS_R)
    if s["mapping"] == api.MAP_CHANNEL:
        u = [um * (1.0 - y * y), torch.zeros_like(y), torch.zeros_like(y)]
        p = torch.full_like(y, RHO0 * GAS_R * T0)
    else:
        u = [torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z),
             torch.zeros_like(x)]
        p = RHO0 * GAS_R * T0 + RHO0 / 16.0 * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)
    noise = torch.rand((4,) + tuple(x.shape), generator=g, dtype=torch.float64, device=x.device) * 2.0 - 1.0
    u = [u[a] + s["noise"] * um * noise[a] for a in range(3)]
    p = p + s["noise"] * RHO0 * um * um * noise[3]
    rho = p / (GAS_R * T0)
    rhoE = rho * (GAS_R / (GAMMA - 1.0) * T0 + 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
    U = torch.stack([rho, rho * u[0], rho * u[1], rho * u[2], rhoE], 3)
    return U.reshape(-1, 5, (s["k"] + 1) ** 3).contiguous()


def _covector(s, seed):
    """Seeded input of the adjoint and of the inverse mass operator: independent uniform values."""
    g = torch.Generator(device=_device())
    g.manual_seed(7000 + int(seed))
    shape = (s["cells"][0] * s["cells"][1] * s["cells"][2], 5, (s["k"] + 1) ** 3)
    w = torch.rand(shape, generator=g, dtype=torch.float64, device=_device()) * 2.0 - 1.0
    return w.to(torch.float32 if s["precision"] == api.MIXED else torch.float64)


def prepare(case, seed):
    s = _setup(case)
    g = api.DGCNS(s["cells"], s["lo"], s["hi"], s["periodic"], s["k"], s["nq_conv"], s["nq_visc"], gamma=GAMMA, Pr=PR,
                  Re=s["Re"], Ma=s["Ma"], R=GAS_R, rho0=RHO0, u_mach=s["u_mach"], body_force=s["body_force"],
                  precision=s["precision"], mapping=s["mapping"], map_param=s["map_param"],
                  geometry=1 if case["geometry"] == "fly" else 0)
    st = {"call": case["call"], "g": g, "dt": s["dt"], "steps": int(case["steps"])}
    if case["call"] in ("adjoint", "inverse_mass"):
        st["W"] = _covector(s, seed)
    if case["call"] != "inverse_mass":
        st["U"] = _state(s, seed)
    if case["call"] in ("apply", "adjoint", "inverse_mass", "stage", "steps"):
        st["R"] = g.empty_residual()
    if case["call"] in ("stage", "steps"):
        st["tmp"] = g.empty_state()
    if case["call"] == "stage":
        # the stage reads the previous stage's increment: a state-like field of the size dt L has
        st["dU0"] = (_covector(s, seed + 1) * 1e-3).contiguous()
        st["R"].copy_(st["dU0"])
    return st


def run(st):
    g = st["g"]
    if st["call"] == "steps":
        return g.dg_cns_rk_steps(st["steps"], st["dt"], 0.0, st["U"], st["tmp"], st["R"])
    if st["call"] == "stage":
        g.dg_cns_rk_stage(1, st["dt"], 0.0, st["U"], st["R"], st["tmp"])
        return {"U": st["tmp"], "dU": st["R"]}
    if st["call"] == "apply":
        return g.dg_cns_apply(st["U"], st["R"])
    if st["call"] == "adjoint":
        return g.dg_cns_adjoint_apply(st["U"], st["W"], st["R"])
    return g.dg_cns_inverse_mass(st["W"], st["R"])


def work(case):
    """Bytes: each input vector read once and each output written once (state 8 B, residual 8 or 4 B a value), the
    stored Jacobians read once.  Operations: the sum-factorized operator on every cell and each face once."""
    k = int(case["k"])
    n, qc, qv = k + 1, (3 * k) // 2 + 1, k + 1
    cells = case["nx"] * case["ny"] * case["nz"]
    vals = cells * 5 * n ** 3
    r = 4 if case["precision"] == "mixed" else 8
    interp = lambda q: 2 * (n * n * n * q + n * n * q * q + n * q * q * q)  # noqa: E731
    diff = lambda q: 6 * q ** 4  # noqa: E731
    face = lambda q: 2 * (n * n * q + n * q * q)  # noqa: E731
    mass = 5 * 12 * n ** 4 + 5 * n ** 3
    cell = 5 * (2 * interp(qc) + diff(qc)) + 60 * qc ** 3 + 5 * (2 * interp(qv) + 2 * diff(qv)) + 150 * qv ** 3
    traces = 5 * 4 * 2 * n ** 3
    faces = 3 * (2 * traces + 5 * 3 * face(qc) + 120 * qc ** 2 + 5 * 8 * face(qv) + 5 * 16 * qv ** 3 + 350 * qv ** 2)
    op = cells * (cell + faces + mass)
    geo = 0
    if case["geometry"] == "stored":
        geo = r * cells * (10 * (qc ** 3 + qv ** 3) + 39 * (qc ** 2 + qv ** 2) + n ** 3)
    call = case["call"]
    if call == "steps":
        return {"bytes": case["steps"] * 5 * vals * (16 + 2 * r), "flops": case["steps"] * 5 * op}
    if call == "stage":
        return {"bytes": vals * (16 + 2 * r) + geo, "flops": op}
    if call == "apply":
        return {"bytes": vals * (8 + r) + geo, "flops": op}
    if call == "adjoint":
        return {"bytes": vals * (8 + 2 * r), "flops": 2 * op}
    return {"bytes": vals * 2 * r, "flops": cells * mass}


# -- the same in plain torch FP64 ---------------------------------------------------------------------------------
def _lagrange(nodes, x):
    """V[p, i] = l_i(x_p), D[p, i] = l_i'(x_p)."""
    V, D = np.ones((len(x), len(nodes))), np.zeros((len(x), len(nodes)))
    for i, xi in enumerate(nodes):
        others = [m for m in range(len(nodes)) if m != i]
        for j in others:
            V[:, i] *= (x - nodes[j]) / (xi - nodes[j])
        for m in others:
            t = np.full(len(x), 1.0 / (xi - nodes[m]))
            for j in others:
                if j != m:
                    t *= (x - nodes[j]) / (xi - nodes[j])
            D[:, i] += t
    return V, D


def _along(M, a, d):
    """M applied along reference axis d (x = 0) of the last three axes (z, y, x)."""
    ax = a.dim() - 1 - d
    return torch.matmul(a.movedim(ax, -1), M.t()).movedim(-1, ax)


class _Exact:
    def __init__(self, s):
        self.s, self.n = s, s["k"] + 1
        dev = _device()
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        nodes = _lgl(s["k"])
        self.rule = {}
        for q in {s["nq_conv"], s["nq_visc"], self.n}:
            x, w = np.polynomial.legendre.leggauss(q)
            V, D = _lagrange(nodes, 0.5 * (x + 1.0))
            self.rule[q] = (t(V), t(D), t(0.5 * w))
        self.end = []
        for side in (0.0, 1.0):
            V, D = _lagrange(nodes, np.array([side]))
            self.end.append((t(V), t(D)))
        self.h = [(s["hi"][d] - s["lo"][d]) / s["cells"][d] for d in range(3)]
        self.xyz = None if s["affine"] else _node_coords(s)
        um = s["u_max"]
        self.mu = RHO0 / s["Re"]
        self.lam_cv = self.mu * GAMMA / PR
        self.T0 = (um / s["Ma"]) ** 2 / (GAMMA * GAS_R)
        self.cv = GAS_R / (GAMMA - 1.0)
        self.ref = [RHO0, 0.0, 0.0, 0.0, RHO0 * self.cv * self.T0]
        self.geo = {}
        self.tau = self._tau()

    # deviations u (5 leading on axis 3 -> list) from the reference state
    def _full(self, u):
        return [u[c] + self.ref[c] if self.ref[c] else u[c] for c in range(5)]

    def _pressure(self, u):
        """p - p_ref"""
        rho = u[0] + self.ref[0]
        return (GAMMA - 1.0) * (u[4] - 0.5 * (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) / rho)

    def conv(self, u):
        """F[c][a], without the constant reference pressure (zero residual on every cell)."""
        v = [u[1 + a] / (u[0] + self.ref[0]) for a in range(3)]
        dp = self._pressure(u)
        H = u[4] + dp + GAMMA * self.ref[4]
        F = [[u[1], u[2], u[3]]]
        for i in range(3):
            F.append([u[1 + i] * v[a] + (dp if a == i else 0.0) for a in range(3)])
        F.append([H * v[a] for a in range(3)])
        return F

    def visc(self, u, G):
        """F[c][a] of the gradient argument G[c][a]."""
        U = self._full(u)
        v = [U[1 + i] / U[0] for i in range(3)]
        E = U[4] / U[0]
        gu = [[(G[1 + i][a] - v[i] * G[0][a]) / U[0] for a in range(3)] for i in range(3)]
        div = gu[0][0] + gu[1][1] + gu[2][2]
        F = [[torch.zeros_like(div)] * 3, [], [], [], []]
        for a in range(3):
            tv = 0.0
            for i in range(3):
                tau = self.mu * (gu[i][a] + gu[a][i] - (2.0 / 3.0 * div if i == a else 0.0))
                F[1 + i].append(tau)
                tv = tv + tau * v[i]
            gE = (G[4][a] - E * G[0][a]) / U[0] - (v[0] * gu[0][a] + v[1] * gu[1][a] + v[2] * gu[2][a])
            F[4].append(tv + self.lam_cv * gE)
        return F

    # geometry: inverse Jacobian Ji[b][a] and |det J| of a list of derivatives dx_a / dxi_b
    @staticmethod
    def _invert(J):
        c = [[J[(a + 1) % 3][(b + 1) % 3] * J[(a + 2) % 3][(b + 2) % 3] -
              J[(a + 1) % 3][(b + 2) % 3] * J[(a + 2) % 3][(b + 1) % 3] for b in range(3)] for a in range(3)]
        det = J[0][0] * c[0][0] + J[0][1] * c[0][1] + J[0][2] * c[0][2]
        return [[c[a][b] / det for a in range(3)] for b in range(3)], det.abs()

    def cell_geo(self, q):
        if ("c", q) not in self.geo:
            if self.xyz is None:
                Ji = [[1.0 / self.h[b] if a == b else None for a in range(3)] for b in range(3)]
                self.geo["c", q] = (Ji, self.h[0] * self.h[1] * self.h[2])
            else:
                V, D, _ = self.rule[q]
                d = []
                for b in range(3):
                    a = self.xyz
                    for ax in range(3):
                        a = _along(D if ax == b else V, a, ax)
                    d.append(a)
                self.geo["c", q] = self._invert([[d[b][:, :, :, a] for b in range(3)] for a in range(3)])
        return self.geo["c", q]

    def face_geo(self, q, d, side):
        """Ji, outward unit normal and area element at the face points of every cell (axis d of extent 1)."""
        key = ("f", q, d, side)
        if key not in self.geo:
            sg = 1.0 if side else -1.0
            if self.xyz is None:
                Ji, _ = self.cell_geo(q)
                self.geo[key] = (Ji, [sg if a == d else None for a in range(3)], self.h[(d + 1) % 3] * self.h[(d + 2) % 3])
            else:
                V, D, _ = self.rule[q]
                g = []
                for b in range(3):
                    x = self.xyz
                    for ax in range(3):
                        M = self.end[side] if ax == d else (V, D)
                        x = _along(M[1] if ax == b else M[0], x, ax)
                    g.append(x)
                Ji, det = self._invert([[g[b][:, :, :, a] for b in range(3)] for a in range(3)])
                nv = [sg * Ji[d][a] for a in range(3)]
                nn = torch.sqrt(nv[0] ** 2 + nv[1] ** 2 + nv[2] ** 2)
                self.geo[key] = (Ji, [v / nn for v in nv], det * nn)
        return self.geo[key]

    def _weights(self, q, skip=None):
        w = self.rule[q][2]
        one = torch.ones(1, dtype=torch.float64, device=w.device)
        wz, wy, wx = (one if skip == 2 else w), (one if skip == 1 else w), (one if skip == 0 else w)
        return wz[:, None, None] * wy[None, :, None] * wx[None, None, :]

    def _tau(self):
        s, q = self.s, self.s["nq_conv"]
        shape = (s["cells"][2], s["cells"][1], s["cells"][0])
        one = torch.ones(shape + (1, 1, 1), dtype=torch.float64, device=_device())
        total = lambda v, w: (one * v * w).sum((-1, -2, -3))  # noqa: E731
        vol = total(self.cell_geo(q)[1], self._weights(q))
        area = torch.zeros_like(vol)
        for d in range(3):
            for side in (0, 1):
                a = total(self.face_geo(q, d, side)[2], self._weights(q, d))
                f = torch.full_like(a, 0.5)
                if not s["periodic"][d]:
                    f.select(2 - d, -1 if side else 0).fill_(1.0)
                area = area + a * f
        return self.mu / RHO0 * self.n ** 2 * area / vol

    @staticmethod
    def _phys(Ji, g):
        """Physical gradient G[c][a] of reference derivatives g[b][c]."""
        return [[sum(Ji[b][a] * g[b][c] for b in range(3) if Ji[b][a] is not None) for a in range(3)] for c in range(5)]

    @staticmethod
    def _ref_flux(Ji, F, w):
        """Contravariant flux [b] -> stacked components, times w."""
        return [torch.stack([w * sum(Ji[b][a] * F[c][a] for a in range(3) if Ji[b][a] is not None) for c in range(5)], 3)
                for b in range(3)]

    def _points(self, dU, q):
        V = self.rule[q][0]
        for d in range(3):
            dU = _along(V, dU, d)
        return dU

    def _cell(self, dU):
        out = 0.0
        for q, viscous in ((self.s["nq_conv"], False), (self.s["nq_visc"], True)):
            V, D, _ = self.rule[q]
            Ji, det = self.cell_geo(q)
            u = self._points(dU, q).unbind(3)
            w = self._weights(q) * det
            if viscous:
                g = []
                for b in range(3):
                    a = dU
                    for ax in range(3):
                        a = _along(D if ax == b else V, a, ax)
                    g.append(a.unbind(3))
                Ft = self._ref_flux(Ji, self.visc(u, self._phys(Ji, g)), w)
            else:
                Ft = self._ref_flux(Ji, self.conv(u), -w)
            for b in range(3):
                a = Ft[b]
                for ax in range(3):
                    a = _along((D if ax == b else V).t(), a, ax)
                out = out + a
        return out

    def _trace(self, dU, q, d, side):
        """Values and reference derivatives [b] at the face points of every cell."""
        V, D, _ = self.rule[q]
        got = []
        for b in (None, 0, 1, 2):
            a = dU
            for ax in range(3):
                M = self.end[side] if ax == d else (V, D)
                a = _along(M[1] if ax == b else M[0], a, ax)
            got.append(a.unbind(3))
        return got[0], got[1:]

    def _test_value(self, f, q, d, side):
        a = torch.stack(f, 3)
        V = self.rule[q][0]
        for ax in range(3):
            a = _along((self.end[side][0] if ax == d else V).t(), a, ax)
        return a

    def _test_grad(self, Ft, q, d, side):
        V, D, _ = self.rule[q]
        out = 0.0
        for b in range(3):
            a = Ft[b]
            for ax in range(3):
                M = self.end[side] if ax == d else (V, D)
                a = _along((M[1] if ax == b else M[0]).t(), a, ax)
            out = out + a
        return out

    def _ghost(self, u):
        """No-slip isothermal wall: rho+ = rho-, u+ = -u-, T+ = 2 T_w - T-, as deviations."""
        rho = u[0] + self.ref[0]
        ke = 0.5 * (u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / rho
        internal = u[4] + self.ref[4] - ke
        return [u[0], -u[1], -u[2], -u[3], 2.0 * rho * self.cv * self.T0 - internal + ke - self.ref[4]]

    def _face(self, dU, d, side):
        """The own shares of every cell on its face (d, side)."""
        s = self.s
        out = 0.0
        shift = -1 if side else 1
        to = lambda a: torch.roll(a, shift, 2 - d)  # noqa: E731
        wall = None
        if not s["periodic"][d]:
            wall = torch.zeros((s["cells"][2], s["cells"][1], s["cells"][0], 1, 1, 1), dtype=torch.bool, device=dU.device)
            wall.select(2 - d, -1 if side else 0).fill_(True)
        for q, viscous in ((s["nq_conv"], False), (s["nq_visc"], True)):
            Ji, nrm, dA = self.face_geo(q, d, side)
            w = self._weights(q, d) * dA
            um, gm = self._trace(dU, q, d, side)
            up, gp = self._trace(dU, q, d, 1 - side)
            up = [to(a) for a in up]
            if wall is not None:
                up = [torch.where(wall, g, a) for g, a in zip(self._ghost(um), up)]
            dot = lambda F: [sum(F[c][a] * nrm[a] for a in range(3) if nrm[a] is not None) for c in range(5)]  # noqa: E731
            if not viscous:
                lam = []
                for u in (um, up):
                    rho = u[0] + self.ref[0]
                    p = self._pressure(u) + (GAMMA - 1.0) * self.ref[4]
                    lam.append(torch.sqrt(u[1] ** 2 + u[2] ** 2 + u[3] ** 2) / rho + torch.sqrt((GAMMA * p / rho).abs()))
                lam = torch.maximum(lam[0], lam[1])
                fm, fp = dot(self.conv(um)), dot(self.conv(up))
                out = out + self._test_value([w * 0.5 * (fm[c] + fp[c] + lam * (um[c] - up[c])) for c in range(5)], q, d, side)
                continue
            Gm = self._phys(Ji, gm)
            Jo = self.face_geo(q, d, 1 - side)[0]
            if self.xyz is not None:
                Jo = [[to(Jo[b][a]) for a in range(3)] for b in range(3)]
            Gp = self._phys(Jo, [[to(a) for a in g] for g in gp])
            tau = self.tau[..., None, None, None]
            other = to(tau)
            if wall is not None:
                Gp = [[torch.where(wall, Gm[c][a], Gp[c][a]) for a in range(3)] for c in range(5)]
                other = torch.where(wall, tau, other)
            tau = torch.maximum(tau, other)
            jump = [um[c] - up[c] for c in range(5)]
            fm, fp = dot(self.visc(um, Gm)), dot(self.visc(up, Gp))
            out = out + self._test_value([-w * (0.5 * (fm[c] + fp[c]) - tau * jump[c]) for c in range(5)], q, d, side)
            Jg = [[jump[c] * nrm[a] if nrm[a] is not None else torch.zeros_like(jump[c]) for a in range(3)] for c in range(5)]
            out = out + self._test_grad(self._ref_flux(Ji, self.visc(um, Jg), -0.5 * w), q, d, side)
        return out

    def inverse_mass(self, r):
        Si = torch.linalg.inv(self.rule[self.n][0])
        for d in range(3):
            r = _along(Si.t(), r, d)
        det = self.cell_geo(self.n)[1]
        w = self._weights(self.n) * det
        r = r / (w.unsqueeze(3) if w.dim() == 6 else w)
        for d in range(3):
            r = _along(Si, r, d)
        return r

    def deviation(self, U):
        s = self.s
        ref = torch.tensor(self.ref, dtype=torch.float64, device=U.device)
        return (U.double() - ref[None, :, None]).reshape(s["cells"][2], s["cells"][1], s["cells"][0], 5, self.n, self.n, self.n)

    def L(self, dU):
        r = self._cell(dU)
        for d in range(3):
            for side in (0, 1):
                r = r + self._face(dU, d, side)
        r = self.inverse_mass(-r)
        if any(self.s["body_force"]):
            f = self.s["body_force"]
            u = self._points(dU, self.n).unbind(3)
            e = (f[0] * u[1] + f[1] * u[2] + f[2] * u[3]) / (u[0] + self.ref[0])
            Si = torch.linalg.inv(self.rule[self.n][0])
            for d in range(3):
                e = _along(Si, e, d)
            one = torch.ones_like(e)
            r = r + torch.stack([0.0 * one, f[0] * one, f[1] * one, f[2] * one, e], 3)
        return r


def exact(case, seed):
    s = _setup(case)
    call = case["call"]
    evaluations = 5 * int(case["steps"]) if call == "steps" else 1
    if evaluations * s["cells"][0] * s["cells"][1] * s["cells"][2] * (s["k"] + 1) ** 3 > 1.8e7:
        return None  # over 20 seconds
    x = _Exact(s)
    shape = (s["cells"][0] * s["cells"][1] * s["cells"][2], 5, (s["k"] + 1) ** 3)
    flat = lambda a: a.reshape(shape)  # noqa: E731
    if call == "inverse_mass":
        W = _covector(s, seed).double().reshape(s["cells"][2], s["cells"][1], s["cells"][0], 5, x.n, x.n, x.n)
        return flat(x.inverse_mass(W))
    U = _state(s, seed)
    if call == "adjoint":
        d = x.deviation(U).requires_grad_(True)
        W = _covector(s, seed).double().reshape(d.shape)
        return flat(torch.autograd.grad((x.L(d) * W).sum(), d)[0])
    with torch.no_grad():
        d = x.deviation(U)
        if call == "apply":
            return flat(x.L(d))
        if call == "stage":
            dU = (_covector(s, seed + 1) * 1e-3).double()
            dU = RK_A[1] * dU + s["dt"] * flat(x.L(d))
            return {"U": U + RK_B[1] * dU, "dU": dU}
        dU = torch.zeros_like(U)
        for _ in range(int(case["steps"])):
            for a, b in zip(RK_A, RK_B):
                dU = a * dU + s["dt"] * flat(x.L(x.deviation(U)))
                U = U + b * dU
        return U
