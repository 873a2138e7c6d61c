"""What this library is measured on, and the same results in plain 64-bit torch.

A case is one call a solver program makes over and over, on the meshes and flow
parameters of the repository's own workloads (ssd_inputs) and on other sizes of
the same families: advance a number of steps and read the state, evaluate a
residual, or exchange the state with a host program around one step.
``listed()`` names twelve of them from the smallest (where launches and latency
count) to the largest; ``draw`` gives others of the same ranges.  ``exact``
evaluates the method (arXiv:1503.02198: Secs. 2.1-2.3, 3.1, 3.2, explicit SSP
Runge-Kutta) with batched torch operations in float64.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1503_02198_gb300 as ssd
from ssd_inputs import meshes, workloads

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
PRECISION = {"fp64": ssd.SD_PREC_FP64, "fp32": ssd.SD_PREC_FP32, "fp32s": ssd.SD_PREC_FP32S}


def _case(name, family, scale, N, precision, call="step", steps=1, rk=3):
    c = {"family": family, "scale": scale, "N": N, "precision": precision, "call": call, "steps": steps, "rk": rk}
    return dict(c, name=name) if name else c


def listed():
    return [
        # Taylor-Couette, 288 cells, Navier-Stokes: the smallest mesh, one step per call as a program does
        # that looks at the flow after every step; launches and latency
        _case("couette_n3_fp64", "couette", 1.0, 3, "fp64"),
        # the same mesh as a long run advances it
        _case("couette_n3_fp32", "couette", 1.0, 3, "fp32", steps=20),
        # Euler vortex through a rotor, 6,016 cells: an ordinary small run
        _case("vortex_n4_fp32", "vortex", 1.0, 4, "fp32", steps=10),
        # the state kept by a host program: in from pinned memory, one step, out to pinned memory
        _case("vortex_n5_fp32_host", "vortex", 1.0, 5, "fp32", call="exchange"),
        # one residual of the reference precision, as an implicit or steady-state driver asks for it
        _case("vortex_n5_fp64_residual", "vortex", 1.0, 5, "fp64", call="residual"),
        # lowest order on a ragged mesh of odd sizes (31,509 cells)
        _case("vortex_n3_fp32_odd", "vortex", 2.29, 3, "fp32", steps=3),
        # stirred tank, 14,752 cells, Navier-Stokes with adiabatic blades, the five-stage scheme of Sec. 4
        _case("tank_n4_fp32_rk5", "tank", 1.0, 4, "fp32", steps=2, rk=5),
        # flow past the rotating ellipse, 20,096 cells, Navier-Stokes, cubic cells, every boundary kind
        _case("ellipse_n5_fp32", "ellipse", 1.0, 5, "fp32", steps=5),
        _case("ellipse_n5_fp64", "ellipse", 1.0, 5, "fp64"),
        # two counter-rotating rotors, 123,450 cells, FP32 state storage
        _case("twin_n6_fp32s", "twin", 1.0, 6, "fp32s", steps=3),
        # the largest configuration, 246,900 cells: production precision, and the reference precision
        _case("rotor_n6_fp32", "rotor", 1.0, 6, "fp32", steps=4),
        _case("rotor_n6_fp64", "rotor", 1.0, 6, "fp64"),
    ]


# scales each family is run at (cells grow with the square): 288 to about 247,000 cells
SCALES = {"couette": (1.0, 9.0), "vortex": (0.4, 5.0), "tank": (0.45, 1.0), "ellipse": (0.3, 1.5), "twin": (0.25, 1.0),
          "rotor": (0.25, 1.0)}


def draw(rng):
    family = rng.choice(sorted(SCALES))
    lo, hi = SCALES[family]
    scale = round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 3)
    N = rng.choice([3, 4, 5, 6])
    precision = rng.choice(["fp32", "fp32", "fp64", "fp32s"])
    call = "residual" if precision == "fp64" and rng.random() < 0.4 else "exchange" if rng.random() < 0.1 else "step"
    rk = 5 if rng.random() < 0.25 else 3
    steps = 1
    if call == "step" and precision != "fp64":
        steps = rng.choice([1, 2, 3, 4] if family in ("rotor", "twin") or scale > 2.0 else [1, 3, 5, 10])
    if family in ("rotor", "twin") and precision == "fp64":
        rk = 3
    return _case(None, family, scale, N, precision, call, steps, rk)


# ---------------------------------------------------------------------------
# meshes and flows
# ---------------------------------------------------------------------------


def _even(x, least):
    return max(least, 2 * int(round(x / 2)))


@functools.lru_cache(maxsize=3)
def _problem(family, scale, N, rk):
    """(mesh, flow parameters, step size) of a family at a scale."""
    s = scale
    if family == "couette":
        m = max(1, int(round(4 * s)))
        mesh = meshes.couette_mesh(m, 8 * m, m, 10 * m)
        c = 0.5 / 0.1  # inner wall at speed 0.5, Mach 0.1
        prm = workloads.FlowParams(Rgas=c * c / 1.4, mu=0.05, omega=0.5, viscous=1)
        speed = c + 0.5
    elif family == "tank":
        mesh = meshes.stirred_tank_mesh(n_theta_in=6 * max(8, int(round(28 * s))), n_theta_out=4 * max(8, int(round(50 * s))),
                                        layers_in=tuple(max(3, int(round(k * s))) for k in (10, 16, 14)),
                                        layers_out=tuple(max(3, int(round(k * s))) for k in (20, 22)))
        prm = workloads.tank_params()
        speed = math.sqrt(prm.gamma * prm.Rgas) + 3.0
    elif family == "ellipse":
        mesh = meshes.ellipse_mesh(n_theta=max(16, 4 * int(round(32 * s))), n_inner=max(3, int(round(40 * s))),
                                   n_outer=max(4, int(round(117 * s))))
        prm = workloads.ellipse_params()
        speed = 1.6 + math.sqrt(prm.gamma * prm.p_inf)
    else:
        # Euler families: (box half width, Cartesian cells, hole, core, rings) at scale 1
        half, cart, hole, r, core, half_core, ring_in, ring_out, omega = {
            "vortex": (10.0, 64, 24, 3.0, 24, 1.5, 16, 4, math.pi / 4),
            "rotor": (20.0, 500, 120, 4.0, 50, 2.0, 20, 10, 0.5),
            "twin": (10.0, 250, 60, 2.0, 25, 1.0, 10, 5, 0.5)}[family]
        nc = _even(cart * s, 8)
        nh = _even(hole * s, 4)
        while nh / nc * half <= 1.02 * r:  # the circle stays inside the hole
            nh += 2
        kw = dict(half_width=half, n_cart=nc, n_hole=nh, r_interface=r, n_core=max(2, int(round(core * s))),
                  core_half=half_core, n_ring_in=max(2, int(round(ring_in * s))), n_ring_out=max(1, int(round(ring_out * s))))
        mesh = meshes.twin_rotor_mesh(omega2=-omega, **kw) if family == "twin" else meshes.rotor_mesh(**kw)
        prm = workloads.FlowParams(omega=omega)
        speed = 2.0 + math.sqrt(1.4) + omega * r
    prm.rk_stages = rk
    return mesh, prm, workloads.stable_dt(mesh, N, prm, speed)


def _problem_of(case):
    return _problem(case["family"], case["scale"], case["N"], case["rk"])


def _begin(case, seed):
    """The time the run starts at (any rotor position) and the seeded field modes."""
    rng = np.random.Generator(np.random.PCG64([seed, 1503]))
    prm = _problem_of(case)[1]
    t0 = float(rng.uniform(0.0, 2.0 * math.pi / prm.omega))
    modes = [[(kx, ky, float(rng.uniform(-1, 1)), float(rng.uniform(0, 2 * math.pi)))
              for kx in (-1, 0, 2) for ky in (-2, 0, 1)] for _ in range(4)]
    return t0, modes, float(rng.uniform(-1.5, 1.5)), float(rng.uniform(-1.5, 1.5))


def _field(case, modes, x0, y0, x, y):
    """Start state [E][4][N][N] at the solution points: the family's flow (vortex, fluid at rest, or the free
    stream that already turns with the body) with smooth seeded waves of one per cent on it."""
    mesh, prm, _ = _problem_of(case)
    rho, p = torch.full_like(x, prm.rho_inf), torch.full_like(x, prm.p_inf)
    u, v = torch.zeros_like(x), torch.zeros_like(x)
    if case["family"] in ("rotor", "twin", "vortex"):
        eps, r2 = 5.0 / (2.0 * math.pi), (x - x0) ** 2 + (y - y0) ** 2
        e1 = torch.exp(0.5 * (1.0 - r2))
        u, v = 1.0 - eps * (y - y0) * e1, eps * (x - x0) * e1
        base = 1.0 - 0.2 * eps * eps / 1.4 * torch.exp(1.0 - r2)
        rho, p = base ** 2.5, base ** 3.5
    elif case["family"] == "ellipse":
        s = torch.sqrt((x / 0.5) ** 2 + (y / 0.1) ** 2) - 1.0
        phi = 1.0 - torch.exp(-torch.clamp(s, min=0.0) ** 2)
        u, v = phi - (1.0 - phi) * prm.omega * y, (1.0 - phi) * prm.omega * x
    else:
        p = torch.full_like(x, prm.Rgas)
    lo, span = mesh["xy"].min(axis=0), np.ptp(mesh["xy"], axis=0)
    kx, ky = 2.0 * math.pi / float(span[0]) * (x - float(lo[0])), 2.0 * math.pi / float(span[1]) * (y - float(lo[1]))
    w = [0.01 / 3.0 * sum(a * torch.sin(i * kx + j * ky + ph) for i, j, a, ph in m) for m in modes]
    rho, p, u, v = rho * (1.0 + w[0]), p * (1.0 + w[1]), u + w[2], v + w[3]
    return torch.stack([rho, rho * u, rho * v, p / (prm.gamma - 1.0) + 0.5 * rho * (u * u + v * v)], dim=1).contiguous()


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------


def prepare(case, seed):
    mesh, prm, dt = _problem_of(case)
    solver = ssd.Solver(mesh, case["N"] - 1, prm, precision=PRECISION[case["precision"]])
    t0, modes, x0, y0 = _begin(case, seed)
    xy = torch.empty((solver.E, solver.N, solver.N, 2), dtype=torch.float64, device=DEVICE)
    solver.sd_sp_coords(t0, xy)
    Q = _field(case, modes, x0, y0, xy[..., 0], xy[..., 1])
    torch.cuda.synchronize()
    state = {"solver": solver, "dt": dt, "steps": case["steps"], "call": case["call"]}
    if case["call"] == "exchange":
        state["host"] = Q.cpu().pin_memory()
    else:
        state["out"] = torch.empty_like(Q)
        solver.sd_set_state(Q)
    solver.sd_set_time(t0)  # (waits until Q has been read)
    return state


def run(state):
    s = state["solver"]
    if state["call"] == "residual":
        return s.sd_residual(state["out"])
    if state["call"] == "exchange":
        s.sd_set_state(state["host"])
        s.sd_step(state["dt"], 1)
        return s.sd_get_state(state["host"])
    s.sd_step(state["dt"], state["steps"])
    return s.sd_get_state(state["out"])


def work(case):
    """One pass: the state read and written once in the form it is stored in, the result written as float64 (or the
    state crossing from and to the host), each cell's and face's geometry once; the operations of the method's
    contractions and fluxes (an FMA is two) for every stage."""
    mesh, prm, _ = _problem_of(case)
    E, N = len(mesh["elem_nodes"]), case["N"]
    values, stored = 4 * E * N * N, 4 if case["precision"] == "fp32s" else 8
    stages = 1 if case["call"] == "residual" else case["steps"] * case["rk"]
    state = values * (stored if case["call"] == "residual" else 2 * stored)
    line = (N - 1) * (8 * N + 28) + (N + 1) * 8 * N + 16 * N  # interpolation and flux, divergence, traces
    flops = 2 * N * line + 34 * N * N + 2 * N * 70            # lines, solution points, two faces of a cell
    if prm.viscous:
        flops += 2 * N * (4 * (2 * N * (N - 1) + 2 * N * (N + 1)) + (N - 1) * (16 * N + 70) + 32 * N) + 24 * N * N + 2 * N * 160
    return {"bytes": float(state + 8 * values * (2 if case["call"] == "exchange" else 1) + E * (64 + 2 * 16)),
            "flops": float(E) * flops * stages}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------

FACE_A, FACE_B = (0, 1, 3, 0), (1, 2, 2, 3)  # corners a face's parameter runs between
SIGMA = (-1.0, 1.0, 1.0, -1.0)               # sign of a face's metric vector against the outward normal


def _lagrange(nodes, x):
    """Values and derivatives [len(x)][len(nodes)] of the Lagrange polynomials on nodes."""
    n = len(nodes)
    val, der = np.empty((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        others = [k for k in range(n) if k != i]
        den = np.prod([nodes[i] - nodes[k] for k in others])
        val[:, i] = np.prod([x - nodes[k] for k in others], axis=0) / den
        for m in others:
            der[:, i] += np.prod([x - nodes[k] for k in others if k != m] or [np.ones(len(x))], axis=0) / den
    return val, der


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=DEVICE)


class _Method:
    """The semi-discrete operator of one mesh: residual(Q, t) and steps."""

    def __init__(self, mesh, N, prm):
        self.N, self.prm = N, prm
        en = mesh["elem_nodes"]
        self.E = E = len(en)
        Xs = 0.5 - 0.5 * np.cos(np.pi * (2 * np.arange(N) + 1) / (2 * N))
        Xf = np.concatenate([[0.0], 0.5 * (1 + np.polynomial.legendre.leggauss(N - 1)[0]), [1.0]])
        z, w = np.polynomial.legendre.leggauss(N)
        z, w = 0.5 * (1 + z), 0.5 * w
        Hz = _lagrange(Xs, z)[0]
        self.Xs_np, self.z_np = Xs, z
        self.Xs, self.Hf, self.Dm, self.Hz, self.wq = _t(Xs), _t(_lagrange(Xs, Xf)[0]), _t(_lagrange(Xf, Xs)[1]), _t(Hz), _t(w)
        self.Minv = _t(np.linalg.inv(np.einsum("q,qi,qj->ij", w, Hz, Hz)))
        # zones: centre and rate, the frame zone each cell's coordinates are taken about
        zones = [{"center": mesh["center"], "omega": prm.omega, "r_interface": mesh["r_interface"],
                  "ifaces_L": mesh["ifaces_L"], "ifaces_R": mesh["ifaces_R"]}] + list(mesh.get("zones", []))
        centres = np.array([[0.0, 0.0]] + [z_["center"] for z_ in zones])
        self.omega = np.array([0.0] + [z_["omega"] for z_ in zones])
        zone = np.asarray(mesh["elem_zone"])
        frame = np.asarray(mesh.get("elem_arc_zone", np.where(zone > 0, zone, 1)))
        self.zone = torch.as_tensor(zone.astype(np.int64), device=DEVICE)
        self.centre = _t(centres[frame])
        self.kind = torch.as_tensor(np.asarray(mesh["edge_arc"]).astype(np.int64), device=DEVICE)
        self.P = _t(mesh["xy"][en]) - self.centre[:, None]
        if "edge_nodes" in mesh:
            self.M = _t(mesh["xy"][np.maximum(mesh["edge_nodes"], 0)]) - self.centre[:, None, None]
        om = _t(self.omega)[self.zone][:, None]
        X, Y = np.meshgrid(Xf, Xs)  # xi flux points [j][i]
        p, dx, de = self._map(X.ravel(), Y.ravel())
        self.a = torch.stack([de[..., 1], -de[..., 0]], -1).view(E, N, N + 1, 2)
        self.ga = (om * (-p[..., 1] * de[..., 1] - p[..., 0] * de[..., 0])).view(E, N, N + 1)
        X, Y = np.meshgrid(Xs, Xf)  # eta flux points [l][i]
        p, dx, de = self._map(X.ravel(), Y.ravel())
        self.b = torch.stack([-dx[..., 1], dx[..., 0]], -1).view(E, N + 1, N, 2)
        self.gb = (om * (p[..., 1] * dx[..., 1] + p[..., 0] * dx[..., 0])).view(E, N + 1, N)
        X, Y = np.meshgrid(Xs, Xs)
        self.xy, dx, de = self._map(X.ravel(), Y.ravel())
        self.J = (dx[..., 0] * de[..., 1] - de[..., 0] * dx[..., 1]).view(E, 1, N, N)
        self.gxi = torch.stack([de[..., 1], -de[..., 0]], -1).view(E, N, N, 2) / self.J[:, 0, ..., None]
        self.get = torch.stack([-dx[..., 1], dx[..., 0]], -1).view(E, N, N, 2) / self.J[:, 0, ..., None]
        self.sigma = _t(np.tile(SIGMA, E))[:, None]
        # faces: boundary, periodic and conforming pairs (both sides' element face, reversed point order)
        xy, ea, eb = mesh["xy"], en[:, FACE_A].ravel(), en[:, FACE_B].ravel()
        taken = np.zeros(4 * E, dtype=bool)
        bf = np.asarray(mesh["bfaces"]).reshape(-1, 3)
        self.bef, self.tag = 4 * bf[:, 0] + bf[:, 1], torch.as_tensor(bf[:, 2].astype(np.int64), device=DEVICE)
        pf = np.asarray(mesh["pfaces"]).reshape(-1, 4)
        pA, pB = 4 * pf[:, 0] + pf[:, 1], 4 * pf[:, 2] + pf[:, 3]
        prev = ((xy[eb[pA]] - xy[ea[pA]]) * (xy[eb[pB]] - xy[ea[pB]])).sum(1) < 0
        taken[np.concatenate([self.bef, pA, pB])] = True
        self.ifaces = []
        for k, z_ in enumerate(zones):
            if len(z_["ifaces_L"]) == 0:
                continue
            sides = []
            for key in ("ifaces_L", "ifaces_R"):
                f = np.asarray(z_[key]).reshape(-1, 2)
                ef = 4 * f[:, 0] + f[:, 1]
                taken[ef] = True
                # angles in extended precision: mortar offsets are differences of nearly equal angles
                A, B = (xy[n[ef]].astype(np.longdouble) - np.asarray(z_["center"], dtype=np.longdouble) for n in (ea, eb))
                d = np.arctan2(A[:, 0] * B[:, 1] - A[:, 1] * B[:, 0], (A * B).sum(1))
                start = np.where(d > 0, np.arctan2(A[:, 1], A[:, 0]), np.arctan2(B[:, 1], B[:, 0])) % self._two_pi()
                o = np.argsort(start)
                sides.append((ef[o], start[o], np.abs(d)[o], (d < 0)[o]))
            self.ifaces.append((k + 1, z_["r_interface"], sides))
        free = np.flatnonzero(~taken)
        key = np.minimum(ea[free], eb[free]).astype(np.int64) * len(xy) + np.maximum(ea[free], eb[free])
        pairs = free[np.argsort(key, kind="stable")].reshape(-1, 2)
        self.efA = np.concatenate([pA, pairs[:, 0]])
        self.efB = np.concatenate([pB, pairs[:, 1]])
        rev = np.concatenate([prev, ea[pairs[:, 0]] != ea[pairs[:, 1]]])
        self.efA, self.efB, self.bef = (torch.as_tensor(v.astype(np.int64), device=DEVICE) for v in (self.efA, self.efB, self.bef))
        self.rev = torch.as_tensor(rev, device=DEVICE)[:, None, None]

    @staticmethod
    def _two_pi():
        return 2 * np.arccos(np.longdouble(-1))

    def _map(self, xi, eta):
        """Position relative to the frame centre and its xi and eta derivatives, [E][points][2], at t = 0: the
        transfinite map of the cell's four edges (straight, circular arc about the centre, or cubic)."""
        xi, eta = _t(xi)[None, :, None], _t(eta)[None, :, None]
        edges = []
        for f in range(4):
            u = xi if f in (0, 2) else eta
            A, B = self.P[:, FACE_A[f], None], self.P[:, FACE_B[f], None]
            off, der = u * (B - A), (B - A) + 0.0 * u
            i = torch.nonzero(self.kind[:, f] == 1)[:, 0]
            if len(i):
                a, b, uu = A[i], B[i], u[..., 0]
                r, phi = a.norm(dim=-1), torch.atan2(a[..., 1], a[..., 0])
                d = torch.atan2(a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0], (a * b).sum(-1))
                chord, mid, end = 2.0 * r * torch.sin(0.5 * uu * d), phi + 0.5 * uu * d, phi + uu * d
                off[i] = torch.stack([-chord * torch.sin(mid), chord * torch.cos(mid)], -1)
                der[i] = (r * d)[..., None] * torch.stack([-torch.sin(end), torch.cos(end)], -1)
            i = torch.nonzero(self.kind[:, f] == 2)[:, 0]
            if len(i):
                val, dv = _lagrange(np.array([0.0, 1 / 3, 2 / 3, 1.0]), u.reshape(-1).cpu().numpy())
                nodes = torch.stack([A[i, 0], self.M[i, f, 0], self.M[i, f, 1], B[i, 0]], 1) - A[i]
                off[i], der[i] = torch.einsum("pk,ekc->epc", _t(val), nodes), torch.einsum("pk,ekc->epc", _t(dv), nodes)
            edges.append((off, der))
        c0, c1, c2, c3 = (self.P[:, k, None] - self.P[:, 0, None] for k in range(4))
        (bo, bd), (ro, rd), (to, td), (lo, ld) = edges
        ro, to = ro + c1, to + c3
        a, b = 1.0 - xi, 1.0 - eta
        x = b * bo + eta * to + a * lo + xi * ro - (xi * b * c1 + xi * eta * c2 + a * eta * c3)
        dxi = b * bd + eta * td - lo + ro - (b * c1 + eta * c2 - eta * c3)
        deta = -bo + to + a * ld + xi * rd - (-xi * c1 + xi * c2 + a * c3)
        return self.P[:, 0, None] + x, dxi, deta

    def _turn(self, v, t, extra):
        th = _t(self.omega * t)[self.zone].view(-1, *([1] * extra))
        c, s = torch.cos(th), torch.sin(th)
        return torch.stack([c * v[..., 0] - s * v[..., 1], s * v[..., 0] + c * v[..., 1]], -1)

    def points(self, t):
        return (self.centre[:, None] + self._turn(self.xy, t, 1)).view(self.E, self.N, self.N, 2)

    # ---- physics (Sec. 2.1); the variables run along dimension 1 ----
    def _pressure(self, q):
        return (self.prm.gamma - 1.0) * (q[:, 3] - 0.5 * (q[:, 1] ** 2 + q[:, 2] ** 2) / q[:, 0])

    def _flux(self, q, nx, ny, vg):
        p, un = self._pressure(q), (q[:, 1] * nx + q[:, 2] * ny) / q[:, 0]
        return torch.stack([q[:, 0] * (un - vg), q[:, 1] * (un - vg) + p * nx, q[:, 2] * (un - vg) + p * ny,
                            (q[:, 3] + p) * un - vg * q[:, 3]], 1)

    def _rusanov(self, qL, qR, nx, ny, vg):
        speed = [torch.abs((q[:, 1] * nx + q[:, 2] * ny) / q[:, 0] - vg) + torch.sqrt(self.prm.gamma * self._pressure(q) / q[:, 0])
                 for q in (qL, qR)]
        lam = torch.maximum(*speed)[:, None]
        return 0.5 * (self._flux(qL, nx, ny, vg) + self._flux(qR, nx, ny, vg)) - 0.5 * lam * (qR - qL)

    def _viscous(self, q, gx, gy, nx, ny, conduct=1.0):
        g = self.prm
        k = g.mu * g.gamma * g.Rgas / ((g.gamma - 1.0) * g.prandtl) * conduct
        rho, u, v = q[:, 0], q[:, 1] / q[:, 0], q[:, 2] / q[:, 0]
        p = self._pressure(q)
        d = []
        for gr in (gx, gy):
            du, dv = (gr[:, 1] - u * gr[:, 0]) / rho, (gr[:, 2] - v * gr[:, 0]) / rho
            dp = (g.gamma - 1.0) * (gr[:, 3] - 0.5 * (u * u + v * v) * gr[:, 0] - rho * (u * du + v * dv))
            d.append((du, dv, (dp - p / rho * gr[:, 0]) / (rho * g.Rgas)))
        (ux, vx, Tx), (uy, vy, Ty) = d
        lam = -2.0 / 3.0 * g.mu * (ux + vy)
        txx, tyy, txy = 2.0 * g.mu * ux + lam, 2.0 * g.mu * vy + lam, g.mu * (uy + vx)
        fx, fy = u * txx + v * txy + k * Tx, u * txy + v * tyy + k * Ty
        return -torch.stack([torch.zeros_like(u), txx * nx + txy * ny, txy * nx + tyy * ny, fx * nx + fy * ny], 1)

    def _boundary(self, q, nx, ny, ug, vg):
        """Ghost state and state on the boundary by tag: wall, slip, inlet, outlet, adiabatic wall."""
        g = self.prm

        def cons(rho, u, v, p):
            return torch.stack([rho, rho * u, rho * v, p / (g.gamma - 1.0) + 0.5 * rho * (u * u + v * v)], 1)

        rho, u, v, p = q[:, 0], q[:, 1] / q[:, 0], q[:, 2] / q[:, 0], self._pressure(q)
        one, wn = torch.ones_like(rho), (u - ug) * nx + (v - vg) * ny
        rw = p / (g.Rgas * g.T_wall)
        free = cons(g.rho_inf * one, g.u_inf * one, g.v_inf * one, g.p_inf * one)
        out = cons(rho, u, v, g.p_inf * one)
        ghost = [cons(rw, 2 * ug - u, 2 * vg - v, p), cons(rho, u - 2 * wn * nx, v - 2 * wn * ny, p), free, out,
                 cons(rho, 2 * ug - u, 2 * vg - v, p)]
        on = [cons(rw, ug, vg, p), cons(rho, u - wn * nx, v - wn * ny, p), free, out, cons(rho, ug, vg, p)]
        pick = lambda s: sum(torch.where((self.tag == k + 1)[:, None, None], x, 0.0) for k, x in enumerate(s))  # noqa: E731
        return pick(ghost), pick(on)

    # ---- sliding interfaces (Sec. 3.2) ----
    def _mortars(self, t):
        """Per interface: mortar start angles and lengths, and per side the face of each mortar, the mapped Lagrange
        values at the quadrature points, the scale, and the faces' point angles."""
        tp = self._two_pi()
        for z, r, sides in self.ifaces:
            turn = np.longdouble(self.omega[z]) * np.longdouble(t)
            start = [(sides[0][1] + turn) % tp, sides[1][1]]
            m = np.sort(np.concatenate(start))
            dm = np.diff(np.append(m, m[0] + tp))
            res = []
            for (ef, _, width, rev), a in zip(sides, start):
                o = np.argsort(a)
                k = o[np.searchsorted(a[o], m, side="right") - 1]
                off = (m - a[k] + tp / 2) % tp - tp / 2
                x = (off / width[k])[:, None] + (dm / width[k])[:, None] * self.z_np
                H = _lagrange(self.Xs_np, x.ravel().astype(np.float64))[0].reshape(len(m), self.N, self.N)
                ang = a[:, None] + width[:, None] * self.Xs_np
                res.append((torch.as_tensor(ef.astype(np.int64), device=DEVICE), torch.as_tensor(k.astype(np.int64), device=DEVICE), _t(H),
                            _t(dm / width[k])[:, None, None], torch.as_tensor(rev.copy(), device=DEVICE)[:, None, None], _t(ang), _t(r * width)[:, None, None]))
            yield _t(m[:, None] + dm[:, None] * self.Xs_np), res

    def _couple(self, t, values, common):
        """values: per element face [4 E][K][N]; common(mortar angles, left, right) on the mortars; yields each side's
        element faces, its sum of back-projected mortar values in face order, and its sign and length."""
        for ang, res in self._mortars(t):
            side = []
            for ef, k, H, s, rev, _, _ in res:
                v = values(ef, rev)[k]
                v = torch.einsum("mqi,mvi->mvq", H, v)
                side.append(torch.einsum("pk,mvk->mvp", self.Minv, torch.einsum("q,qj,mvq->mvj", self.wq, self.Hz, v)))
            F = torch.einsum("qj,mvj->mvq", self.Hz, common(ang, *side))
            for n, (ef, k, H, s, rev, _, S) in enumerate(res):
                c = s * torch.einsum("pk,mvk->mvp", self.Minv, torch.einsum("q,mqp,mvq->mvp", self.wq, H, F))
                tot = torch.zeros((len(ef), c.shape[1], self.N), dtype=c.dtype, device=c.device).index_add_(0, k, c)
                yield ef, torch.where(rev, tot.flip(-1), tot), (1.0 - 2.0 * n) * S

    def _ends(self, fx, fy):
        """[4 E][K][N]: the end-point values of both directions' flux-point arrays, by element face."""
        return torch.stack([fy[:, :, 0], fx[..., -1], fy[:, :, -1], fx[..., 0]], 1).flatten(0, 1)

    def _with_ends(self, fx, fy, C):
        C = C.view(self.E, 4, -1, self.N)
        return (torch.cat([C[:, 3, ..., None], fx[..., 1:-1], C[:, 1, ..., None]], -1),
                torch.cat([C[:, 0, :, None], fy[:, :, 1:-1], C[:, 2, :, None]], 2))

    def _at_flux_points(self, Q):
        return torch.einsum("ik,evjk->evji", self.Hf, Q), torch.einsum("lk,evki->evli", self.Hf, Q)

    def _divide(self, fx, fy):
        return torch.einsum("ki,evji->evjk", self.Dm, fx), torch.einsum("kl,evli->evki", self.Dm, fy)

    def residual(self, Q, t):
        a, b = self._turn(self.a, t, 2), self._turn(self.b, t, 2)
        qx, qy = self._at_flux_points(Q)
        tr = self._ends(qx, qy)
        vec = self._ends(a.permute(0, 3, 1, 2), b.permute(0, 3, 1, 2))  # [4 E][2][N]
        S = torch.sqrt((vec ** 2).sum(1))
        n = self.sigma[..., None] * vec / S[:, None]
        vgn = (self.sigma * self._ends(self.ga[:, None], self.gb[:, None])[:, 0]) / S
        A, B = self.efA, self.efB
        flip = lambda v: torch.where(self.rev, v.flip(-1), v)  # noqa: E731
        fx, fy = self._flux(qx, a[..., 0], a[..., 1], self.ga), self._flux(qy, b[..., 0], b[..., 1], self.gb)
        Fn = self._rusanov(tr[A], flip(tr[B]), n[A, 0], n[A, 1], vgn[A])
        ghost = None
        if len(self.bef):
            e, nb = self.bef // 4, n[self.bef]
            pos = self._face_positions(t)
            om = _t(self.omega)[self.zone[e]][:, None]
            ghost, on = self._boundary(tr[self.bef], nb[:, 0], nb[:, 1], -om * pos[..., 1], om * pos[..., 0])
            Fb = self._rusanov(tr[self.bef], ghost, nb[:, 0], nb[:, 1], vgn[self.bef])
        values = lambda ef, rev: torch.where(rev, tr[ef].flip(-1), tr[ef])  # noqa: E731
        if self.prm.viscous:
            CQ = torch.zeros_like(tr)
            CQ[A] = 0.5 * (tr[A] + flip(tr[B]))
            CQ[B] = flip(CQ[A])
            if ghost is not None:
                CQ[self.bef] = on
            for ef, tot, _ in self._couple(t, values, lambda ang, l, r: 0.5 * (l + r)):
                CQ[ef] = tot
            dxi, deta = self._divide(*self._with_ends(qx, qy, CQ))
            m1, m2 = self._turn(self.gxi, t, 2), self._turn(self.get, t, 2)
            gx = m1[:, None, ..., 0] * dxi + m2[:, None, ..., 0] * deta
            gy = m1[:, None, ..., 1] * dxi + m2[:, None, ..., 1] * deta
            (gxx, gxy), (gyx, gyy) = self._at_flux_points(gx), self._at_flux_points(gy)
            fx = fx + self._viscous(qx, gxx, gyx, a[..., 0], a[..., 1])
            fy = fy + self._viscous(qy, gxy, gyy, b[..., 0], b[..., 1])
            tx, ty = self._ends(gxx, gxy), self._ends(gyx, gyy)
            for g1, g2 in ((tx[A], ty[A]), (flip(tx[B]), flip(ty[B]))):
                Fn = Fn + 0.5 * self._viscous(CQ[A], g1, g2, n[A, 0], n[A, 1])
            if ghost is not None:
                conduct = (self.tag != 5).to(Fb.dtype)[:, None]
                Fb = Fb + self._viscous(on, tx[self.bef], ty[self.bef], nb[:, 0], nb[:, 1], conduct)
            angles = {int(ef[0]): ang for _, res in self._mortars(t) for ef, _, _, _, _, ang, _ in res}

            def values(ef, rev):  # traces, and the viscous flux along the radial normal with the face's own gradient
                q, c, g1, g2 = (torch.where(rev, v[ef].flip(-1), v[ef]) for v in (tr, CQ, tx, ty))
                ang = angles[int(ef[0])]
                return torch.cat([q, self._viscous(c, g1, g2, torch.cos(ang), torch.sin(ang))], 1)

        def common(ang, l, r):
            F = self._rusanov(l[:, :4], r[:, :4], torch.cos(ang), torch.sin(ang), 0.0)
            return F + 0.5 * (l[:, 4:] + r[:, 4:]) if self.prm.viscous else F

        CF = torch.zeros_like(tr)
        out = (self.sigma * S)[:, None]
        CF[A] = out[A] * Fn
        CF[B] = -out[B] * flip(Fn)
        if ghost is not None:
            CF[self.bef] = out[self.bef] * Fb
        for ef, tot, length in self._couple(t, values, common):
            CF[ef] = self.sigma[ef][..., None] * length * tot
        rx, ry = self._divide(*self._with_ends(fx, fy, CF))
        return -(rx + ry) / self.J

    def _face_positions(self, t):
        """Points of the boundary faces relative to the frame centre at time t, [faces][N][2]."""
        e, f = self.bef // 4, self.bef % 4
        if not hasattr(self, "_bpos"):
            end = lambda v: np.full(self.N, v)  # noqa: E731
            s = self.Xs_np
            p = [self._map(*xe)[0] for xe in ((s, end(0.0)), (end(1.0), s), (s, end(1.0)), (end(0.0), s))]
            self._bpos = torch.stack(p, 1)[e, f]
        th = _t(self.omega * t)[self.zone[e]][:, None]
        c, sn = torch.cos(th), torch.sin(th)
        return torch.stack([c * self._bpos[..., 0] - sn * self._bpos[..., 1], sn * self._bpos[..., 0] + c * self._bpos[..., 1]], -1)

    def step(self, u, t, dt):
        L = self.residual
        if self.prm.rk_stages != 5:
            u1 = u + dt * L(u, t)
            u2 = 0.75 * u + 0.25 * (u1 + dt * L(u1, t + dt))
            return u / 3.0 + 2.0 / 3.0 * (u2 + dt * L(u2, t + 0.5 * dt))
        # SSP-RK(5,4) of Spiteri and Ruuth; stage times by the same recurrences
        c1 = 0.391752226571890
        c2 = 0.555629506348765 * c1 + 0.368410593050371
        c3 = 0.379898148511597 * c2 + 0.251891774271694
        c4 = 0.821920045606868 * c3 + 0.544974750228521
        u1 = u + c1 * dt * L(u, t)
        u2 = 0.444370493651235 * u + 0.555629506348765 * u1 + 0.368410593050371 * dt * L(u1, t + c1 * dt)
        u3 = 0.620101851488403 * u + 0.379898148511597 * u2 + 0.251891774271694 * dt * L(u2, t + c2 * dt)
        k3 = dt * L(u3, t + c3 * dt)
        u4 = 0.178079954393132 * u + 0.821920045606868 * u3 + 0.544974750228521 * k3
        return (0.517231671970585 * u2 + 0.096059710526147 * u3 + 0.063692468666290 * k3 + 0.386708617503269 * u4
                + 0.226007483236906 * dt * L(u4, t + c4 * dt))


def exact(case, seed):
    mesh, prm, dt = _problem_of(case)
    m = _Method(mesh, case["N"], prm)
    t, modes, x0, y0 = _begin(case, seed)
    xy = m.points(t)
    Q = _field(case, modes, x0, y0, xy[..., 0], xy[..., 1])
    if case["call"] == "residual":
        return m.residual(Q, t)
    for _ in range(case["steps"]):
        Q, t = m.step(Q, t, dt), t + dt
    return Q
