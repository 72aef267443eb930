"""The calls whose speed counts: right-hand sides, Runge-Kutta steps and served cases over the flows, degrees, mesh
sizes, node sets and precisions that this library is used with (the Taylor-Green, channel, shock-tube, vortex and
serving configurations of its benchmark and tests).  `listed` names them, `draw` gives others of the same ranges."""
import functools
import math

import numpy as np
import torch

from paper_2404_12703_gb300 import dg
from paper_2404_12703_gb300 import workloads as W

GAMMA, PR = 1.4, 0.72


def _case(op, flow, N, nel, precision, steps=1, curved=0.1, **kw):
    return {"op": op, "flow": flow, "N": N, "nx": nel[0], "ny": nel[1], "nz": nel[2], "precision": precision,
            "steps": steps, "curved": curved, "nodes": "lgl", "kinetic": False, **kw}


def listed():
    return [
        # one right-hand side of the smallest validation mesh: what a coupled or verifying caller asks for; launches count
        dict(_case("rhs", "tgv", 3, (4, 4, 4), "fp64"), name="rhs_tgv_4x4x4_N3_fp64"),
        # ten steps of the same mesh in single precision: the shortest time-stepping loop
        dict(_case("steps", "tgv", 3, (4, 4, 4), "fp32", 10), name="steps_tgv_4x4x4_N3_fp32"),
        # four small requests at once through the server, each to its end time: the serving form at its small end
        dict(_case("serve", "tgv", 7, (4, 4, 4), "fp64", 4), name="serve_4_requests_fp64"),
        # an inviscid run on a ragged mesh of an even degree (odd node counts)
        dict(_case("steps", "vortex", 4, (11, 10, 9), "fp32", 2, 0.05), name="steps_vortex_11x10x9_N4_fp32"),
        # a viscous run on a ragged mesh of an even degree, with the energy diagnostics of an output time
        dict(_case("steps", "tgv", 6, (9, 7, 5), "fp64", 1, kinetic=True), name="steps_tgv_9x7x5_N6_fp64_kinetic"),
        # the compressible vortex: Sutherland's law, shock indicator and blending
        dict(_case("steps", "compressible", 7, (8, 8, 8), "fp32", 1, 0.0), name="steps_compressible_8x8x8_N7_fp32"),
        # the shock tube at its full size, where the blending works
        dict(_case("steps", "sod", 5, (64, 8, 8), "fp64", 1, 0.0), name="steps_sod_64x8x8_N5_fp64"),
        # a wall-bounded channel: boundary conditions, single precision
        dict(_case("steps", "channel", 7, (16, 8, 16), "fp32", 2), name="steps_channel_16x8x16_N7_fp32"),
        # the standard scheme on Gauss-Legendre nodes
        dict(_case("steps", "tgv", 7, (12, 12, 12), "fp64", 1, nodes="gauss"), name="steps_gauss_12x12x12_N7_fp64"),
        # the long validation run: 7 million unknowns of degree 5, single precision
        dict(_case("steps", "tgv", 5, (32, 32, 32), "fp32", 2, 0.0), name="steps_tgv_32x32x32_N5_fp32"),
        # the benchmark mesh (curved, renumbered, rotated, degree 7) in both precisions
        dict(_case("steps", "tgv", 7, (24, 24, 24), "fp32", 2), name="steps_tgv_24x24x24_N7_fp32"),
        dict(_case("steps", "tgv", 7, (24, 24, 24), "fp64", 1), name="steps_tgv_24x24x24_N7_fp64"),
    ]


def draw(rng):
    op = rng.choices(("rhs", "steps", "serve"), (2, 8, 1))[0]
    flow = rng.choices(("tgv", "vortex", "compressible", "sod", "channel"), (5, 2, 1, 1, 1))[0]
    precision = "fp64" if op == "rhs" else rng.choice(("fp32", "fp64"))
    N = rng.choices((1, 2, 3, 4, 5, 6, 7), (1, 2, 3, 2, 4, 2, 5))[0]
    if op == "serve":
        nel = tuple(rng.randint(3, 6) for _ in range(3))
        return _case("serve", "tgv", rng.choice((3, 5, 7)), nel, "fp64", rng.randint(2, 6))
    # sizes spread over the logarithm of the node count, from 4^3 elements of degree 3 to a sixth of the largest
    nodes = math.exp(rng.uniform(math.log(4096.0), math.log(1.2e6)))
    m = max(3.0, (nodes / (N + 1) ** 3) ** (1.0 / 3.0))
    nel = tuple(max(3, int(round(m * rng.uniform(0.75, 1.3)))) for _ in range(3))
    gauss = flow == "tgv" and rng.random() < 0.25
    steps = rng.randint(1, 2)
    return _case(op, flow, N, nel, precision, 1 if op == "rhs" else steps,
                 0.0 if flow in ("sod", "compressible") else rng.choice((0.0, 0.05, 0.1)),
                 nodes="gauss" if gauss else "lgl", kinetic=precision == "fp64" and op == "steps" and rng.random() < 0.3)


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
BOX = {"tgv": (2 * math.pi,) * 3, "compressible": (2 * math.pi,) * 3, "vortex": (10.0,) * 3, "sod": (2.0, 0.25, 0.25),
       "channel": (4.0, 1.0, 4.0)}
MU = {"tgv": 1.0 / 1600.0, "compressible": 1.0 / 1600.0, "vortex": 0.0, "sod": 0.0, "channel": 1e-3}
MACH = {"tgv": 0.1, "compressible": 1.25}
WALLS = [(1, 0.0, 0.0, 0.0, 1.0), (1, 1.0, 0.0, 0.0, 1.0)]  # isothermal, at rest and moving
T_END = 0.02  # of a served request


@functools.lru_cache(maxsize=2)
def _mesh(flow, N, nel, curved):
    """A user's mesh file: nodes and corner ids, renumbered and rotated where the mesh is curved."""
    m = W.box_mesh(N, nel, length=BOX[flow], curved=curved, seed=20240419 if curved else None,
                   periodic=(True, flow != "channel", True))
    if flow == "channel":
        m["face_bc"] = W.box_face_bc(m, {"y-": 1, "y+": 2})
        m["bcs"] = WALLS
    return m


def _mesh_of(case):
    return _mesh(case["flow"], case["N"], (case["nx"], case["ny"], case["nz"]), case["curved"])


def _flow_state(flow, X, seed):
    """The flow at the points X [..., 3], shifted by the seed."""
    rng = np.random.Generator(np.random.PCG64(seed))
    L = np.array(BOX[flow])
    if flow in MACH:
        return W.tgv_state(X + rng.uniform(0.0, 1.0, 3) * L, Ma=MACH[flow])
    if flow == "vortex":
        return W.isentropic_vortex_state(X, center=rng.uniform(0.0, 1.0, 2) * L[:2], period=L)
    if flow == "sod":
        return W.sod_state(X, x_split=rng.uniform(0.8, 1.2))
    U = W.couette_state(X, U_wall=1.0, T_wall=1.0, p=10.0, mu=MU[flow])
    return W.random_perturbation(U, 1e-3, int(rng.integers(1 << 30)))


def _fixed_dt(case):
    """Single-precision runs step with a fixed time step well inside the stability limit (as the long runs do); double
    precision takes the library's own rule, dt = 0."""
    if case["precision"] == "fp64":
        return 0.0
    h = min(l / m for l, m in zip(BOX[case["flow"]], (case["nx"], case["ny"], case["nz"])))
    speed = 1.0 + {"tgv": 10.0, "compressible": 1.0, "vortex": 2.0, "sod": 2.0, "channel": 4.0}[case["flow"]]
    return 0.2 * h / (speed * (case["N"] + 1) ** 2)


def _settings(case):
    flow = case["flow"]
    kw = {"mu": MU[flow], "viscous": int(MU[flow] > 0), "precision": case["precision"]}
    if flow == "compressible":
        kw.update(sutherland=1, T_ref=1.0 / (GAMMA * MACH[flow] ** 2), shock_capturing=int(case["nodes"] == "lgl"))
    if flow == "sod":
        kw.update(riemann="lf", shock_capturing=1)
    return kw


def _requests(case, seed):
    """The requests of a served case: the given mesh and smaller ones of other degrees, each with its state."""
    out = []
    for k, (N, nel) in enumerate(_request_sizes(case)):
        m = _request_mesh(N, nel)
        out.append((m, _flow_state("tgv", m["xyz"], 1000 * seed + k).reshape(m["E"], -1, 5)))
    return out


def _request_sizes(case):
    return [(case["N"], (case["nx"], case["ny"], case["nz"])) if k == 0 else ((case["N"], 3, 5)[k % 3], (3 + k % 2,) * 3)
            for k in range(case["steps"])]


@functools.lru_cache(maxsize=8)
def _request_mesh(N, nel):
    return W.box_mesh(N, nel, curved=0.1, seed=1000 + nel[0])


def prepare(case, seed):
    if case["op"] == "serve":
        pool = sum(a * b * c for _, (a, b, c) in _request_sizes(case))
        server = dg.Server(pool_elems={3: pool, 5: pool, 7: pool}, max_cases=16)
        return {"op": "serve", "server": server, "requests": _requests(case, seed)}
    m = _mesh_of(case)
    solver = dg.Solver(m, nodes=case["nodes"], **_settings(case))
    X = solver.node_coords() if case["nodes"] == "gauss" else m["xyz"]
    U = torch.from_numpy(np.ascontiguousarray(_flow_state(case["flow"], X, seed).reshape(m["E"], -1, 5))).cuda()
    return {"op": case["op"], "solver": solver, "U": U, "out": torch.empty_like(U), "steps": case["steps"],
            "dt": _fixed_dt(case), "kinetic": case["kinetic"]}


def run(state):
    if state["op"] == "serve":  # submit every request, then collect the results
        server = state["server"]
        tickets = [server.submit(m, U, T_END, mu=MU["tgv"]) for m, U in state["requests"]]
        return [server.wait(t)[0] for t in tickets]
    s = state["solver"]
    if state["op"] == "rhs":
        return s.rhs(state["U"], out=state["out"])
    s.set_state(state["U"])
    s.step(state["steps"], state["dt"])
    U, t = s.get_state(out=state["out"])
    return {"U": U, "t": t, "kinetic": np.array(s.kinetic())} if state["kinetic"] else {"U": U, "t": t}


def work(case):
    """Per stage and node: the state and the Runge-Kutta register in and out, the ten metric terms, the side normals; the
    two-point fluxes of every pair of a line, the derivative sums of the lifting and of the viscous term."""
    n = case["N"] + 1
    word = 8 if case["precision"] == "fp64" else 4
    viscous = MU[case["flow"]] > 0
    if case["op"] == "serve":
        stages = 5 * 10  # about ten steps each on average
        count = sum(a * b * c * (N + 1) ** 3 for N, (a, b, c) in _request_sizes(case))
    else:
        count, stages = case["nx"] * case["ny"] * case["nz"] * n ** 3, 1 if case["op"] == "rhs" else 5 * case["steps"]
    per_stage = 80 + (10 + 10 + 12 / n) * word if case["op"] != "rhs" else 80 + (10 + 12 / n) * word
    flux = 54 if case["nodes"] == "lgl" else 0
    flops = 1.5 * (n - 1) * flux + (0 if flux else 30 * n + 45) + 3 * 5 * 4 + 6 * 150 / n
    if viscous:
        flops += 72 * n + 36 + 24 * n + 100
    return {"bytes": count * per_stage * stages, "flops": count * flops * stages}


# ---------------------------------------------------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------------------------------------------------
RK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
RK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0, 1720146321549.0 / 2090206949498.0,
        3134564353537.0 / 4481467310338.0, 2277821191437.0 / 14882151754819.0)


def _lagrange(x, y):
    """Row r: the Lagrange polynomials of the nodes x at y[r]."""
    return np.array([[np.prod([(b - x[m]) / (x[j] - x[m]) for m in range(len(x)) if m != j]) for j in range(len(x))]
                     for b in y])


def _derivative(x):
    n = len(x)
    w = np.array([1.0 / np.prod([x[j] - x[m] for m in range(n) if m != j]) for j in range(n)])
    D = np.array([[w[j] / w[i] / (x[i] - x[j]) if i != j else 0.0 for j in range(n)] for i in range(n)])
    return D - np.diag(D.sum(axis=1))


class _Exact:
    """The discontinuous Galerkin operator on one mesh, fields as [component][element, k, j, i]."""

    def __init__(self, case, mesh):
        self.case, self.n, self.E = case, case["N"] + 1, mesh["E"]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.gauss, self.N = case["nodes"] == "gauss", case["N"]
        n, E, N = self.n, self.E, self.N
        lgl = W.lgl_points(N)
        lw = 2.0 / (N * n * np.polynomial.legendre.legval(lgl, [0] * N + [1]) ** 2)
        x, w = np.polynomial.legendre.leggauss(n) if self.gauss else (lgl, lw)
        D = _derivative(x)
        ends = _lagrange(x, [-1.0, 1.0])
        if not self.gauss:
            ends = np.eye(n)[[0, -1]]
        self.w, self.D = self._t(w), self._t(D)
        self.Dhat = self._t(-(w[None, :] * D.T) / w[:, None])
        self.ends, self.lhat = self._t(ends), self._t(ends / w)
        split = 2 * D
        split[0, 0] += 1 / w[0]
        split[-1, -1] -= 1 / w[-1]
        self.split = split
        V = np.array([[math.sqrt(k + 0.5) * np.polynomial.legendre.legval(a, [0] * k + [1]) for k in range(n)] for a in x])
        self.Vinv = self._t(np.linalg.inv(V))
        # curl-form metrics at the LGL nodes, relative to each element's first node
        X = self._t(mesh["xyz"]).reshape(E, n, n, n, 3)
        X = [X[..., c] - X[:, :1, :1, :1, c] for c in range(3)]
        Dl = self._t(_derivative(lgl))
        dx = [[self._along(Dl, X[c], d) for d in range(3)] for c in range(3)]
        Ja = [[None] * 3 for _ in range(3)]
        for c in range(3):
            m, l = (c + 1) % 3, (c + 2) % 3
            V = [X[l] * dx[m][d] for d in range(3)]
            for i in range(3):
                a, b = (i + 1) % 3, (i + 2) % 3
                Ja[i][c] = self._along(Dl, V[a], b) - self._along(Dl, V[b], a)
        if self.gauss:
            to = self._t(_lagrange(lgl, x))
            put = lambda f: self._along(to, self._along(to, self._along(to, f, 0), 1), 2)  # noqa: E731
            Ja = [[put(f) for f in r] for r in Ja]
            dx = [[put(f) for f in r] for r in dx]
        self.Ja = Ja
        self.J = (dx[0][0] * (dx[1][1] * dx[2][2] - dx[1][2] * dx[2][1])
                  - dx[0][1] * (dx[1][0] * dx[2][2] - dx[1][2] * dx[2][0])
                  + dx[0][2] * (dx[1][0] * dx[2][1] - dx[1][1] * dx[2][0]))
        # outward scaled normals [3][E, 6, n^2], and the partner of every face point
        self.nv = [torch.stack([(2 * s - 1) * self._face(Ja[d][c], d, s) for d in range(3) for s in (0, 1)], 1)
                   for c in range(3)]
        self.area = torch.sqrt(sum(v * v for v in self.nv))
        self.nu = [v / self.area for v in self.nv]
        self.partner, bc = self._partners(mesh)
        self.wall = None if bc is None else torch.from_numpy(bc.astype(np.int64)).to(self.dev)
        self.mu = MU[case["flow"]]
        self.sutherland = case["flow"] == "compressible"
        self.shock = not self.gauss and case["flow"] in ("compressible", "sod")
        self.T_ref = 1.0 / (GAMMA * MACH["compressible"] ** 2)

    def _t(self, a):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)

    def _along(self, M, f, d):
        """The matrix M applied along local direction d."""
        return torch.movedim(torch.movedim(f, -1 - d, -1) @ M.T, -1, -1 - d)

    def _face(self, f, d, s):
        return torch.tensordot(f, self.ends[s], dims=([f.dim() - 1 - d], [0])).reshape(f.shape[0], -1)

    def _faces(self, f):
        return torch.stack([self._face(f, d, s) for d in range(3) for s in (0, 1)], 1)

    def _spread(self, acc, val):
        """Adds the face values val [E, 6, n^2] to the nodes with l(+-1) / w."""
        n = self.n
        for d in range(3):
            shape = [1, 1, 1, 1]
            shape[3 - d] = n
            for s in (0, 1):
                acc += val[:, 2 * d + s].reshape(-1, n, n).unsqueeze(3 - d) * self.lhat[s].reshape(shape)

    def _partners(self, mesh):
        """Flat index [E, 6, n^2] of the face point opposite each one, from the corner ids (itself at a wall)."""
        n, E = self.n, self.E
        q, p = np.divmod(np.arange(n * n), n)
        ids = np.empty((E, 6, 4), dtype=np.int64)
        for d in range(3):
            a, b = [x for x in range(3) if x != d]
            for s in (0, 1):
                for k, (cp, cq) in enumerate(((0, 0), (1, 0), (0, 1), (1, 1))):
                    ids[:, 2 * d + s, k] = mesh["corner_vid"][:, s * (1 << d) + cp * (1 << a) + cq * (1 << b)]
        flat = ids.reshape(-1, 4)
        key = np.sort(flat, axis=1)
        order = np.lexsort(key.T)
        same = (key[order][1:] == key[order][:-1]).all(axis=1)
        other = np.arange(E * 6)
        i = np.nonzero(same)[0]
        other[order[i]], other[order[i + 1]] = order[i + 1], order[i]
        out = np.repeat(np.arange(E * 6)[:, None] * n * n, n * n, 1) + np.arange(n * n)
        for t in range(8):  # the face frame of the partner: swapped, then reversed
            turn = lambda a, b, m: [(m - v if t >> k & 1 else v) for k, v in enumerate((b, a) if t & 4 else (a, b))]  # noqa: E731
            c = [x + 2 * y for x, y in (turn(cp, cq, 1) for cp, cq in ((0, 0), (1, 0), (0, 1), (1, 1)))]
            fit = (flat == flat[other][:, c]).all(axis=1) & (other != np.arange(E * 6))
            pm, qm = turn(p, q, n - 1)
            out[fit] = other[fit][:, None] * n * n + (pm + n * qm)
        bc = mesh.get("face_bc")
        return torch.from_numpy(out.reshape(E, 6, n * n)).to(self.dev), bc

    @staticmethod
    def _prims(U):
        u = [U[c] / U[0] for c in (1, 2, 3)]
        p = (GAMMA - 1) * (U[4] - 0.5 * (U[1] * u[0] + U[2] * u[1] + U[3] * u[2]))
        return U[0], u[0], u[1], u[2], p, (U[4] + p) / U[0], p / U[0]  # rho, u, v, w, p, H, T

    def _viscosity(self, T):
        if not self.sutherland:
            return self.mu
        th = T / self.T_ref
        return self.mu * 1.4042 * th * torch.sqrt(th) / (th + 0.4042)

    def _viscous(self, u, T, g, nv):
        """F_v . nv of the velocity u, temperature T and gradients g[4][3]."""
        mu = self._viscosity(T)
        lam = GAMMA * mu / ((GAMMA - 1) * PR)
        div = g[0][0] + g[1][1] + g[2][2]
        tau = [[mu * (g[a][b] + g[b][a]) - (mu * (2.0 / 3.0) * div if a == b else 0.0) for b in range(3)] for a in range(3)]
        f = [sum(tau[a][b] * nv[b] for b in range(3)) for a in range(3)]
        heat = [sum(tau[b][a] * u[a] for a in range(3)) + lam * g[3][b] for b in range(3)]
        return f + [sum(heat[b] * nv[b] for b in range(3))]

    @staticmethod
    def _euler(q, nv):
        m = q[0] * sum(q[1 + c] * nv[c] for c in range(3))
        return [m] + [m * q[1 + c] + q[4] * nv[c] for c in range(3)] + [m * q[5]]

    def _riemann(self, L, R, UL, UR, nu):
        fL, fR = self._euler(L, nu), self._euler(R, nu)
        if self.case["flow"] == "sod":
            return self._rusanov(L, R, UL, UR, fL, fR, nu)
        a, b = torch.sqrt(L[0]), torch.sqrt(R[0])
        u = [(a * L[1 + c] + b * R[1 + c]) / (a + b) for c in range(3)]
        H = (a * L[5] + b * R[5]) / (a + b)
        q2 = sum(v * v for v in u)
        c2 = (GAMMA - 1) * (H - q2 / 2)
        c, un = torch.sqrt(c2), sum(u[k] * nu[k] for k in range(3))
        dr, dp, du = R[0] - L[0], R[4] - L[4], [R[1 + k] - L[1 + k] for k in range(3)]
        dun = sum(du[k] * nu[k] for k in range(3))
        a1, a2, a5 = (dp - a * b * c * dun) / (2 * c2), dr - dp / c2, (dp + a * b * c * dun) / (2 * c2)
        w1, w5, w2 = (un - c).abs() * a1, (un + c).abs() * a5, un.abs()
        sh = [w2 * a * b * (du[k] - dun * nu[k]) for k in range(3)]
        D = [w1 + w2 * a2 + w5]
        D += [w1 * (u[k] - c * nu[k]) + w2 * a2 * u[k] + w5 * (u[k] + c * nu[k]) + sh[k] for k in range(3)]
        D += [w1 * (H - un * c) + w2 * a2 * q2 / 2 + w5 * (H + un * c) + sum(u[k] * sh[k] for k in range(3))]
        return [(fL[k] + fR[k] - D[k]) / 2 for k in range(5)]

    @staticmethod
    def _rusanov(L, R, UL, UR, fL, fR, nu):
        s = [sum(q[1 + c] * nu[c] for c in range(3)).abs() + torch.sqrt(GAMMA * q[4] / q[0]) for q in (L, R)]
        lm = torch.maximum(*s)
        return [(fL[k] + fR[k] - lm * (UR[k] - UL[k])) / 2 for k in range(5)]

    def _blend(self, U, q, conv):
        """The shock indicator and the blend of conv with first-order sub-cell fluxes."""
        n, N = self.n, self.N
        m = q[0] * q[4]
        for d in range(3):
            m = self._along(self.Vinv, m, d)
        i = torch.arange(n, device=self.dev)
        deg = torch.maximum(torch.maximum(i[None, None, :], i[None, :, None]), i[:, None, None])
        part = [(m * m * (deg == k)).sum(dim=(1, 2, 3)) for k in range(n)]
        tot, tot1 = sum(part), sum(part[:-1])
        ratio = torch.maximum(part[N] / tot, part[N - 1] / tot1)
        T, sharp = 0.5 * 10.0 ** (-1.8 * (N + 1) ** 0.25), math.log((1 - 1e-4) / 1e-4)
        al = 1.0 / (1.0 + torch.exp(-sharp * (ratio - T) / T))
        al = torch.where(al < 1e-3, 0.0, al).clamp(max=0.5)[:, None, None, None]
        fv = [torch.zeros_like(U[0]) for _ in range(5)]
        for d in range(3):
            ax = 3 - d
            shape = [1, 1, 1, 1]
            shape[ax] = n
            wd = self.w.reshape(shape)
            lo, hi = (lambda f: f.narrow(ax, 0, n - 1)), (lambda f: f.narrow(ax, 1, n - 1))
            mv = [f.narrow(ax, 0, 1) + lo(torch.cumsum(wd * self._along(self.D, f, d), ax)) for f in self.Ja[d]]
            s = torch.sqrt(sum(v * v for v in mv))
            nu = [v / s for v in mv]
            L, R = [lo(f) for f in q], [hi(f) for f in q]
            f = self._rusanov(L, R, [lo(f) for f in U], [hi(f) for f in U], self._euler(L, nu), self._euler(R, nu), nu)
            for k in range(5):
                lo(fv[k]).add_(f[k] * s / lo(wd))
                hi(fv[k]).sub_(f[k] * s / hi(wd))
        return [(1 - al) * conv[k] + al * fv[k] for k in range(5)]

    def rhs(self, U):
        n = self.n
        q = self._prims(U)
        Uf = [self._faces(f) for f in U]
        L = self._prims(Uf)
        UR = [f.reshape(-1)[self.partner] for f in Uf]
        R = self._prims(UR)
        wall = None if self.wall is None else (self.wall > 0)[:, :, None]
        uw = None if wall is None else [torch.where(self.wall == 2, WALLS[1][1 + c], WALLS[0][1 + c])[:, :, None].double() for c in range(3)]
        conv = [torch.zeros_like(U[0]) for _ in range(5)]
        rest = [torch.zeros_like(U[0]) for _ in range(5)]
        for d in range(3):
            Ja, ax = self.Ja[d], 3 - d
            if self.gauss:
                for k, f in enumerate(self._euler(q, Ja)):
                    conv[k] += self._along(self.Dhat, f, d)
                continue
            for a in range(n):
                shape = [1, 1, 1, 1]
                shape[ax] = n
                c = self._t(self.split[:, a]).reshape(shape)
                mean = lambda f: (f + f.narrow(ax, a, 1)) / 2  # noqa: E731
                nv, (r, u, v, w, p, H) = [mean(f) for f in Ja], [mean(f) for f in q[:6]]
                m = r * (u * nv[0] + v * nv[1] + w * nv[2])
                for k, f in enumerate((m, m * u + p * nv[0], m * v + p * nv[1], m * w + p * nv[2], m * H)):
                    conv[k] += c * f
        if self.shock:
            conv = self._blend(U, q, conv)
        f = self._riemann(L, R, Uf, UR, self.nu)
        f = [v * self.area for v in f]
        if wall is not None:
            un = sum(uw[c] * self.nv[c] for c in range(3))
            solid = [0.0 * un] + [L[4] * self.nv[c] for c in range(3)] + [L[4] * un]
            f = [torch.where(wall, a, b) for a, b in zip(solid, f)]
        if self.mu > 0:
            g = [[None] * 3 for _ in range(4)]
            for k, v in enumerate((1, 2, 3, 6)):
                qs = (L[v] + R[v]) / 2
                if wall is not None:
                    qs = torch.where(wall, uw[k] if k < 3 else torch.ones_like(qs), qs)
                for x in range(3):
                    acc = sum(self._along(self.Dhat, self.Ja[d][x] * q[v], d) for d in range(3))
                    self._spread(acc, qs * self.nv[x])
                    g[k][x] = acc / self.J
            for d in range(3):
                for k, v in enumerate(self._viscous(q[1:4], q[6], g, self.Ja[d])):
                    rest[1 + k] -= self._along(self.Dhat, v, d)
            gL = [[self._faces(v) for v in r] for r in g]
            gR = [[v.reshape(-1)[self.partner] for v in r] for r in gL]
            a, b = self._viscous(L[1:4], L[6], gL, self.nv), self._viscous(R[1:4], R[6], gR, self.nv)
            fv = [(x + y) / 2 for x, y in zip(a, b)]
            if wall is not None:
                fw = self._viscous(uw, torch.ones_like(L[6]), gL, self.nv)
                fv = [torch.where(wall, x, y) for x, y in zip(fw, fv)]
            f = [f[0]] + [f[1 + k] - fv[k] for k in range(4)]
        for k in range(5):
            self._spread(rest[k], f[k])
        return [-(conv[k] + rest[k]) / self.J for k in range(5)]

    def time_step(self, U):
        rho, u, v, w, p, _, T = self._prims(U)
        c, a, b = torch.sqrt(GAMMA * p / rho), 0.0, 0.0
        for Ja in self.Ja:
            j2 = sum(f * f for f in Ja)
            a = a + (u * Ja[0] + v * Ja[1] + w * Ja[2]).abs() + c * torch.sqrt(j2)
            b = b + j2
        dt = 0.9 * 2 / (self.n ** 2 * float((a / self.J).max()))
        if self.mu > 0:
            lv = float((max(4 / 3, GAMMA / PR) * self._viscosity(T) / rho * b / self.J ** 2).max())
            dt = min(dt, 0.9 * 4 / (self.n ** 4 * lv))
        return dt

    def steps(self, U, count, dt0, t_end=math.inf):
        t, dU = 0.0, [torch.zeros_like(f) for f in U]
        while count and t < t_end:
            count -= 1
            dt = dt0 if dt0 > 0 else self.time_step(U)
            t, dt = (t_end, t_end - t) if t + dt >= t_end else (t + dt, dt)
            for A, B in zip(RK_A, RK_B):
                R = self.rhs(U)
                dU = [A * x + dt * r for x, r in zip(dU, R)]
                U = [x + B * y for x, y in zip(U, dU)]
        return U, t

    def fields(self, U):
        return [self._t(U).reshape(self.E, self.n, self.n, self.n, 5)[..., k].contiguous() for k in range(5)]

    def public(self, U):
        return torch.stack(U, -1).reshape(self.E, -1, 5)

    def kinetic(self, U):
        R = self.rhs(U)
        wq = self.w[:, None, None] * self.w[:, None] * self.w * self.J
        u = [U[c] / U[0] for c in (1, 2, 3)]
        v2, vol = sum(v * v for v in u), wq.sum()
        rate = wq * (sum(u[c] * R[1 + c] for c in range(3)) - v2 * R[0] / 2)
        return torch.stack([(wq * U[0] * v2 / 2).sum() / vol, rate.sum() / vol, vol])


def exact(case, seed):
    if case["op"] == "serve":
        out = []
        for m, U in _requests(case, seed):
            ex = _Exact(dict(case, N=m["N"]), m)
            out.append(ex.public(ex.steps(ex.fields(U), 1 << 20, 0.0, T_END)[0]).cpu().numpy())
        return out
    m = _mesh_of(case)
    ex = _Exact(case, m)
    X = m["xyz"]
    if ex.gauss:
        to = ex._t(_lagrange(W.lgl_points(ex.N), np.polynomial.legendre.leggauss(ex.n)[0]))
        X = ex._t(X)
        X = torch.stack([ex._along(to, ex._along(to, ex._along(to, X[..., c], 0), 1), 2) for c in range(3)], -1).cpu().numpy()
    U = ex.fields(_flow_state(case["flow"], X, seed))
    if case["op"] == "rhs":
        return ex.public(ex.rhs(U))
    U, t = ex.steps(U, case["steps"], _fixed_dt(case))
    out = {"U": ex.public(U), "t": t}
    return dict(out, kinetic=ex.kinetic(U)) if case["kinetic"] else out
