"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``op`` is the call: "step" advances a handle's state by
LSRK(5,4) steps (``Solver.step``), "rhs" evaluates one right-hand side (``Solver.rhs``, what a
program with its own time integrator calls), "slabs" steps a mesh cut into slabs
(``PartitionedSolver``), "monitor" evaluates the time-step bound and the conserved integrals
(``Solver.cfl_dt``, ``Solver.integrals``), "server" sends a batch of requests to the
continuous-batching server and waits for the final states.  ``flow`` is the set-up: "bubble" and
"sharp" (smooth and sharp rising bubble in a box with walls in z), "channel" (stratified rotating
channel, the background at rest in mixed precision) and "jet" (the same with the jet as a moving
background).

Every stepping pass starts from the state that the program holds on the device, so a pass can be
repeated and always does the same work.
"""
import math
import random

import numpy as np
import torch

from paper_2605_16684_gb300 import _lib

GAMMA, GRAV, RGAS, P0 = 1.4, 9.81, 287.0, 1.0e5
RK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
RK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
        1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
        2277821191437.0 / 14882151754819.0)


# ---- the cases ---------------------------------------------------------------
def _c(name, op, flow, precision, K, N, steps, warp=0.0, **more):
    return dict(name=name, op=op, flow=flow, precision=precision, kx=K[0], ky=K[1], kz=K[2], N=N,
                steps=steps, warp=warp, **more)


def listed():
    return [
        # the smallest run of the tests and of the smoke check: a 4^3 box, where launches count
        _c("fp64_bubble_4_n3", "step", "bubble", "fp64", (4, 4, 4), 3, 1),
        # the smallest member of an ensemble, solved by itself in mixed precision
        _c("mixed_bubble_8_n4", "step", "bubble", "mixed", (8, 8, 8), 4, 1),
        # the benchmark's headline: the warped 32^3 box at N = 4 in FP64 ...
        _c("fp64_bubble_32_n4", "step", "bubble", "fp64", (32, 32, 32), 4, 2, 0.05),
        # ... and in mixed precision
        _c("mixed_bubble_32_n4", "step", "bubble", "mixed", (32, 32, 32), 4, 4, 0.05),
        # a ragged box at an even number of nodes, called by a program with its own integrator
        _c("fp64_rhs_13x9x7_n5", "rhs", "bubble", "fp64", (13, 9, 7), 5, 1, 0.05),
        # high order: FP64 and mixed
        _c("fp64_bubble_12_n7", "step", "bubble", "fp64", (12, 12, 12), 7, 1, 0.05),
        _c("mixed_bubble_16_n7", "step", "bubble", "mixed", (16, 16, 16), 7, 2),
        # the serving workload's channel (scale 2) on its resting background, every vertical
        # pair on the logarithm branch, with rotation
        _c("mixed_channel_80x16x8_n3", "step", "channel", "mixed", (80, 16, 8), 3, 2),
        # the channel benchmark with its jet carried as a moving background
        _c("mixed_jet_120x24x12_n4", "step", "jet", "mixed", (120, 24, 12), 4, 1),
        # the largest: the sharp bubble on the 64^3 box (32.8 million nodes)
        _c("mixed_sharp_64_n4", "step", "sharp", "mixed", (64, 64, 64), 4, 2),
        # a batch of served requests: eight bubbles of mixed sizes and orders
        _c("server_mixed_8", "server", "bubble", "mixed", (8, 8, 8), 4, 20, members=8, kmax=20,
           mix=1),
        # the monitors of a long run: time-step bound, mass, energy and entropy
        _c("monitor_32_n4", "monitor", "bubble", "fp64", (32, 32, 32), 4, 1, 0.05),
    ]


def _box(rng, elems):
    """Three counts with a product near elems, of uneven sides, odd ones among them."""
    side = elems ** (1.0 / 3.0)
    k = [max(1, int(round(side * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(3)]
    return tuple(k)


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp64", "mixed", "mixed", "rhs", "channel", "channel64",
                       "jet", "slabs", "server", "monitor"])
    N = rng.choice([1, 2, 3, 3, 4, 4, 4, 5, 6, 7, 7])
    # nodes from the smallest test meshes to the benchmark's, evenly in their logarithm
    most = {"fp64": 3.0e6, "rhs": 3.0e6, "channel64": 2.0e6}.get(kind, 4.0e6)
    nodes = math.exp(rng.uniform(math.log(2.0e3), math.log(most)))
    K = _box(rng, nodes / (N + 1) ** 3)
    warp = rng.choice([0.0, 0.05])
    steps = rng.choice([1, 2])
    if kind in ("channel", "channel64", "jet"):
        s = max(0.1, min(3.0, (nodes / (N + 1) ** 3 / 1280.0) ** (1.0 / 3.0)))
        K = tuple(max(1, int(round(k * s * math.exp(rng.uniform(-0.1, 0.1))))) for k in (40, 8, 4))
        flow = "jet" if kind == "jet" else "channel"
        return _d("step", flow, "fp64" if kind == "channel64" else "mixed", K, N, steps)
    if kind == "server":
        return _d("server", "bubble", "mixed", (8, 8, 8), 4, rng.randint(5, 20),
                  members=rng.randint(3, 8), kmax=rng.randint(10, 20), mix=rng.randint(2, 10 ** 6))
    if kind == "slabs":
        K = (max(4, K[0]), K[1], K[2])
        return _d("slabs", "bubble", rng.choice(["fp64", "mixed"]), K, min(N, 4), steps, warp,
                  slabs=rng.randint(2, 4))
    if kind == "monitor":
        return _d("monitor", "bubble", "fp64", K, N, 1, warp)
    if kind == "rhs":
        return _d("rhs", "bubble", rng.choice(["fp64", "fp64", "mixed"]), K, N, 1, warp)
    return _d("step", rng.choice(["bubble", "bubble", "sharp"]), kind, K, N, steps, warp)


def _d(*a, **more):
    c = _c("", *a, **more)
    del c["name"]
    return c


def _members(case):
    """(K, N) of a served batch's requests: cubes of 8 .. kmax elements, N = 3, 4 or 7."""
    r = random.Random(case["mix"])
    return [(r.randint(8, case["kmax"]), r.choice((3, 4, 7))) for _ in range(case["members"])]


# ---- meshes and states -------------------------------------------------------
def _rotating(case):
    return case["flow"] in ("channel", "jet")


def _mesh(case):
    if _rotating(case):
        return dict(lo=(0.0, 0.0, 0.0), hi=(40000e3, 6000e3, 30e3), periodic=(1, 0, 0))
    if case["flow"] == "sharp":
        return dict(lo=(-1000.0, -1000.0, 0.0), hi=(1000.0, 1000.0, 2000.0), periodic=(1, 1, 0))
    return dict(lo=(0.0, 0.0, 0.0), hi=(1000.0, 1000.0, 1000.0), periodic=(1, 1, 0))


def _lgl(N):
    """LGL points, weights and the differentiation matrix."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # Newton on P'_N for the interior points
        if N > 1:
            x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    dx = x[:, None] - x[None, :] + np.eye(N + 1)
    b = 1.0 / dx.prod(axis=1)
    D = b[None, :] / b[:, None] / dx
    D -= np.diag(np.diag(D))
    D -= np.diag(D.sum(axis=1))
    return x, w, D


def _nodes(case, dev="cuda"):
    """Node coordinates [E][3][np] in 64 bits: uniform boxes, then the smooth warp."""
    m, K, N = _mesh(case), (case["kx"], case["ky"], case["kz"]), case["N"]
    xi = torch.tensor(_lgl(N)[0], device=dev)
    r = []
    for d in range(3):
        L = m["hi"][d] - m["lo"][d]
        e = torch.arange(K[d], device=dev, dtype=torch.float64)
        r.append(L * (e[:, None] + 0.5 * (1.0 + xi[None, :])) / K[d])
    X = r[0].view(1, 1, K[0], 1, 1, -1)
    Y = r[1].view(1, K[1], 1, 1, -1, 1)
    Z = r[2].view(K[2], 1, 1, -1, 1, 1)
    L = [m["hi"][d] - m["lo"][d] for d in range(3)]
    s = [torch.sin(2 * math.pi * v / l) for v, l in zip((X, Y, Z), L)]
    w = case["warp"]
    c = [X + w * L[0] * s[1] * s[2], Y + w * L[1] * s[2] * s[0], Z + w * L[2] * s[0] * s[1]]
    shape = (K[2], K[1], K[0], N + 1, N + 1, N + 1)
    E = K[0] * K[1] * K[2]
    return torch.stack([(v + m["lo"][d]).expand(shape).reshape(E, -1) for d, v in enumerate(c)], 1)


def _phys(case):
    return dict(f0=1.0e-4) if _rotating(case) else {}


def _state(case, seed, x):
    """A developed flow: the set-up's stratification with a seeded bubble or wind perturbation
    and smooth winds of a few metres per second (sums of random Fourier modes)."""
    rng = random.Random(seed)
    m = _mesh(case)
    X, Y, Z = x[:, 0], x[:, 1], x[:, 2]
    xs = [(x[:, d] - m["lo"][d]) / (m["hi"][d] - m["lo"][d]) for d in range(3)]

    def modes(z_even):
        f = torch.zeros_like(X)
        for _ in range(3):
            kx, ky, kz = rng.randint(1, 3), rng.randint(1, 3), rng.randint(1, 3)
            ph = rng.uniform(0.0, 2.0 * math.pi)
            f += rng.uniform(0.5, 1.0) * torch.sin(2 * math.pi * (kx * xs[0] + ky * xs[1]) + ph) * (
                torch.cos(math.pi * kz * xs[2]) if z_even else torch.sin(math.pi * kz * xs[2]))
        return f / 3.0

    if _rotating(case):
        th = torch.tanh((Y - 3.0e6) / 6.0e5)
        H = 7500.0 + 60.0 * (1.0 - th)
        dH = -60.0 * (1.0 - th * th) / 6.0e5
        p = P0 * torch.exp(-Z / H)
        rho = p / (GRAV * H)
        cx, cy, amp = 2.0e6 * rng.uniform(0.8, 1.2), 2.5e6 * rng.uniform(0.8, 1.2), rng.uniform(0.5, 1.5)
        u = -GRAV * Z * dH / (1.0e-4 * H)
        u = u + amp * torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / 6.0e5 ** 2)
        v = 0.2 * modes(True) * torch.sin(math.pi * xs[1])
        w = 0.01 * modes(False)
    else:
        big = case["flow"] == "sharp"
        c0 = (0.0, 0.0, 260.0) if big else (500.0, 500.0, 350.0)
        c = [v + rng.uniform(-100.0, 100.0) for v in c0]
        amp = rng.uniform(0.25, 1.0)
        r = torch.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2)
        bump = 1.0 if big else 0.5 * (1.0 + torch.cos(math.pi * r / 250.0))
        th = 300.0 + torch.where(r <= 250.0, amp * bump * torch.ones_like(r), torch.zeros_like(r))
        cp = GAMMA * RGAS / (GAMMA - 1.0)
        ex = 1.0 - GRAV * Z / (cp * 300.0)
        p = P0 * ex ** (cp / RGAS)
        rho = p / (RGAS * th * ex)
        u, v, w = 2.0 * modes(True), 2.0 * modes(True), 2.0 * modes(False)
    E = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v + w * w) + rho * GRAV * Z
    return torch.stack([rho, rho * u, rho * v, rho * w, E], 1).contiguous()


def _dt(case):
    """A fixed step below the acoustic bound of the smallest node spacing."""
    m, N = _mesh(case), case["N"]
    xi = _lgl(N)[0]
    h = min((m["hi"][d] - m["lo"][d]) / k for d, k in enumerate((case["kx"], case["ky"], case["kz"])))
    return 0.25 * h * (xi[1] - xi[0]) / (2.0 * 360.0)


def _bubble_args(case):
    if case["flow"] == "sharp":
        return dict(centre=(0.0, 0.0, 260.0), radius=250.0, profile="sharp")
    return {}


def prepare(case, seed):
    K, N = (case["kx"], case["ky"], case["kz"]), case["N"]
    if case["op"] == "server":
        rng = random.Random(seed)
        reqs = [dict(kind="bubble", K=(k, k, k), N=n, precision=case["precision"],
                     nsteps=case["steps"], amp=rng.uniform(0.25, 1.0),
                     centre=(500.0 + rng.uniform(-100, 100), 500.0 + rng.uniform(-100, 100),
                             350.0 + rng.uniform(-100, 100))) for k, n in _members(case)]
        srv = _lib.Server(hbm_budget_bytes=64 << 30, max_slots=64)
        srv.warmup(tuple(sorted({n for _, n in _members(case)})), case["precision"])
        return dict(op="server", srv=srv, reqs=reqs)
    q = _state(case, seed, _nodes(case))
    kw = dict(precision=case["precision"], warp=case["warp"], **_mesh(case), **_phys(case))
    if case["op"] == "slabs":
        s = _lib.PartitionedSolver(*K, N, P=case["slabs"], **kw)
        s.init_bubble(**_bubble_args(case))
        g = q.view(K[2], K[1], K[0], 5, -1)
        parts = [g[:, :, b:e].reshape(-1, 5, (N + 1) ** 3).contiguous() for b, e in s.bounds]
        return dict(op="slabs", s=s, q=parts, out=[torch.empty_like(p) for p in parts],
                    dt=_dt(case), n=case["steps"])
    s = _lib.Solver(*K, N, **kw)
    if case["flow"] == "jet":
        s.init_channel(background="jet")
    elif case["flow"] == "channel":
        s.init_channel()
    else:
        s.init_bubble(**_bubble_args(case))
    if case["op"] == "monitor":
        s.set_state(q)
    return dict(op=case["op"], s=s, q=q, out=torch.empty_like(q), dt=_dt(case), n=case["steps"])


def run(st):
    op = st["op"]
    if op == "step":
        s = st["s"]
        s.set_state(st["q"])
        s.step(st["dt"], st["n"])
        return s.get_state(st["out"])
    if op == "rhs":
        return st["s"].rhs(st["q"], st["out"])
    if op == "slabs":
        s = st["s"]
        for p, q in zip(s.parts, st["q"]):
            p.set_state(q)
        s.step(st["dt"], st["n"])
        return [p.get_state(o) for p, o in zip(s.parts, st["out"])]
    if op == "monitor":
        return dict(dt=st["s"].cfl_dt(0.5), integrals=st["s"].integrals())
    tickets = [st["srv"].submit(**r) for r in st["reqs"]]
    done = [st["srv"].wait(t) for t in tickets]
    return [dict(status=d["status"], nsteps=d["nsteps"], q=d["q"]) for d in done]


# ---- the work a pass cannot do without ---------------------------------------
def _stage_work(K, N, mixed, faces_periodic=2):
    nq = N + 1
    E = K[0] * K[1] * K[2]
    npn, pairs = E * nq ** 3, E * 3 * nq * nq * nq * (nq - 1) // 2
    fn = 3 * E * nq * nq
    # per node: the state in and out, the Runge-Kutta register in and out, eleven geometry
    # values; per face node: normal, scaling and geopotential.  Flops: 114 per unordered pair
    # and 56 per node (counted from the scheme's definition), about 200 per face node.
    word = 4 if mixed else 8
    return dict(bytes=npn * (80 + 10 * word + 11 * word) + fn * 40,
                flops=114 * pairs + 56 * npn + 200 * fn)


def work(case):
    if case["op"] == "server":
        b = f = 0
        for k, n in _members(case):
            w = _stage_work((k, k, k), n, case["precision"] == "mixed")
            b += w["bytes"] * 5 * case["steps"]
            f += w["flops"] * 5 * case["steps"]
        return dict(bytes=b, flops=f)
    K, N = (case["kx"], case["ky"], case["kz"]), case["N"]
    nodes = K[0] * K[1] * K[2] * (N + 1) ** 3
    if case["op"] == "monitor":
        # the state and coordinate z twice, J twice and the nine metric terms
        return dict(bytes=nodes * 8 * (2 * 7 + 9), flops=nodes * 120)
    w = _stage_work(K, N, case["precision"] == "mixed")
    n = 1 if case["op"] == "rhs" else 5 * case["steps"]
    return dict(bytes=w["bytes"] * n, flops=w["flops"] * n)


# ---- the same in plain 64-bit torch ------------------------------------------
class _Plain:
    """The semi-discrete right-hand side from its definition: flux differencing with the
    two-point entropy-conservative flux, matrix dissipation at the faces, mirror walls."""

    def __init__(self, case):
        self.case, self.N = case, case["N"]
        self.K = (case["kx"], case["ky"], case["kz"])
        self.per = _mesh(case)["periodic"]
        self.f0 = _phys(case).get("f0", 0.0)
        xi, w, D = _lgl(self.N)
        nq = self.N + 1
        self.nq, self.w = nq, w
        Dt = 2.0 * D
        Dt[0, 0] += 1.0 / w[0]
        Dt[-1, -1] -= 1.0 / w[-1]
        Dt -= np.diag(np.diag(Dt))
        self.D, self.Dt = torch.tensor(D, device="cuda"), torch.tensor(Dt, device="cuda")
        self.w3 = torch.tensor(np.einsum("i,j,k->kji", w, w, w).reshape(-1), device="cuda")
        self.x = _nodes(case)
        E = self.x.shape[0]
        X = self.x.view(E, 3, nq, nq, nq)
        self.phi = GRAV * self.x[:, 2]
        der = lambda f, d: torch.einsum("ab,...b->...a", self.D, f.movedim(4 - d - 1, -1)).movedim(-1, 4 - d - 1)
        dX = [[der(X[:, c], d) for d in range(3)] for c in range(3)]
        self.J = (dX[0][0] * (dX[1][1] * dX[2][2] - dX[1][2] * dX[2][1])
                  - dX[0][1] * (dX[1][0] * dX[2][2] - dX[1][2] * dX[2][0])
                  + dX[0][2] * (dX[1][0] * dX[2][1] - dX[1][1] * dX[2][0])).reshape(E, -1)
        Ja = torch.empty(E, 3, 3, nq, nq, nq, dtype=torch.float64, device="cuda")
        for c in range(3):
            m, l = (c + 1) % 3, (c + 2) % 3
            Xl = X[:, l] - X[:, l, :1, :1, :1]
            V = [Xl * dX[m][d] for d in range(3)]
            for d in range(3):
                a, b = (d + 1) % 3, (d + 2) % 3
                Ja[:, d, c] = der(V[a], b) - der(V[b], a)
        self.Ja = Ja.view(E, 3, 3, -1)

    @staticmethod
    def prims(q, phi):
        """rho, u, b = rho/(2p) of the state along dim 1."""
        rho = q[:, 0]
        u = [q[:, 1] / rho, q[:, 2] / rho, q[:, 3] / rho]
        p = (GAMMA - 1.0) * (q[:, 4] - rho * phi - 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
        return rho, u, rho / (2.0 * p)

    @staticmethod
    def logs(a, b):
        """The logarithmic mean of a and b, and log(b/a)."""
        f = (b - a) / (b + a)
        v = f * f
        near = v < 1e-4
        A = 1.0 + v * (1.0 / 3.0 + v * (1.0 / 5.0 + v * (1.0 / 7.0 + v / 9.0)))
        lj = torch.where(near, 2.0 * f * A, torch.log1p((b - a) / a))
        safe = torch.where(near, torch.ones_like(lj), lj)
        return torch.where(near, 0.5 * (a + b) / A, (b - a) / safe), lj

    def ec(self, r, rm, um, u2, bm, b_log, n, phi):
        """The symmetric flux from means: log mean r of rho, mean rho, u, u-.u+, b."""
        un = sum(a * b for a, b in zip(um, n))
        ps = rm / (2.0 * bm)
        F = r * un
        out = [F] + [F * um[c] + ps * n[c] for c in range(3)]
        out.append(F * (1.0 / (2.0 * (GAMMA - 1.0) * b_log) + 0.5 * u2 + phi) + ps * un)
        return out

    def volume(self, q, out):
        nq, E = self.nq, q.shape[0]
        step = max(1, int(2.0e6 // nq ** 4))
        for e0 in range(0, E, step):
            e1 = min(E, e0 + step)
            sh = (e1 - e0, nq, nq, nq)
            phi = self.phi[e0:e1]
            rho, u, b = self.prims(q[e0:e1], phi)
            for d in range(3):
                ax = 3 - d
                v = lambda f: f.reshape(sh).movedim(ax, -1)
                A = lambda f: v(f).unsqueeze(-1)
                B = lambda f: v(f).unsqueeze(-2)
                n = [0.5 * (A(self.Ja[e0:e1, d, c]) + B(self.Ja[e0:e1, d, c])) for c in range(3)]
                rl = self.logs(A(rho), B(rho))[0]
                bl = self.logs(A(b), B(b))[0]
                um = [0.5 * (A(c) + B(c)) for c in u]
                u2 = sum(A(c) * B(c) for c in u)
                bm = 0.5 * (A(b) + B(b))
                F = self.ec(rl, 0.5 * (A(rho) + B(rho)), um, u2, bm, bl, n, 0.5 * (A(phi) + B(phi)))
                g = 0.5 * bm * rl / A(b) * (B(phi) - A(phi))
                for c in range(3):
                    F[1 + c] = F[1 + c] + g * n[c]
                for k in range(5):
                    s = (self.Dt * F[k]).sum(-1).movedim(-1, ax)
                    out[e0:e1, k] += s.reshape(e1 - e0, -1)

    def face(self, d, qm, qp, n, phi):
        """The interface flux of "-" and "+" states [F][5][nq][nq] with unit normal n."""
        rm, um, bm = self.prims(qm, phi)
        rp, up, bp = self.prims(qp, phi)
        r, ljr = self.logs(rm, rp)
        bl, ljb = self.logs(bm, bp)
        u = [0.5 * (a + b) for a, b in zip(um, up)]
        F = self.ec(r, 0.5 * (rm + rp), u, sum(a * b for a, b in zip(um, up)), 0.5 * (bm + bp), bl,
                    n, phi)
        pt = 0.5 * (rm + rp) / (bm + bp)
        db = bp - bm
        sq = lambda a: a[0] ** 2 + a[1] ** 2 + a[2] ** 2
        j1 = ljr + ljb / (GAMMA - 1.0) - (bp * sq(up) - bm * sq(um)) + 2.0 * phi * db
        jm = [2.0 * (bp * up[c] - bm * um[c]) for c in range(3)]
        j5 = -2.0 * db
        a2 = GAMMA * pt / r
        a = torch.sqrt(a2)
        un = sum(x * y for x, y in zip(u, n))
        k2 = 0.5 * sq(u) + phi
        H = a2 / (GAMMA - 1.0) + k2
        # R |Lambda| T R^T [[v]]: the two acoustic waves, the entropy wave and the shear part
        dm = 0.0
        waves = [(un - a, 0.5 * r / GAMMA, [u[c] - a * n[c] for c in range(3)], H - a * un),
                 (un, r * (GAMMA - 1.0) / GAMMA, u, k2),
                 (un + a, 0.5 * r / GAMMA, [u[c] + a * n[c] for c in range(3)], H + a * un)]
        D = [0.0, 0.0, 0.0, 0.0, 0.0]
        for lam, T, m, e in waves:
            c = lam.abs() * T * (j1 + sum(x * y for x, y in zip(m, jm)) + e * j5)
            for k, z in enumerate([1.0] + m + [e]):
                D[k] = D[k] + c * z
        y = [jm[c] + u[c] * j5 for c in range(3)]
        yn = sum(x * z for x, z in zip(y, n))
        t = [un.abs() * pt * (y[c] - yn * n[c]) for c in range(3)]
        for c in range(3):
            D[1 + c] = D[1 + c] + t[c]
        D[4] = D[4] + sum(x * z for x, z in zip(u, t))
        return torch.stack([f - 0.5 * x for f, x in zip(F, D)], 1)

    def rhs(self, q):
        K, nq, N = self.K, self.nq, self.N
        out = torch.zeros_like(q)
        self.volume(q, out)
        grid = lambda f, k: f.reshape(K[2], K[1], K[0], k, nq, nq, nq)
        Q, O, P = grid(q, 5), grid(out, 5), grid(self.phi, 1)
        for d in range(3):
            ea, na = 2 - d, 6 - d
            lo, hi = Q.select(na, 0), Q.select(na, N)        # [K2][K1][K0][5][nq][nq]
            M = grid(self.Ja[:, d], 3)
            mhi, mlo = M.select(na, N), M.select(na, 0)
            ph, pl = P.select(na, N), P.select(na, 0)
            k = K[d]
            cat = lambda *t: torch.cat(t, ea)
            if self.per[d]:                                    # plane above each element
                qm, qp, m, p = hi, torch.roll(lo, -1, ea), mhi, ph
            else:
                fst, lst = lo.narrow(ea, 0, 1), hi.narrow(ea, k - 1, 1)
                qm, qp = cat(fst, hi), cat(lo, lst)
                m, p = cat(mlo.narrow(ea, 0, 1), mhi), cat(pl.narrow(ea, 0, 1), ph)
            shape = qm.shape
            fl = lambda f: f.reshape((-1,) + f.shape[3:])
            qm, qp, m, p = fl(qm).clone(), fl(qp).clone(), fl(m), fl(p)[:, 0]
            s = torch.sqrt((m * m).sum(1))
            n = [m[:, c] / s for c in range(3)]
            if not self.per[d]:                                # mirror states at the walls
                qg, pg = qm.view(shape), qp.view(shape)
                ng = torch.stack(n, 1).view(shape[:3] + (3,) + shape[4:])
                for at, dst, src in ((0, qg, pg), (k, pg, qg)):
                    a, b, v = dst.narrow(ea, at, 1), src.narrow(ea, at, 1), ng.narrow(ea, at, 1)
                    Un = (b[:, :, :, 1:4] * v).sum(3, keepdim=True)
                    a.copy_(b)
                    a[:, :, :, 1:4] -= 2.0 * Un * v
            F = (self.face(d, qm, qp, n, p) * (s / self.w[-1]).unsqueeze(1)).view(shape)
            if self.per[d]:
                O.select(na, N).add_(F)
                O.select(na, 0).sub_(torch.roll(F, 1, ea))
            else:
                O.select(na, N).add_(F.narrow(ea, 1, k))
                O.select(na, 0).sub_(F.narrow(ea, 0, k))
        out = -out / self.J.unsqueeze(1)
        if self.f0:
            out[:, 1] += self.f0 * q[:, 2]
            out[:, 2] -= self.f0 * q[:, 1]
        return out

    def steps(self, q, dt, n):
        q, dq = q.clone(), torch.zeros_like(q)
        for _ in range(n):
            for a, b in zip(RK_A, RK_B):
                dq = a * dq + dt * self.rhs(q)
                q = q + b * dq
        return q


def exact(case, seed):
    if case["op"] == "server":
        return None  # minutes of plain 64-bit steps
    P = _Plain(case)
    q = _state(case, seed, P.x)
    if case["op"] == "rhs":
        return P.rhs(q)
    if case["op"] == "monitor":
        rho, u, b = P.prims(q, P.phi)
        p = rho / (2.0 * b)
        c = torch.sqrt(GAMMA * p / rho)
        lam = 0.0
        for d in range(3):
            j = [P.Ja[:, d, k] for k in range(3)]
            sp = sum(a * v for a, v in zip(u, j)).abs() + c * torch.sqrt(sum(a * a for a in j))
            lam = max(lam, float((sp / P.J).max()))
        xi = _lgl(case["N"])[0]
        wJ = P.w3 * P.J
        ent = -rho * (torch.log(p) - GAMMA * torch.log(rho)) / (GAMMA - 1.0)
        return dict(dt=0.5 * float(xi[1] - xi[0]) / lam,
                    integrals=np.array([float((wJ * v).sum()) for v in (rho, q[:, 4], ent)]))
    z = P.steps(q, _dt(case), case["steps"])
    if case["op"] == "slabs":
        K = P.K
        from_, parts = 0, []
        for k in range(case["slabs"]):
            n = K[0] // case["slabs"] + (1 if k < K[0] % case["slabs"] else 0)
            g = z.view(K[2], K[1], K[0], 5, -1)[:, :, from_:from_ + n]
            parts.append(g.reshape(-1, 5, P.nq ** 3))
            from_ += n
        return parts
    return z
