"""The work that users of the solver have it do, as cases for measuring it.

Three kinds of case:

  steps    a body that a program keeps: one pass advances it by `steps` time
           steps and reads fields back into the program's pinned buffer (the
           step / read loop of every simulation, short or long);
  batch    several uneven bodies grouped into one lbm.Batch (the batched
           workload, and the inner loop of the serving loop): one pass
           advances all of them and reads each one's displacement;
  solve    a whole request as the serving loop answers it: create the body
           from host arrays, step, read the displacement, close.

A case names the grid, the edges, the storage format and the displacement
carry, the scheme, the step count of a pass and the fields it reads.
exact() is Algorithm 1 of arXiv 2208.13769 with its boundary rules in plain
torch, 64 bits, written here from the method's equations.
"""
import math

import numpy as np
import torch

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300.workloads import DIRICHLET, NEUMANN, PERIODIC, Edge, Problem

U, V = lbm.LBM_FIELD_U, lbm.LBM_FIELD_V
MASKS = {"u": U, "uv": U | V, "all": 127}
FIELDS = {"u": ("u",), "uv": ("u", "v"), "all": ("u", "v", "P", "Pbar", "r", "sigma", "J")}
COMPS = {"u": 2, "v": 2, "P": 4, "Pbar": 3, "r": 1, "sigma": 3, "J": 1}
CARRY = {"plain": False, "pair": True, "lo16": "lo16", "": None}
SCHEME = {"explicit": lbm.LBM_SCHEME_EXPLICIT, "predictor": lbm.LBM_SCHEME_PREDICTOR}


def _steps(name, nx, ny, edges, storage, carry, scheme, steps, read):
    return {"name": name, "kind": "steps", "nx": nx, "ny": ny, "edges": edges, "storage": storage, "carry": carry,
            "scheme": scheme, "steps": steps, "read": read}


def _batch(name, bodies, lo, hi, storage, carry, steps):
    return {"name": name, "kind": "batch", "bodies": bodies, "side_lo": lo, "side_hi": hi, "storage": storage,
            "carry": carry, "scheme": "predictor", "steps": steps, "read": "u"}


def listed():
    return [
        # the smallest call: a program that watches its body after every step
        _steps("watch 128x128 f32", 128, 128, "clamped", "f32", "pair", "explicit", 1, "uv"),
        # the 64 x 64 shear wave for its 1000 steps, in the library's default storage
        _steps("wave 64x64 f64", 64, 64, "periodic", "f64", "", "predictor", 1000, "uv"),
        # the paper's plate with a square hole, pulled at top and bottom, to its t = 3
        _steps("plate 80x80 f64", 80, 80, "plate", "f64", "", "explicit", 416, "uv"),
        # a small ragged body in the default FP32 form
        _steps("clamped 301x203 f32", 301, 203, "clamped", "f32", "pair", "explicit", 500, "uv"),
        # a middling body with every observable read back (stresses included)
        _steps("periodic 512x512 f32", 512, 512, "periodic", "f32", "lo16", "predictor", 200, "all"),
        # the ordinary serving size in 16-bit storage, odd sides
        _steps("clamped 1000x777 f16", 1000, 777, "clamped", "f16", "", "predictor", 200, "uv"),
        # double precision at size: a moving wall, a ramped traction, a periodic axis
        _steps("mixed 701x900 f64", 701, 900, "mixed", "f64", "", "explicit", 64, "uv"),
        # the 4096 x 2048 clamped body, FP32 with the 16-bit low words and with FP16 populations
        _steps("clamped 4096x2048 f32", 4096, 2048, "clamped", "f32", "lo16", "explicit", 100, "uv"),
        _steps("clamped 4096x2048 f16", 4096, 2048, "clamped", "f16", "", "explicit", 100, "uv"),
        # uneven bodies advanced together: the batched workload's sizes, and the serving trace's
        _batch("batch 32 f32", 32, 64, 1024, "f32", "lo16", 130),
        _batch("batch 12 f16", 12, 128, 2048, "f16", "", 100),
        # a request from arrival to answer
        {"name": "solve 640x384 f16", "kind": "solve", "nx": 640, "ny": 384, "edges": "clamped", "storage": "f16",
         "carry": "", "scheme": "predictor", "steps": 500, "read": "u"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    storage, carry = rng.choice([("f64", ""), ("f32", "pair"), ("f32", "lo16"), ("f32", "plain"), ("f16", ""),
                                 ("bf16", "")])
    kind = rng.choice(["steps", "steps", "steps", "steps", "batch", "solve"])
    if kind == "batch":
        lo, hi = rng.choice([(64, 512), (64, 1024), (128, 1024)])
        if storage == "f64":
            storage, carry = "f16", ""
        c = _batch("", rng.randint(3, 24), lo, hi, storage, carry, rng.randint(20, 130))
        del c["name"]
        return c
    scheme = rng.choice(["explicit", "predictor"])
    edges = rng.choice(["periodic", "clamped", "clamped", "mixed", "plate"])
    nx = _log(rng, 40, 3000)
    ny = min(3000, max(40, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    # a pass of at most about 4e8 node updates (an eighth of that in FP64), 1000 steps
    most = (5e7 if storage == "f64" else 4e8) / (nx * ny)
    steps = max(1, min(_log(rng, 1, 1000), int(most)))
    read = rng.choice(["u", "uv", "uv", "all"]) if kind == "steps" else "u"
    return {"kind": kind, "nx": nx, "ny": ny, "edges": edges, "storage": storage, "carry": carry, "scheme": scheme,
            "steps": steps, "read": read}


# ------------------------------------------------------------------ inputs

def _axis(n, dX, periodic):
    return (np.arange(n) + (0.0 if periodic else 0.5)) * dX


def _problem(nx, ny, edges, rng):
    """One body with the seed's material and initial fields.  Poisson ratio
    0.25 (lambda = mu, the paper's) except in a fully periodic body, strains
    of a few per cent, so that it stays stable over many passes."""
    mu, dX, omega, hole = float(rng.uniform(0.2, 0.4)), 1.0, 1.8, None
    lam = mu
    if edges == "periodic":
        e = [Edge(PERIODIC) for _ in range(4)]
        nu = float(rng.uniform(0.2, 0.25))
        lam = 2.0 * mu * nu / (1.0 - 2.0 * nu)
    elif edges == "clamped":  # left edge held, the others free
        e = [Edge(DIRICHLET), Edge(NEUMANN), Edge(NEUMANN), Edge(NEUMANN)]
        omega = 1.9
    elif edges == "mixed":  # a slowly moving wall, a ramped traction, periodic along y
        w = rng.uniform(-1e-5, 1e-5, 2)
        T = rng.uniform(-1e-3, 1e-3, 2)
        e = [Edge(DIRICHLET, rate=(float(w[0]), float(w[1]))),
             Edge(NEUMANN, rate=(float(T[0]), float(T[1])), times=(0.0, 50.0, math.inf)), Edge(PERIODIC), Edge(PERIODIC)]
    else:  # the plate: a centred square hole of 0.4 of the shorter side, pulled for a while at top and bottom
        dX = 1.0 / nx
        T = float(rng.uniform(0.01, 0.03)) * mu
        pull = dict(times=(0.0, 0.0, 1.0))
        e = [Edge(NEUMANN), Edge(NEUMANN), Edge(NEUMANN, rate=(0.0, -T), **pull), Edge(NEUMANN, rate=(0.0, T), **pull)]
        h = int(round(0.4 * min(nx, ny)))
        hole = ((nx - h) // 2, (nx - h) // 2 + h, (ny - h) // 2, (ny - h) // 2 + h)
    px, py = e[0].kind == PERIODIC, e[2].kind == PERIODIC
    x, y = _axis(nx, dX, px) / (nx * dX), _axis(ny, dX, py) / (ny * dX)
    C = math.sqrt(mu)  # transverse wave speed (rho0 = 1)
    u0, v0 = np.zeros((ny, nx, 2)), np.zeros((ny, nx, 2))
    if edges == "clamped":  # swings about its held edge; u0 = 0
        v0[:, :, 1] = np.multiply.outer(1.0 + 0.1 * rng.uniform(-1, 1) * np.cos(np.pi * y),
                                        rng.uniform(0.5, 1.0) * 0.01 * x)
    elif edges != "plate":
        amp = float(rng.uniform(0.5, 1.0)) * 2e-3 * min(nx, ny) * dX
        for c in range(2):
            kx, ky = int(rng.integers(0, 3)), int(rng.integers(1, 3))
            a, b = rng.uniform(0, 2 * np.pi, 2)
            fx, fy = np.cos(2 * np.pi * kx * x + a), np.cos(2 * np.pi * ky * y + b)
            if not px:
                fx = np.sin(0.5 * np.pi * x) ** 2  # at rest at the wall
            u0[:, :, c] = np.multiply.outer(fy, amp * fx)
            v0[:, :, c] = np.multiply.outer(np.roll(fy, 3) if py else fy, 1e-3 * C * fx)
    return Problem(nx=nx, ny=ny, lam=lam, mu=mu, omega=omega, dX=dX, edges=e, u0=u0, v0=v0, hole=hole)


def _problems(case, seed):
    rng = np.random.default_rng([int(seed), 2208])
    if case["kind"] != "batch":
        return [_problem(case["nx"], case["ny"], case["edges"], rng)]
    # the sizes are the case's, not the seed's; half of the bodies periodic, half clamped
    sides = np.random.default_rng([case["bodies"], case["side_lo"], case["side_hi"]])
    out = []
    for k in range(case["bodies"]):
        nx, ny = (int(n) for n in sides.integers(case["side_lo"], case["side_hi"] + 1, 2))
        out.append(_problem(nx, ny, "periodic" if k % 2 else "clamped", rng))
    return out


def _buffer(problem, read):
    """The program's own result buffer for one body: pinned host memory."""
    n = sum(COMPS[f] for f in FIELDS[read]) * problem.nx * problem.ny
    return torch.empty(n, dtype=torch.float64, pin_memory=torch.cuda.is_available()).numpy()


def _views(buf, problem, read):
    out, at = {}, 0
    for f in FIELDS[read]:
        n = COMPS[f] * problem.nx * problem.ny
        out[f] = buf[at:at + n].reshape(problem.ny, problem.nx, COMPS[f])
        at += n
    return out


def _body(case, problem):
    return lbm.Body(problem, storage=case["storage"], compensated=CARRY[case["carry"]], scheme=SCHEME[case["scheme"]])


def prepare(case, seed):
    probs = _problems(case, seed)
    state = {"case": case, "bufs": [_buffer(p, case["read"]) for p in probs]}
    state["views"] = [_views(b, p, case["read"]) for b, p in zip(state["bufs"], probs)]
    if case["kind"] == "solve":
        state["problem"] = probs[0]
    else:
        state["bodies"] = [_body(case, p) for p in probs]
        if case["kind"] == "batch":
            state["batch"] = lbm.Batch(state["bodies"])
    return state


def run(state):
    case = state["case"]
    mask = MASKS[case["read"]]
    if case["kind"] == "solve":
        with _body(case, state["problem"]) as body:
            body.step(case["steps"])
            lbm.lbm_read_fields(body.ctx, mask, state["bufs"][0], allow_unstable=True)
        return state["views"][0]
    (state["batch"] if case["kind"] == "batch" else state["bodies"][0]).step(case["steps"])
    for body, buf in zip(state["bodies"], state["bufs"]):
        lbm.lbm_read_fields(body.ctx, mask, buf, allow_unstable=True)
    return state["views"] if case["kind"] == "batch" else state["views"][0]


def work(case):
    """Per step and node: nine populations and two components each of the
    displacement and of the source, read once and written once; about 230
    operations.  Then the fields that are read."""
    e = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[case["storage"]]
    carry = 8 if case["storage"] == "f64" else 4
    # 16-bit populations go with a displacement of 64 bits
    per = 2 * (9 * e + 2 * (8 if e != 4 else 4) + 2 * carry)
    nodes = sum(p.nodes for p in _shapes(case))
    read = 8 * sum(COMPS[f] for f in FIELDS[case["read"]])
    return {"bytes": float(nodes) * (case["steps"] * per + read), "flops": 230.0 * nodes * case["steps"]}


def _shapes(case):
    if case["kind"] != "batch":
        n = case["nx"] * case["ny"]
        if case["edges"] == "plate":
            n -= int(round(0.4 * min(case["nx"], case["ny"]))) ** 2
        return [_Shape(n)]
    sides = np.random.default_rng([case["bodies"], case["side_lo"], case["side_hi"]])
    return [_Shape(int(np.prod(sides.integers(case["side_lo"], case["side_hi"] + 1, 2))))
            for _ in range(case["bodies"])]


class _Shape:
    def __init__(self, nodes):
        self.nodes = nodes


# ------------------------------------------------------------------ the method in 64 bits

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Exact:
    """Algorithm 1 (or the footnote's predictor) on one body, 64-bit torch.

    Moments are kept in units of the lattice speed c = dX / dt: jh = j / c,
    pi = Pbar / c^2, s = (dt / c) 1S."""

    def __init__(self, p, predictor, dev):
        self.p, self.predictor, self.dev = p, predictor, dev
        self.nx, self.ny = p.nx, p.ny
        self.dt = p.dX / math.sqrt(3.0 * p.mu / p.rho0)
        self.c = p.dX / self.dt
        self.kind = [e.kind for e in p.edges]
        self.per = (self.kind[0] == PERIODIC, self.kind[2] == PERIODIC)
        self.ku = p.dX / (2.0 * p.rho0)
        self.mask = torch.ones(p.ny, p.nx, dtype=torch.float64, device=dev)
        if p.hole:
            x0, x1, y0, y1 = p.hole
            self.mask[y0:y1, x0:x1] = 0.0
        self._links()

    # the links that leave the body: (direction, row, column, wall normal, the walls crossed)
    def _links(self):
        nx, ny, hole = self.nx, self.ny, self.p.hole
        rows = []

        def inside_hole(x, y):
            return hole is not None and hole[0] <= x < hole[1] and hole[2] <= y < hole[3]

        near = set()
        for x in range(nx):
            near.update(((x, 0), (x, ny - 1)))
        for y in range(ny):
            near.update(((0, y), (nx - 1, y)))
        if hole:
            x0, x1, y0, y1 = hole
            near.update((x, y) for x in range(x0 - 1, x1 + 1) for y in (y0 - 1, y1))
            near.update((x, y) for y in range(y0 - 1, y1 + 1) for x in (x0 - 1, x1))
        for x, y in near:
            for i in range(1, 9):
                tx, ty = x + EX[i], y + EY[i]
                if inside_hole(tx, ty):
                    cx = EX[i] != 0 and inside_hole(tx, y)
                    cy = EY[i] != 0 and inside_hole(x, ty)
                    sx = EX[i] if cx or not cy else 0
                    sy = EY[i] if cy or not cx else 0
                    a = (4 if sx > 0 else 5) if sx else 8
                    b = (6 if sy > 0 else 7) if sy else 8
                else:
                    bx = not self.per[0] and not 0 <= tx < nx
                    by = not self.per[1] and not 0 <= ty < ny
                    if not bx and not by:
                        continue
                    sx, sy = (EX[i] if bx else 0), (EY[i] if by else 0)
                    a = (0 if sx < 0 else 1) if bx else 8
                    b = (2 if sy < 0 else 3) if by else 8
                rows.append((i, y, x, sx, sy, a, b))
        self.link = None
        if rows:
            t = torch.tensor(rows, dtype=torch.int64, device=self.dev).T
            self.link = t
            d = torch.tensor([k == DIRICHLET for k in self.kind] + [False] * 5, device=self.dev)
            self.da, self.db = d[t[5]].double(), d[t[6]].double()
            f64 = dict(dtype=torch.float64, device=self.dev)
            self.lex, self.ley = torch.tensor(EX, **f64)[t[0]], torch.tensor(EY, **f64)[t[0]]
            self.lw = torch.tensor(W, **f64)[t[0]]
            self.opp = torch.tensor(OPP, device=self.dev)[t[0]]
            self.il = 1.0 / torch.sqrt((t[3] ** 2 + t[4] ** 2).double())

    # wall data at time t: tractions and wall momenta of the 4 edges, 4 faces of the hole, none
    def _walls(self, t):
        T, J = [], []
        for e in self.p.edges:
            s = 0.0
            if e.times[0] <= t < e.times[2]:
                s = min(1.0, (t - e.times[0]) / e.times[1]) if e.times[1] > 0 else 1.0
            T.append([a + (b - a) * s for a, b in zip(e.value, e.rate)] if e.kind == NEUMANN else [0.0, 0.0])
            J.append([r * self.p.rho0 / self.c for r in e.rate] if e.kind == DIRICHLET else [0.0, 0.0])
        T += self.p.hole_traction or [[0.0, 0.0]] * 4
        pad = [[0.0, 0.0]] * (9 - len(J))
        f64 = dict(dtype=torch.float64, device=self.dev)
        return torch.tensor([list(r) for r in T] + [[0.0, 0.0]], **f64), torch.tensor(J + pad, **f64)

    # a(+1) - a(-1) along x (0) or y (1); ustar: (low, high) wall values of a Dirichlet axis, else linear ghosts
    def _diff(self, a, axis, ustar=(None, None)):
        dim = 1 - axis
        d = torch.roll(a, -1, dim) - torch.roll(a, 1, dim)
        at = (lambda k: a[:, k]) if axis == 0 else (lambda k: a[k])
        out = (lambda k: d[:, k]) if axis == 0 else (lambda k: d[k])
        if not self.per[axis]:
            lo, hi = ustar
            out(0).copy_(at(1) - (2 * lo - at(0)) if lo is not None else 2 * (at(1) - at(0)))
            out(-1).copy_((2 * hi - at(-1)) - at(-2) if hi is not None else 2 * (at(-1) - at(-2)))
        if self.p.hole:
            x0, x1, y0, y1 = self.p.hole
            if axis == 0:
                d[y0:y1, x0 - 1] = 2 * (a[y0:y1, x0 - 1] - a[y0:y1, x0 - 2])
                d[y0:y1, x1] = 2 * (a[y0:y1, x1 + 1] - a[y0:y1, x1])
            else:
                d[y0 - 1, x0:x1] = 2 * (a[y0 - 1, x0:x1] - a[y0 - 2, x0:x1])
                d[y1, x0:x1] = 2 * (a[y1 + 1, x0:x1] - a[y1, x0:x1])
        return d

    def grad(self, u, t):
        H = []
        for c in range(2):
            wall = [e.value[c] + e.rate[c] * t if e.kind == DIRICHLET else None for e in self.p.edges]
            H += [self._diff(u[c], 0, wall[:2]) / (2 * self.p.dX) * self.mask,
                  self._diff(u[c], 1, wall[2:]) / (2 * self.p.dX) * self.mask]
        return H

    def stress(self, H):
        """P (11, 12, 21, 22), Pbar (11, 12, 22), J of the neo-Hooke material."""
        h11, h12, h21, h22 = H
        lam, mu = self.p.lam, self.p.mu
        d = h11 + h22 + (h11 * h22 - h12 * h21)
        J = 1 + d
        F = (1 + h11, h12, h21, 1 + h22)
        G = (F[3] / J, -F[2] / J, -F[1] / J, F[0] / J)  # F^-T
        vol = 0.5 * lam * d * (2 + d)
        P = [mu * (f - g) + vol * g for f, g in zip(F, G)]
        tr = h11 + h22
        return P, [-mu * (2 * h11 + tr), -mu * (h12 + h21), -mu * (2 * h22 + tr)], J, F

    def source(self, u, t):
        """s and Q = P + Pbar (11, 12, 21, 22)."""
        P, B, _, _ = self.stress(self.grad(u, t))
        Q = (P[0] + B[0], P[1] + B[1], P[2] + B[1], P[3] + B[2])
        k = self.dt ** 2 / (2 * self.p.dX ** 2)
        return [k * (self._diff(Q[0], 0) + self._diff(Q[1], 1)) * self.mask,
                k * (self._diff(Q[2], 0) + self._diff(Q[3], 1)) * self.mask], Q

    @staticmethod
    def _even(e2, ex, ey, r, a, b, c):
        return r * (2 - 1.5 * e2) + 1.5 * (3 * (ex * ex * a + 2 * ex * ey * b + ey * ey * c) - (a + c))

    def collide(self, f, r, pi, jh, s, Q, t):
        """Post-collision populations with a ring of ghost cells: images across a seam, what the walls send back."""
        om = self.p.omega
        g = torch.zeros(9, self.ny + 2, self.nx + 2, dtype=torch.float64, device=self.dev)
        for i in range(9):
            even = self._even(EX[i] ** 2 + EY[i] ** 2, EX[i], EY[i], r, *pi)
            odd = 3 * (EX[i] * jh[0] + EY[i] * jh[1])
            force = 3 * (1 - 0.5 * om) * (EX[i] * s[0] + EY[i] * s[1])
            eq = W[i] * (even + odd)
            g[i, 1:-1, 1:-1] = eq + W[i] * force if f is None else (1 - om) * f[i] + om * eq + W[i] * force
        if self.per[0]:
            g[:, :, 0], g[:, :, -1] = g[:, :, -2], g[:, :, 1]
        if self.per[1]:
            g[:, 0], g[:, -1] = g[:, -2], g[:, 1]
        if self.link is not None:
            i, y, x, sx, sy, a, b = self.link
            T, J = self._walls(t)
            fi = g[i, y + 1, x + 1]
            # bounce-back off a moving wall
            n = torch.clamp(self.da + self.db, min=1.0)
            jw = (J[a] * self.da[:, None] + J[b] * self.db[:, None]) / n[:, None]
            back = fi - 2 * self.lw * 3 * (self.lex * jw[:, 0] + self.ley * jw[:, 1])
            # anti-bounce-back with the wall's Poisson stress
            N0, N1 = sx * self.il, sy * self.il
            t0, t1 = -N1, N0
            q = [v[y, x] for v in Q]
            Tw = (T[a] + T[b]) * self.il[:, None]
            g0, g1 = q[0] * N0 + q[1] * N1 - Tw[:, 0], q[2] * N0 + q[3] * N1 - Tw[:, 1]
            nn, nt = (N0 * g0 + N1 * g1) / self.c ** 2, (t0 * g0 + t1 * g1) / self.c ** 2
            pw = [v[y, x] for v in pi]
            tt = t0 * t0 * pw[0] + 2 * t0 * t1 * pw[1] + t1 * t1 * pw[2]
            S = [nn * A + nt * B + tt * C for A, B, C in (
                (N0 * N0, 2 * N0 * t0, t0 * t0), (N0 * N1, N0 * t1 + t0 * N1, t0 * t1), (N1 * N1, 2 * N1 * t1, t1 * t1))]
            anti = -fi + 2 * self.lw * self._even(self.lex ** 2 + self.ley ** 2, self.lex, self.ley, r[y, x], *S)
            val = torch.where(self.da + self.db > 0, back, anti)
            g[self.opp, y + 1 + self.ley.long(), x + 1 + self.lex.long()] = val
        return g

    def solve(self, steps):
        p, c = self.p, self.c
        put = lambda a: [torch.from_numpy(np.ascontiguousarray(a[:, :, k])).to(self.dev) * self.mask for k in range(2)]  # noqa: E731
        u, v = put(p.u0), put(p.v0)
        H = self.grad(u, 0.0)
        _, B, _, _ = self.stress(H)
        r = -p.rho0 * (H[0] + H[3])
        jh = [a * (p.rho0 / c) for a in v]
        s, Q = self.source(u, 0.0)
        g = self.collide(None, r, [b / c ** 2 for b in B], jh, s, Q, 0.0)
        for n in range(1, steps + 1):
            t = n * self.dt
            f = torch.stack([g[i, 1 - EY[i]:1 - EY[i] + self.ny, 1 - EX[i]:1 - EX[i] + self.nx] for i in range(9)])
            f *= self.mask
            r = f.sum(0)
            m = [f[1] - f[3] + f[5] - f[6] + f[8] - f[7], f[2] - f[4] + f[5] - f[8] + f[6] - f[7]]
            diag = f[5] + f[6] + f[7] + f[8]
            pi = [f[1] + f[3] + diag, f[5] - f[6] + f[7] - f[8], f[2] + f[4] + diag]
            now = [a + 0.5 * b for a, b in zip(m, s)]
            trial = [a + self.ku * (b + d) for a, b, d in zip(u, jh, now)]
            s, Q = self.source(trial, t)
            if self.predictor:
                now = [a + 0.5 * b for a, b in zip(m, s)]
                trial = [a + self.ku * (b + d) for a, b, d in zip(u, jh, now)]
            u, jh = trial, now
            g = self.collide(f, r, pi, jh, s, Q, t)
        P, B, J, F = self.stress(self.grad(u, steps * self.dt))
        sig = [(P[2 * a] * F[2 * b] + P[2 * a + 1] * F[2 * b + 1]) / J for a, b in ((0, 0), (0, 1), (1, 1))]
        v = [a * (c / p.rho0) for a in jh]
        out = {"u": u, "v": v, "P": P, "Pbar": B, "r": [r], "sigma": sig, "J": [J]}
        return {k: torch.stack([a.cpu() for a in x], -1).numpy() for k, x in out.items()}


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    out = []
    for p in _problems(case, seed):
        got = _Exact(p, case["scheme"] == "predictor", dev).solve(case["steps"])
        out.append({f: got[f] for f in FIELDS[case["read"]]})
        # how the library hands back the nodes of a hole: at rest, undeformed
        if p.hole is not None and "J" in out[-1]:
            out[-1]["J"][p.hole[2]:p.hole[3], p.hole[0]:p.hole[1]] = 1.0
    return out if case["kind"] == "batch" else out[0]
