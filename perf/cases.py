"""Workloads of the asynchronous DG library at the sizes its users run, for timing and for
comparing results: the solver in its three arithmetics, two and three dimensions and every
subdomain-face rule, the batched solver, the bare operator, a whole short study, the
learned ghost-trace predictor in the solver, and a training step of that predictor.

A case is a dict of plain values; `prepare` makes what a program holds before its call
(handles, states on the device), `run` is one pass through the public entry points,
`exact` the same pass in plain 64-bit torch arithmetic.
"""
import math

import numpy as np
import torch

from paper_2603_28710_gb300 import adg, learned

GAMMA = 1.4
RK_STAGES = {"rk22": 2, "rk33": 3, "ck45": 5}


# ---- the cases ------------------------------------------------------------------------

def _step(name, dim, blocks, block, degree, precision, flux="at", delay_mode="caa", max_delay=0,
          random_delay_max=0, at_np=0, rk="ck45", steps=1, kind="step"):
    """blocks x block elements per direction (blocks = subdomains along it)."""
    c = {"kind": kind, "dim": dim, "degree": degree, "precision": precision, "flux": flux,
         "delay_mode": delay_mode, "max_delay": max_delay, "random_delay_max": random_delay_max,
         "at_np": at_np, "rk": rk, "steps": steps}
    for d in range(3):
        c["P%d" % d] = blocks[d] if d < dim else 1
        c["n%d" % d] = blocks[d] * block[d] if d < dim else 1
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run: a check-out mesh of 16 x 16 elements, one schedule cycle
        # (L + N_p + 1 steps) and the state read back; launches and latency count
        _step("vortex16_fp64", 2, (2, 2), (8, 8), 2, "fp64", max_delay=2, steps=5),
        # the standard 2D production run, one schedule cycle, in each arithmetic
        _step("vortex256_fp64", 2, (8, 8), (32, 32), 4, "fp64", max_delay=3, steps=8),
        _step("vortex256_df64", 2, (8, 8), (32, 32), 4, "df64", max_delay=3, steps=8),
        _step("vortex256_fp32", 2, (8, 8), (32, 32), 4, "fp32", max_delay=3, steps=8),
        # a 2D mesh of odd extents with seeded random delays at every subdomain interface
        _step("random195x105_fp64", 2, (5, 3), (39, 35), 5, "fp64", delay_mode="random",
              random_delay_max=2, at_np=2, steps=4),
        # the 3D Taylor-Green production run, one schedule cycle: the largest case
        _step("tgv64_fp64", 3, (8, 8, 8), (8, 8, 8), 3, "fp64", max_delay=4, steps=8),
        # a 3D mesh of odd extents in the fast single-precision operator
        _step("tgv54x45x35_fp32", 3, (6, 5, 5), (9, 9, 7), 3, "fp32", max_delay=4, steps=8),
        # a short accuracy study as experiments.run_vortex does one: set the state (time
        # step from the CFL number), advance, check, L2 error and conserved totals
        _step("study64_fp64", 2, (16, 16), (4, 4), 2, "fp64", flux="std", max_delay=4,
              rk="rk33", steps=24, kind="study"),
        # the bare operator for a caller with a time integrator of its own
        _step("rhs45x36x27_fp64", 3, (1, 1, 1), (45, 36, 27), 2, "fp64", flux="sync",
              kind="rhs"),
        # many uneven instances advanced together (parameter sweep): 64 vortices
        {"name": "batch64_fp32", "kind": "batch", "count": 64, "mix": 7, "largest": 256,
         "precision": "fp32", "steps": 4},
        # the learned ghost-trace predictor in the solver, one schedule cycle
        _step("learned32_fp64", 3, (4, 4, 4), (8, 8, 8), 3, "fp64", flux="learned", max_delay=4,
              at_np=2, steps=7, kind="learned"),
        # one training step of the predictor at the batch size of learned.train
        {"name": "train65536", "kind": "train", "samples": 65536},
    ]


def _loguni(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(rng, dim, nodes, degree):
    """Subdomains and elements per subdomain for about `nodes` nodes, extents uneven."""
    elems = max(1.0, nodes / (degree + 1) ** dim)
    side = elems ** (1.0 / dim)
    stretch = [rng.uniform(0.75, 1.3) for _ in range(dim)]
    blocks, block = [], []
    for d in range(dim):
        n = max(2, int(side * stretch[d]))
        p = rng.choice([q for q in (1, 2, 3, 4, 5, 6, 8) if q <= max(1, n // 2)])
        blocks.append(p)
        block.append(max(1, n // p))
    return tuple(blocks), tuple(block)


def _rule(rng, degree):
    """Subdomain-face rule and schedule in the range in which the scheme is stable."""
    flux = rng.choice(["at", "at", "at", "std", "at_trace", "sync"])
    if flux == "sync":
        return {"flux": flux}, 4
    if rng.random() < 0.25:
        return {"flux": flux, "delay_mode": "random", "random_delay_max": rng.randint(1, 2),
                "at_np": min(degree, 2)}, 4
    np_ = degree if degree <= 4 else 2
    delay = rng.randint(1, 4) if degree <= 3 else rng.randint(1, 3)
    return {"flux": flux, "max_delay": delay, "at_np": np_}, delay + np_ + 1


def draw(rng):
    kind = rng.choice(["step2", "step2", "step2", "step2", "step3", "step3", "step3", "study",
                       "rhs", "batch", "learned", "train"])
    if kind == "train":
        return {"kind": "train", "samples": int(_loguni(rng, 1000, 200000))}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(6, 48), "mix": rng.randint(0, 10 ** 6),
                "largest": rng.choice([64, 128, 256]), "precision": rng.choice(["fp32", "fp64"]),
                "steps": rng.randint(1, 3)}
    precision = rng.choice(["fp64", "fp64", "df64", "fp32"])
    if kind == "study":
        degree = rng.randint(1, 3)
        blocks, block = _mesh(rng, 2, _loguni(rng, 4000, 400000), degree)
        rule, cycle = _rule(rng, degree)
        return _step(None, 2, blocks, block, degree, precision, steps=rng.randint(8, 24),
                     rk="rk22" if degree == 1 else "rk33", kind="study", **rule)
    if kind == "learned":
        degree = rng.randint(2, 4)
        blocks, block = _mesh(rng, 3, _loguni(rng, 30000, 2000000), degree)
        return _step(None, 3, tuple(max(2, b) for b in blocks), block, degree, "fp64",
                     flux="learned", max_delay=rng.randint(1, 4), at_np=2, steps=7, kind="learned")
    dim = 3 if kind == "step3" or (kind == "rhs" and rng.random() < 0.5) else 2
    degree = rng.randint(1, 5 if dim == 3 else 7)
    nodes = _loguni(rng, 20000, 9.0e6) if dim == 3 else _loguni(rng, 2000, 1.8e6)
    blocks, block = _mesh(rng, dim, nodes, degree)
    if kind == "rhs":
        return _step(None, dim, blocks, block, degree, precision, flux="sync", kind="rhs")
    rule, cycle = _rule(rng, degree)
    rk = "rk22" if degree == 1 and rng.random() < 0.4 else (
        "rk33" if degree in (2, 3) and rng.random() < 0.3 else "ck45")
    return _step(None, dim, blocks, block, degree, precision, rk=rk, steps=min(cycle, 8), **rule)


# ---- inputs ---------------------------------------------------------------------------

def _box(dim):
    return (((-5.0,) * 2, (5.0,) * 2) if dim == 2
            else ((0.0,) * 3, (2.0 * math.pi,) * 3))


def _extent(case):
    return tuple(case["n%d" % d] for d in range(case["dim"]))


def _coords(dim, n, degree, lo, hi):
    """Node coordinates per direction, broadcastable over [elements z.. x][nodes z.. x]."""
    xi = np.polynomial.legendre.leggauss(degree + 1)[0]
    out = []
    for d in range(dim):
        h = (hi[d] - lo[d]) / n[d]
        x = lo[d] + (np.arange(n[d])[:, None] + 0.5 * (xi[None, :] + 1.0)) * h
        shape = [1] * (2 * dim)
        shape[dim - 1 - d] = n[d]
        shape[2 * dim - 1 - d] = degree + 1
        out.append(torch.from_numpy(x.reshape(shape)).cuda())
    return out


def _vortex(n, degree, rng, lo=(-5.0, -5.0), hi=(5.0, 5.0)):
    """Isentropic vortex of random strength and centre, [4][elements][nodes]."""
    beta, x0, y0 = rng.uniform(1.0, 5.0), rng.uniform(-2.0, 2.0), rng.uniform(-2.0, 2.0)
    x, y = _coords(2, n, degree, lo, hi)
    Lx, Ly = hi[0] - lo[0], hi[1] - lo[1]
    dx, dy = x - x0, y - y0
    dx = dx - Lx * torch.floor(dx / Lx + 0.5)
    dy = dy - Ly * torch.floor(dy / Ly + 0.5)
    ex = torch.exp(1.0 - (dx * dx + dy * dy))
    u = 1.0 - beta * ex * dy / (2.0 * math.pi)
    v = beta * ex * dx / (2.0 * math.pi)
    g = GAMMA
    rho = (1.0 - (g - 1.0) / (16.0 * g * math.pi ** 2) * beta ** 2 * ex * ex) ** (1.0 / (g - 1.0))
    p = rho ** g
    w = torch.stack([rho, rho * u, rho * v, p / (g - 1.0) + 0.5 * rho * (u * u + v * v)])
    return w.reshape(4, n[0] * n[1], (degree + 1) ** 2).contiguous(), (beta, x0, y0)


def _taylor_green(n, degree, rng):
    """Taylor-Green vortex of random phase and Mach number near 0.1, [5][elements][nodes]."""
    lo, hi = _box(3)
    mach = rng.uniform(0.08, 0.12)
    x, y, z = (c + rng.uniform(0.0, 2.0 * math.pi) for c in _coords(3, n, degree, lo, hi))
    p0 = 1.0 / (GAMMA * mach ** 2)
    ux = torch.sin(x) * torch.cos(y) * torch.cos(z)
    uy = -torch.cos(x) * torch.sin(y) * torch.cos(z)
    p = p0 + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
    rho = p / p0
    w = torch.stack([rho, rho * ux, rho * uy, torch.zeros_like(rho),
                     p / (GAMMA - 1.0) + 0.5 * rho * (ux * ux + uy * uy)])
    return w.reshape(5, n[0] * n[1] * n[2], (degree + 1) ** 3).contiguous()


def _state(case, seed):
    rng = np.random.default_rng(seed)
    n = _extent(case)
    if case["dim"] == 2:
        return _vortex(n, case["degree"], rng)
    return _taylor_green(n, case["degree"], rng), None


def _solver(case):
    dim = case["dim"]
    lo, hi = _box(dim)
    return adg.Solver(dim=dim, n_elem=_extent(case), lo=lo, hi=hi, degree=case["degree"],
                      P=tuple(case["P%d" % d] for d in range(dim)), max_delay=case["max_delay"],
                      flux=case["flux"], rk=case["rk"], cfl=0.1, delay_mode=case["delay_mode"],
                      seed=20260301, random_delay_max=case["random_delay_max"],
                      at_np=case["at_np"], precision=case["precision"])


def _instances(case):
    """Uneven vortex instances: mesh, degree and largest delay drawn per instance."""
    rng = np.random.default_rng(case["mix"])
    sizes = [n for n in (32, 64, 128, 256) if n <= case["largest"]]
    return [dict(n_elem=(int(n), int(n)), degree=int(rng.integers(2, 6)), P=(8, 8),
                 max_delay=int(rng.integers(2, 5)))
            for n in rng.choice(sizes, size=case["count"])]


def _samples(case, seed):
    """Network inputs as the solver forms them (level differences over their spread, delay,
    stage offset) and targets within the accepted range."""
    n = case["samples"]
    rng = np.random.default_rng(seed)
    a = rng.uniform(-1.0, 1.0, n)
    b = (1.0 - np.abs(a)) * rng.choice([-1.0, 1.0], n)
    c = _rk("ck45")[2]
    x = np.stack([a, b, rng.integers(1, 5, n) / 8.0, np.asarray(c)[rng.integers(0, 5, n)]], 1)
    t = np.clip(0.4 * a * (1.0 + b) + 0.3 * rng.standard_normal(n), -2.0, 2.0)
    return x.astype(np.float32), t.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t = _samples(case, seed)
        return {"case": case, "trainer": learned.Trainer(learned.init_params(seed % 1000)),
                "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda()}
    if kind == "batch":
        insts = _instances(case)
        b = adg.Batch(insts, flux="at", rk="ck45", cfl=0.1, precision=case["precision"])
        b.autotune(trials=3)
        rng = np.random.default_rng(seed)
        out = []
        for i, q in enumerate(insts):
            u, _ = _vortex(q["n_elem"], q["degree"], rng)
            b.set_state(i, u)
            out.append(torch.empty_like(u))
        return {"case": case, "batch": b, "out": out}
    u, vortex = _state(case, seed)
    s = _solver(case)
    state = {"case": case, "solver": s, "u": u, "out": torch.empty_like(u), "vortex": vortex}
    if kind == "learned":
        s.set_learned_model(learned.load()[0], 1.0)
    if kind in ("step", "learned"):
        s.set_state(u)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        tr = state["trainer"]
        loss = tr.grad(state["x"], state["t"])
        tr.adam(1e-3)
        return {"loss": loss, "params": tr.p, "m": tr.m, "v": tr.v}
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        return [b.get_state(i, o) for i, o in enumerate(state["out"])]
    s = state["solver"]
    if kind == "rhs":
        return s.rhs(state["u"], state["out"])
    if kind == "study":
        s.set_state(state["u"])
        s.step(case["steps"])
        beta, x0, y0 = state["vortex"]
        return {"finite": s.check_finite(), "l2": s.l2_error_vortex(s.info()["t"], beta, x0, y0),
                "totals": s.conservation(), "state": s.get_state(state["out"])}
    s.step(case["steps"])
    return s.get_state(state["out"])


# ---- what a pass cannot do without ----------------------------------------------------

def _stage_work(dim, nodes, degree, stages, precision, steps):
    """Bytes and operations of `steps` time steps over `nodes` nodes: every stage reads and
    writes the solution (64 bits) and, between stages, the Runge-Kutta register."""
    n, nv = degree + 1, dim + 2
    reg = 4 if precision == "fp32" else 8
    per_dof = sum(16 + (reg if m > 0 else 0) + (reg if m < stages - 1 else 0)
                  for m in range(stages))
    flux = 19 if dim == 2 else 30
    per_node = flux + 2 * dim * n * nv + 4 * dim * nv + 5 * nv + 4 * dim * nv + 70 * dim / n
    return {"bytes": float(steps * per_dof * nodes * nv),
            "flops": float(steps * stages * nodes * per_node)}


def work(case):
    kind = case["kind"]
    if kind == "train":
        mac = 4 * 64 + 64 * 64 + 64
        return {"bytes": 20.0 * case["samples"] + 4545 * (4 * 8 + 2 * 2),
                "flops": float(case["samples"] * 6 * mac)}
    if kind == "batch":
        ws = [_stage_work(2, q["n_elem"][0] * q["n_elem"][1] * (q["degree"] + 1) ** 2, q["degree"],
                          5, case["precision"], case["steps"]) for q in _instances(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    nodes = math.prod(_extent(case)) * (case["degree"] + 1) ** case["dim"]
    if kind == "rhs":
        w = _stage_work(case["dim"], nodes, case["degree"], 1, case["precision"], 1)
        return w
    return _stage_work(case["dim"], nodes, case["degree"], RK_STAGES[case["rk"]],
                       case["precision"], case["steps"])


# ---- the same in plain 64-bit arithmetic ----------------------------------------------

def _rk(name):
    """(A, B, c, two_register) of a low-storage scheme."""
    if name == "ck45":
        a = [0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
             -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0]
        b = [1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
             1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
             2277821191437.0 / 14882151754819.0]
        c, y, q = [], 0.0, 0.0
        for am, bm in zip(a, b):
            c.append(y)
            q = am * q + 1.0
            y += bm * q
        return a, b, c, False
    if name == "rk22":
        a, b = [1.0, 0.0], [0.5, 0.5]
    else:
        a, b = [0.755726352, 0.386954477, 0.0], [0.245170287, 0.184896052, 0.569933661]
    c, y, r = [], 0.0, 0.0
    for am, bm in zip(a, b):
        c.append(r)
        r, y = y + am, y + bm
    return a, b, c, True


def _splitmix(x):
    m = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


class _Exact:
    """The method in float64 torch: state [variables][elements z.. x][nodes z.. x]."""

    def __init__(self, dim, n, degree, P, lo, hi, flux, rk, delay_mode="caa", max_delay=0,
                 random_delay_max=0, at_np=0, seed=20260301, model=None):
        N = degree + 1
        x, w = np.polynomial.legendre.leggauss(N)
        lam = np.array([1.0 / np.prod([x[j] - x[k] for k in range(N) if k != j]) for j in range(N)])
        D = np.zeros((N, N))  # D[a][i] = l_i'(x_a)
        for a in range(N):
            for i in range(N):
                if i != a:
                    D[a, i] = lam[i] / lam[a] / (x[a] - x[i])
            D[a, a] = -D[a].sum()
        at = lambda y: (lam / (y - x)) / (lam / (y - x)).sum()  # noqa: E731
        self.lp, self.lm = (torch.from_numpy(at(y)).cuda() for y in (1.0, -1.0))
        self.Q = torch.from_numpy((w[:, None] * D / w[None, :]).T.copy()).cuda()  # [i][a]
        self.w = torch.from_numpy(w).cuda()
        self.dim, self.n, self.N, self.P, self.flux = dim, n, N, P, flux
        self.h = [(hi[d] - lo[d]) / n[d] for d in range(dim)]
        self.degree, self.rk = degree, _rk(rk)
        self.L, self.np, self.random = max_delay, at_np or degree, delay_mode == "random"
        self.dmax, self.seed, self.model = random_delay_max, seed, model
        self.n_if = math.prod(P) * sum(1 for p in P if p > 1)
        self.ring = [[] for _ in range(dim)]  # newest first

    def view(self, u):
        d = self.dim
        return u.reshape((d + 2,) + tuple(self.n[::-1]) + (self.N,) * d)

    def flux_along(self, w, d):
        """Euler flux along d and |u|^2 + c^2."""
        dim = self.dim
        vel = w[1:1 + dim] / w[0]
        kin = (w[1:1 + dim] * vel).sum(0)
        p = (GAMMA - 1.0) * (w[dim + 1] - 0.5 * kin)
        f = w * vel[d]
        f[1 + d] += p
        f[dim + 1] += p * vel[d]
        return f, (kin + GAMMA * p) / w[0]

    def rusanov(self, wm, wp, d):
        fm, sm = self.flux_along(wm, d)
        fp, sp = self.flux_along(wp, d)
        lam = 0.5 * torch.sqrt(torch.maximum(sm, sp))
        return 0.5 * (fm + fp + lam * (wm - wp))

    def at_weights(self, km):
        return [math.prod((km + j) / (j - l) for j in range(self.np + 1) if j != l)
                for l in range(self.np + 1)]

    def extrapolate(self, d, off, km):
        """AT combination of the stored levels off, off + 1, ... for stage delay km."""
        if self.flux == "std":
            return self.ring[d][off]
        return sum(c * self.ring[d][off + l] for l, c in enumerate(self.at_weights(km)))

    def corrected(self, d, kt, cm, E):
        """The learned correction of extrapolated traces E (three stored levels)."""
        W1, b1, W2, b2, w3, b3 = self.model
        a0, a1, a2 = self.ring[d][:3]
        e = E - (a0 + (kt + cm) * (a0 - a1))
        s = (a0 - a1).abs() + (a1 - a2).abs()
        good = (e.abs() > 1e-9 * (a0.abs() + a1.abs() + a2.abs())) & (s > 1e-300)
        inv = torch.where(good, 1.0 / s, torch.zeros_like(s))
        x = torch.stack([(a0 - a1) * inv, (a1 - a2) * inv, torch.full_like(s, 0.125 * kt),
                         torch.full_like(s, cm)], -1)
        flat, y = x.reshape(-1, 4), []
        for q in flat.split(1 << 20):
            h = torch.tanh(q @ W1.T + b1)
            y.append(torch.tanh(h @ W2.T + b2) @ w3 + b3)
        y = torch.cat(y).reshape(s.shape)
        return torch.where(good & (y.abs() <= 1.0), E + e * y, E)

    def face_flux(self, u, d, step, stage, cm):
        """Numerical flux on the +d face of every element."""
        dim = self.dim
        ea, na = dim - d, 2 * dim - d  # element and node axis of direction d
        wm = torch.tensordot(u, self.lp, ([na], [0]))
        wp = torch.tensordot(u, self.lm, ([na], [0])).roll(-1, ea)
        f = self.rusanov(wm, wp, d)
        if self.flux == "sync" or self.P[d] == 1:
            return f
        b = self.n[d] // self.P[d]
        pe = torch.arange(b - 1, self.n[d], b, device=u.device)
        pick = lambda t, a=ea: t.index_select(a, pe)  # noqa: E731
        traces = self.flux in ("at_trace", "learned")
        comm, delay = True, {0}
        if self.random:
            off = sum(math.prod(self.P) for q in range(d) if self.P[q] > 1)
            sub = [torch.arange(self.P[q], device=u.device) for q in range(dim)]
            ids = torch.zeros([1] * dim, dtype=torch.int64, device=u.device)
            stride = 1
            for q in range(dim):
                # subdomain index along q of every element (of every face along d)
                v = sub[q] if q == d else sub[q].repeat_interleave(self.n[q] // self.P[q])
                shape = [1] * dim
                shape[dim - 1 - q] = -1
                ids = ids + v.reshape(shape) * stride
                stride *= self.P[q]
            kt_of = []
            for i in range(stride):
                kt = _splitmix(self.seed ^ (step * self.n_if + off + i)) % (self.dmax + 1)
                need = kt if self.flux == "std" else kt + self.np
                kt_of.append(0 if step - need < 0 else kt)
            kt_face = torch.tensor(kt_of, device=u.device)[ids]
            kt_face = kt_face.reshape((1,) + tuple(kt_face.shape) + (1,) * (dim - 1))
            delay = set(kt_of)
        elif self.flux == "std":
            k = step % self.L
            comm, delay = k == 0, {k}
        else:
            ph = step % (self.L + self.np + 1)
            comm = ph <= self.np
            delay = {0 if comm else ph - self.np}
        fresh = pick(f)
        if stage == 0 and (self.random or comm):
            self.ring[d].insert(0, torch.stack([pick(wm), pick(wp)]) if traces else fresh)
            del self.ring[d][self.dmax + self.np + 2:]
        out = fresh
        for kt in sorted(delay - {0}):
            v = self.extrapolate(d, kt if self.random else 0, kt + cm)
            if self.flux == "learned":
                v = self.corrected(d, kt, cm, v)
            if traces:
                v = self.rusanov(v[0], v[1], d)
            out = torch.where(kt_face == kt, v, out) if self.random else v
        return f.index_copy(ea, pe, out)

    def rhs(self, u, step=0, stage=0, cm=0.0):
        dim, k = self.dim, torch.zeros_like(u)
        for d in range(dim):
            ea, na = dim - d, 2 * dim - d
            F = self.flux_along(u, d)[0]
            k += 2.0 / self.h[d] * torch.tensordot(F, self.Q, ([na], [1])).movedim(-1, na)
            f = self.face_flux(u, d, step, stage, cm).unsqueeze(na)
            shape = [1] * (2 * dim + 1)
            shape[na] = self.N
            k -= 2.0 / self.h[d] * f * (self.lp / self.w).reshape(shape)
            k += 2.0 / self.h[d] * f.roll(1, ea) * (self.lm / self.w).reshape(shape)
        return k

    def time_step(self, u, cfl):
        dim = self.dim
        vel = u[1:1 + dim] / u[0]
        p = (GAMMA - 1.0) * (u[dim + 1] - 0.5 * (u[1:1 + dim] * vel).sum(0))
        smax = (torch.sqrt((vel * vel).sum(0)) + torch.sqrt(GAMMA * p / u[0])).max()
        return cfl * min(self.h) / ((2 * self.degree + 1) * float(smax))

    def advance(self, u, dt, steps):
        a, b, c, two_r = self.rk
        w = u
        for n in range(steps):
            x, q = w, None
            for m in range(len(a)):
                k = self.rhs(x, n, m, c[m])
                if two_r:
                    x = w + dt * a[m] * k
                    w = w + dt * b[m] * k
                else:
                    q = dt * k if q is None else a[m] * q + dt * k
                    w = w + b[m] * q
                    x = w
        return w

    def l2_vortex(self, u, t, beta, x0, y0, lo, hi):
        """L2 errors against the translated vortex with degree + 2 Gauss points."""
        xe, we = np.polynomial.legendre.leggauss(self.N + 1)
        x = np.polynomial.legendre.leggauss(self.N)[0]
        I = np.array([[np.prod([(y - x[k]) / (x[j] - x[k]) for k in range(self.N) if k != j])
                       for j in range(self.N)] for y in xe])
        I = torch.from_numpy(I).cuda()
        uh = torch.einsum("vyxba,qb,pa->vyxqp", u, I, I)
        pts = [torch.from_numpy(lo[d] + (np.arange(self.n[d])[:, None] + 0.5 * (xe + 1)) * self.h[d]).cuda()
               for d in range(2)]
        X, Y = pts[0][None, :, None, :], pts[1][:, None, :, None]
        Lx, Ly = hi[0] - lo[0], hi[1] - lo[1]
        dx, dy = X - (x0 + t), Y - y0
        dx = dx - Lx * torch.floor(dx / Lx + 0.5)
        dy = dy - Ly * torch.floor(dy / Ly + 0.5)
        ex, g = torch.exp(1.0 - (dx * dx + dy * dy)), GAMMA
        vx, vy = 1.0 - beta * ex * dy / (2 * math.pi), beta * ex * dx / (2 * math.pi)
        rho = (1 - (g - 1) / (16 * g * math.pi ** 2) * beta ** 2 * ex * ex) ** (1 / (g - 1))
        E = rho ** g / (g - 1) + 0.5 * rho * (vx * vx + vy * vy)
        W = torch.from_numpy(np.outer(we, we)).cuda() * self.h[0] * self.h[1] / 4
        d = [uh[0] - rho, uh[1] - rho * vx, uh[2] - rho * vy, uh[3] - E]
        sq = [(W * d[0] ** 2).sum(), (W * (d[1] ** 2 + d[2] ** 2)).sum(), (W * d[3] ** 2).sum()]
        return torch.stack(sq).sqrt().cpu().numpy()

    def totals(self, u):
        W = torch.einsum("b,a->ba", self.w, self.w) * self.h[0] * self.h[1] / 4
        return (u * W).sum((1, 2, 3, 4)).cpu().numpy()


def _mlp(params):
    p = params.to(torch.bfloat16).double()
    return (p[:256].reshape(64, 4), p[256:320], p[320:4416].reshape(64, 64), p[4416:4480],
            p[4480:4544], p[4544])


def _exact_train(case, seed):
    x, t = _samples(case, seed)
    p = torch.from_numpy(learned.init_params(seed % 1000)).cuda()
    W1, b1, W2, b2, w3, b3 = _mlp(p)
    X, T = torch.from_numpy(x).cuda().double(), torch.from_numpy(t).cuda().double()
    h1 = torch.tanh(X @ W1.T + b1)
    h2 = torch.tanh(h1 @ W2.T + b2)
    r = h2 @ w3 + b3 - T
    dy = 2.0 * r / len(r)
    dz2 = torch.outer(dy, w3) * (1 - h2 * h2)
    dz1 = (dz2 @ W2) * (1 - h1 * h1)
    g = torch.cat([(dz1.T @ X).reshape(-1), dz1.sum(0), (dz2.T @ h1).reshape(-1), dz2.sum(0),
                   h2.T @ dy, dy.sum().reshape(1)])
    m, v = 0.1 * g, 0.001 * g * g
    new = p.double() - 1e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"loss": (r * r).mean().reshape(1), "params": new, "m": m, "v": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "batch":
        rng = np.random.default_rng(seed)
        out = []
        for q in _instances(case):
            u, _ = _vortex(q["n_elem"], q["degree"], rng)
            e = _Exact(2, q["n_elem"], q["degree"], q["P"], *_box(2), "at", "ck45",
                       max_delay=q["max_delay"])
            w = e.view(u)
            out.append(e.advance(w, e.time_step(w, 0.1), case["steps"]).reshape(u.shape))
        return out
    u, vortex = _state(case, seed)
    dim, (lo, hi) = case["dim"], _box(case["dim"])
    model = None
    if kind == "learned":
        bits = torch.from_numpy(learned.load()[0].view(np.int16).copy()).cuda()
        model = _mlp(bits.view(torch.bfloat16).float())
    e = _Exact(dim, _extent(case), case["degree"], tuple(case["P%d" % d] for d in range(dim)), lo, hi,
               case["flux"], case["rk"], case["delay_mode"], case["max_delay"],
               case["random_delay_max"], case["at_np"], model=model)
    w = e.view(u)
    if kind == "rhs":
        return e.rhs(w).reshape(u.shape)
    dt = e.time_step(w, 0.1)
    w = e.advance(w, dt, case["steps"])
    if kind == "study":
        beta, x0, y0 = vortex
        return {"finite": None, "l2": e.l2_vortex(w, dt * case["steps"], beta, x0, y0, lo, hi),
                "totals": e.totals(w), "state": w.reshape(u.shape)}
    return w.reshape(u.shape)
