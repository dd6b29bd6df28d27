"""Performance cases: the work a user has the library do, through its public entry points.

A case is a dict of plain values.  Its ``kind`` names the entry point:

  residual   Solver.residual, one evaluation of the right-hand side (dV/dt and E)
  solver     Solver.set_state / advance / get_state_device, one instance
  batch      Batch.set_state / advance / get_state_device, many instances with tuned launch shapes
  implicit   Implicit.set_state / run / get_state, the 1D backward-Euler Newton integrator
  newton     Newton.run, 1D/2D backward Euler with the Newton-Krylov solve

and its ``problem`` the flow: the dam breaks, the bump, the slump, the dry bed and the mixed ensemble of the
benchmark.  Meshes and parameters belong to the case; depths and velocities come from the seed: the problem's
initial state plus smooth seeded perturbations, so that the flow moves, yields in places and differs by seed.

FP32 contexts hold FP32 values; their outputs are returned in that type.

``exact`` solves the same discrete equations in 64 bits with plain torch: weak form on elements, every face seen
from both sides, dense algebra, no code of the library.
"""
import math

import numpy as np
import torch

import paper_2301_11238_gb300 as G

COPY, DIRICHLET, WALL = 0, 1, 2
NEWTON_KW = dict(rtol=1e-10, atol=1e-11, krylov_dim=30, krylov_rtol=1e-4)


def listed():
    return [
        # the smallest run: 200 intervals, a few hundred degrees of freedom; latency and launches are all of it
        dict(name="dam1d", kind="solver", problem="dam1d", n=200, order=1, fp32=False, steps=64),
        # one right-hand side of a small 2D mesh, as a caller's own time integrator evaluates it
        dict(name="residual", kind="residual", problem="radial", n=64, order=2, fp32=False),
        # a parameter sweep (3 yield stresses x 3 regularizations) of the radial dam break in one batch
        dict(name="sweep_f64", kind="batch", problem="radial", n=64, order=2, fp32=False, instances=9, steps=4),
        dict(name="sweep_f32", kind="batch", problem="radial", n=64, order=2, fp32=True, instances=9, steps=16),
        # dam break over a bump on a jittered mesh, the highest order, one context
        dict(name="bump_f32", kind="solver", problem="bump", n=512, order=3, fp32=True, steps=4),
        # ragged sizes, 1D and 2D and all orders mixed, in one batch
        dict(name="ensemble_f32", kind="batch", problem="ensemble", n=16, order=0, fp32=True, instances=32, steps=16),
        # large Bingham slump over a rough bed: the benchmark's workload, FP64 and FP32
        dict(name="slump_f64", kind="batch", problem="slump", n=512, order=2, fp32=False, instances=1, steps=2),
        dict(name="slump_f32", kind="batch", problem="slump", n=1024, order=2, fp32=True, instances=1, steps=4),
        # dam break onto a dry bed: wet/dry stages with the depth limiter
        dict(name="drybed_f64", kind="batch", problem="dry", n=512, order=1, fp32=False, instances=1, steps=4),
        # the paper's own integrator and test: 100 intervals, constant E per element, dt = 1e-6
        dict(name="implicit_dam", kind="implicit", problem="paperdam", n=100, order=1, m3=0, mixed=False, steps=20),
        # one backward-Euler step of the 2D radial dam break, ten times the explicit step
        dict(name="newton2d", kind="newton", problem="radial_tanh", n=64, order=2, dt_factor=10.0, steps=1),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["dam1d", "residual", "sweep", "bump", "ensemble", "slump", "dry", "implicit", "newton"])
    order = rng.randint(1, 3)
    if kind == "dam1d":
        return dict(kind="solver", problem="dam1d", n=log_int(50, 20000), order=order, fp32=rng.random() < 0.3,
                    steps=rng.choice([16, 40, 64]))
    if kind == "residual":
        return dict(kind="residual", problem=rng.choice(["radial", "bump"]), n=log_int(8, 256), order=order, fp32=False)
    if kind == "sweep":
        return dict(kind="batch", problem="radial", n=log_int(12, 96), order=order, fp32=rng.random() < 0.5,
                    instances=rng.randint(2, 9), steps=rng.choice([2, 4, 5]))
    if kind == "bump":
        return dict(kind="solver", problem="bump", n=log_int(48, 400), order=order, fp32=rng.random() < 0.8, steps=2)
    if kind == "ensemble":
        return dict(kind="batch", problem="ensemble", n=rng.randint(17, 9999), order=0, fp32=rng.random() < 0.8,
                    instances=rng.randint(4, 28), steps=rng.choice([4, 16]))
    if kind == "slump":
        fp32 = rng.random() < 0.5
        return dict(kind=rng.choice(["batch", "solver"]), problem="slump", n=log_int(100, 900 if fp32 else 400),
                    order=rng.choice([1, 2, 2]), fp32=fp32, instances=1, steps=rng.choice([1, 2]))
    if kind == "dry":
        return dict(kind=rng.choice(["batch", "solver"]), problem="dry", n=log_int(40, 500), order=1, fp32=False,
                    instances=1, steps=rng.choice([1, 2, 4]))
    if kind == "implicit":
        p = rng.randint(1, 2)
        return dict(kind="implicit", problem="paperdam", n=log_int(20, 150), order=p, m3=rng.randint(0, p),
                    mixed=rng.random() < 0.5, steps=rng.randint(3, 15))
    return dict(kind="newton", problem="radial_tanh", n=log_int(8, 72), order=order,
                dt_factor=round(rng.uniform(2.0, 20.0), 2), steps=1)


# ------------------------------------------------------------------ meshes, parameters, states


def _bc(modes=(), values=()):
    m, v = [COPY] * 7, [0.0] * 7
    for slot, x in modes:
        m[slot] = x
    for slot, x in values:
        v[slot] = x
    return m, v


def _interval(n, length):
    x = np.linspace(0.0, length, n + 1)
    etov = np.stack([np.arange(n), np.arange(1, n + 1)], axis=1).astype(np.int32)
    tags = np.zeros((n, 2), dtype=np.int8)
    tags[:, 1] = 1
    return x.reshape(-1, 1), etov, tags


def _square(n, jitter=0.0):
    """[-1, 1]^2 in n x n squares, each cut into two counter-clockwise triangles."""
    xs = np.linspace(-1.0, 1.0, n + 1)
    X, Y = np.meshgrid(xs, xs, indexing="xy")
    coords = np.stack([X.ravel(), Y.ravel()], axis=1)
    if jitter:
        d = np.random.default_rng(3).uniform(-jitter, jitter, size=coords.shape) * (2.0 / n)
        inner = (np.abs(coords) < 1.0 - 1e-12).all(axis=1)
        coords[inner] += d[inner]
    i, j = np.tile(np.arange(n), n), np.repeat(np.arange(n), n)
    a = j * (n + 1) + i
    etov = np.empty((2 * n * n, 3), dtype=np.int32)
    etov[0::2] = np.stack([a, a + 1, a + n + 2], axis=1)
    etov[1::2] = np.stack([a, a + n + 2, a + n + 1], axis=1)
    return coords, etov, np.zeros((2 * n * n, 3), dtype=np.int8)


def _waves(seed, dim, amp, modes=3, kmax=3.0):
    """A smooth function of the points x (..., dim): a seeded sum of low-wavenumber sinusoids, at most amp."""
    r = np.random.default_rng(seed)
    k, ph, a = r.uniform(-kmax, kmax, (modes, dim)), r.uniform(0, 2 * math.pi, modes), r.uniform(0.3, 1.0, modes)

    def f(x):
        out = torch.zeros(x.shape[:-1], dtype=torch.float64, device=x.device)
        for m in range(modes):
            arg = sum(float(k[m, d]) * x[..., d] for d in range(dim)) + float(ph[m])
            out = out + float(a[m]) * torch.sin(arg)
        return out * (amp / float(a.sum()))

    return f


def _params(**kw):
    p = dict(g=9.81, rho=1.0, alpha=0.0, eta=0.01, sigma0=0.0, gamma=1e3, beta=1e3, pap_m=1e3, h_floor=1e-6, cfl=0.3,
             reg=0, positivity=0)
    p.update(kw)
    return p


class _Instance:
    """One instance of a problem: mesh, order, parameters, boundaries, bed, and the initial state for a seed."""

    def __init__(self, problem, n, order, which=0, dim=2, m3=-1):
        self.order, self.m3, self.bcs, self.bed_fn = order, m3, [_bc()], None
        self.dam = lambda c: torch.ones_like(c[..., 0])
        wave = 0.05
        if problem == "dam1d":
            self.mesh = _interval(n, 1.0)
            self.bcs = [_bc(), _bc()]
            self.prm = _params(reg=4, sigma0=0.05)
            self.dam = lambda c: torch.where(c[..., 0] < 0.5, 1.0, 0.5).double()
        elif problem == "paperdam":
            self.mesh = _interval(n, 3.0)
            self.prm = _params(reg=1, sigma0=0.2, eta=0.02, gamma=1e2, beta=1e2)
            self.bcs = [_bc([(0, DIRICHLET), (2, DIRICHLET)], [(0, h)]) for h in (1.5, 0.5)]
            self.dam = lambda c: torch.where(c[..., 0] < 1.5, 1.5, 0.5).double()
        elif problem in ("radial", "radial_tanh"):
            self.mesh = _square(n)
            s0, reg = (0.02, 3) if problem == "radial_tanh" else ((0.0, 0.02, 0.1)[which // 3 % 3], 1 + which % 3)
            self.prm = _params(reg=reg, sigma0=s0, gamma=50.0 if problem == "radial_tanh" else 1e3)
            self.dam = lambda c: torch.where(c[..., 0] ** 2 + c[..., 1] ** 2 < 0.09, 2.0, 0.5).double()
        elif problem == "bump":
            self.mesh = _square(n, jitter=0.1)
            self.prm = _params(reg=3, sigma0=0.05)
            self.bed_fn = lambda x: 0.2 * torch.exp(-(x[..., 0] ** 2 + x[..., 1] ** 2) / (2 * 0.1 ** 2))
            self.dam = lambda c: torch.where(c[..., 0] < -0.5, 1.0, 0.5).double()
        elif problem == "slump":
            self.mesh = _square(n)
            self.prm = _params(reg=5, sigma0=0.05, alpha=math.atan(0.05))
            self.bed_fn = _waves(5, 2, 0.05, modes=16, kmax=4 * math.pi)
        elif problem == "dry":
            self.mesh = _square(n)
            self.prm = _params(eta=0.0, positivity=1)
            self.bcs = [_bc([(1, WALL), (2, WALL)])]
            self.dam = lambda c: torch.where(c[..., 0] < 0.0, 1.0, 0.0).double()
            wave = 0.1
        elif problem == "ensemble":
            r = np.random.default_rng([n, which])
            k = int(round(math.exp(r.uniform(math.log(1000), math.log(50000)))))
            dim, self.order = int(r.integers(1, 3)), int(r.integers(1, 4))
            s0, hl = float(math.exp(r.uniform(math.log(1e-3), math.log(0.2)))), 0.5 * float(r.uniform(1.5, 4.0))
            self.mesh = _interval(k, 1.0) if dim == 1 else _square(max(2, int(round(math.sqrt(k / 2)))))
            self.bcs = [_bc(), _bc()]
            self.prm = _params(reg=1 + which % 3, sigma0=s0)
            x_dam = 0.5 if dim == 1 else 0.0
            self.dam = lambda c: torch.where(c[..., 0] < x_dam, hl, 0.5).double()
        else:
            raise ValueError(problem)
        self.problem, self.wave = problem, wave
        self.dim = self.mesh[0].shape[1]

    def points(self, ref, device):
        """Physical positions (K, len(ref), dim) of reference points, and each element's centroid (K, 1, dim)."""
        v = torch.from_numpy(self.mesh[0]).to(device)[torch.from_numpy(self.mesh[1]).to(device).long()]
        lam = 0.5 * (1.0 + torch.as_tensor(ref, dtype=torch.float64, device=device).reshape(-1, self.dim))
        x = v[:, :1] + sum(lam[None, :, d:d + 1] * (v[:, d + 1:d + 2] - v[:, :1]) for d in range(self.dim))
        return x, v.mean(dim=1, keepdim=True)

    def state(self, seed, device):
        """Nodal (h, u_1[, u_2]) of shape (1 + dim, K, Np)."""
        x, c = self.points(_nodes(self.dim, self.order), device)
        h = self.dam(c.expand_as(x)) * (1.0 + _waves(seed, self.dim, self.wave)(x))
        if self.bed_fn is not None and self.problem == "bump":
            h = h - self.bed_fn(x)
        if self.problem == "slump":
            h = torch.clamp(h * torch.exp(-(x[..., 0] ** 2 + x[..., 1] ** 2) / (2 * 0.15 ** 2)), min=1e-3)
        u = [_waves(seed + 1000003 * (d + 1), self.dim, self.wave)(x) for d in range(self.dim)]
        wet = (h > 0).to(torch.float64)
        return torch.stack([h] + [ud * wet for ud in u]).contiguous()

    def bed(self, device):
        if self.bed_fn is None:
            return None
        return self.bed_fn(self.points(_nodes(self.dim, self.order), device)[0])

    def spec(self):
        bed = self.bed("cuda")
        return dict(dim=self.dim, coords=self.mesh[0], etov=self.mesh[1], order=self.order, reg=self.prm["reg"],
                    prm=self.prm, face_bc=self.mesh[2], bcs=self.bcs, bed=None if bed is None else bed.cpu().numpy())


def _instances(case):
    if case["kind"] == "batch":
        return [_Instance(case["problem"], case["n"], case["order"], which=i) for i in range(case["instances"])]
    return [_Instance(case["problem"], case["n"], case["order"], which=4, m3=case.get("m3", -1))]


# ------------------------------------------------------------------ the library's side


def prepare(case, seed):
    inst = _instances(case)
    s = dict(case=case)
    if case["kind"] == "implicit":
        i = inst[0]
        s["V"] = [i.state(seed, "cpu").numpy()]
        s["h"] = G.Implicit(i.mesh[0], i.mesh[1], i.order, i.prm["reg"], i.prm, 1e-6, m3=i.m3, face_bc=i.mesh[2],
                            bcs=i.bcs, mixed=case["mixed"])
        return s
    prec = G.PREC_FP32 if case.get("fp32") else G.PREC_FP64
    s["V"] = [i.state(seed + 7919 * k, "cuda") for k, i in enumerate(inst)]
    s["out"] = [torch.empty_like(v) for v in s["V"]]
    if case["kind"] == "batch":
        s["h"] = G.Batch([i.spec() for i in inst], precision=prec)
        for k, v in enumerate(s["V"]):
            s["h"].set_state(k, v)
        s["h"].autotune(5)
        return s
    sp = inst[0].spec()
    s["h"] = G.Solver(sp["dim"], sp["coords"], sp["etov"], sp["order"], sp["reg"], sp["prm"], face_bc=sp["face_bc"],
                      bcs=sp["bcs"], bed=sp["bed"], precision=prec)
    if case["kind"] == "newton":
        dt = case["dt_factor"] * float(_Exact(inst[0], "cuda").step_bound(s["V"][0]))
        s["newton"] = G.Newton(s["h"], dt, **NEWTON_KW)
    return s


def run(s):
    case, h = s["case"], s["h"]
    if case["kind"] == "residual":
        return h.residual(s["V"][0])
    if case["kind"] == "implicit":
        h.set_state(s["V"][0])
        h.run(case["steps"])
        return h.get_state()
    if case["kind"] == "batch":
        for k, v in enumerate(s["V"]):
            h.set_state(k, v)
        h.advance(case["steps"])
        for k, o in enumerate(s["out"]):
            h.get_state_device(k, o)
    else:
        h.set_state(s["V"][0])
        if case["kind"] == "newton":
            s["newton"].run(case["steps"])
        else:
            h.advance(case["steps"])
        h.get_state_device(s["out"][0])
    return [o.float() for o in s["out"]] if case.get("fp32") else list(s["out"])


def work(case):
    """State in, state out and the mesh once; the arithmetic of every right-hand side of the pass."""
    size = 4 if case.get("fp32") else 8
    total_b = total_f = 0.0
    for i in _instances(case):
        d, p, K = i.dim, i.order, i.mesh[1].shape[0]
        Np = p + 1 if d == 1 else (p + 1) * (p + 2) // 2
        nq = ((3 * p + 1) // 2) ** d
        nfp, nfq = (1, 1) if d == 1 else (p + 1, (3 * p + 2) // 2)
        nV, nE, nf = d + 1, d * d, d + 1
        estep = 2 * d * d * Np * Np + 2 * nE * d * Np + nf * (nfp * (d + 1) + Np * d * 2 * (nfp + d))
        face = nf / 2 * nfq * (4 * nfp * (nV + nE) + 90)
        vol = nq * (2 * Np * (nV + nE) + 45 + 2 * Np * (nV * d + d)) + nf * 2 * nfp * nfq * nV
        mass = 2 * Np * Np + nq * (2 * Np + Np * (Np + 1) + 2 * d * Np) + Np ** 3 / 3 + 2 * d * Np * Np
        rhs = K * (estep + face + vol + mass)
        # residual evaluations: three per explicit step; per implicit step about two Newton iterations of one
        # (1D, with its block-tridiagonal solve) or of five (Newton-Krylov)
        evals = {"residual": 1, "solver": 3, "batch": 3, "implicit": 2, "newton": 14}[case["kind"]]
        solve = 0.0
        if case["kind"] == "implicit":
            nb = 2 * Np + case["m3"] + 1
            solve = 2 * K * (2 * nb ** 3 / 3 + 4 * nb ** 3)
        total_f += case.get("steps", 1) * (evals * rhs + solve)
        mesh = K * (size * (7 + nf * (d + 1)) + 4 * nf) + (K * Np * size if i.bed_fn is not None else 0)
        total_b += mesh + 8 * K * Np * nV + size * K * Np * nV + (8 * K * Np * nE if case["kind"] == "residual" else 0)
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------ the same equations in plain torch, 64 bits


def _nodes(dim, p):
    if dim == 1:
        return np.array([[-1.0 + 2.0 * i / p] for i in range(p + 1)]) if p else np.zeros((1, 1))
    return np.array([[-1.0 + 2.0 * i / p, -1.0 + 2.0 * j / p] for j in range(p + 1) for i in range(p + 1 - j)])


def _gauss(n, a):
    """Gauss-Jacobi rule of weight (1 - x)^a on [-1, 1], a in {0, 1} (Golub-Welsch)."""
    k = np.arange(n, dtype=np.float64)
    if a == 0:
        x, w = np.polynomial.legendre.leggauss(n)
        return x, w
    diag = -1.0 / ((2 * k + 1) * (2 * k + 3))
    k = k[1:]
    off = np.sqrt(k * (k + 1)) / (2 * k + 1)
    x, v = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return x, 2.0 * v[0] ** 2


def _basis(dim, p, pts):
    """Lagrange basis of the equispaced nodes at pts: values (n, Np) and reference derivatives (dim, n, Np)."""
    ex = [(i,) for i in range(p + 1)] if dim == 1 else [(i, j) for j in range(p + 1) for i in range(p + 1 - j)]
    pts = np.asarray(pts, dtype=np.float64).reshape(-1, dim)

    def mono(x, der=None):
        cols = []
        for e in ex:
            c = np.ones(len(x))
            for d in range(dim):
                n = e[d]
                c = c * ((n * x[:, d] ** (n - 1) if n else 0.0 * x[:, d]) if d == der else x[:, d] ** n)
            cols.append(c)
        return np.stack(cols, axis=1)

    inv = np.linalg.inv(mono(_nodes(dim, p)))
    return mono(pts) @ inv, np.stack([mono(pts, d) @ inv for d in range(dim)])


class _Exact:
    """The DG scheme of one instance: E from the velocity, the residual, the mass solve, and its integrators."""

    def __init__(self, inst, device):
        self.i, self.dim, self.p = inst, inst.dim, inst.order
        self.m3 = self.p if inst.m3 < 0 else inst.m3
        d, p, dev = self.dim, self.p, device

        def t(x):
            return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=dev)

        nq, nfq = (3 * p + 1) // 2, (3 * p + 2) // 2
        a, wa = _gauss(nq, 0)
        if d == 1:
            pts, w = a[:, None], wa
            face_pts, wf = [np.array([[-1.0]]), np.array([[1.0]])], np.array([1.0])
        else:
            b, wb = _gauss(nq, 1)
            pts = np.array([[0.5 * (1 + x) * (1 - y) - 1, y] for x in a for y in b])
            w = np.array([0.5 * x * y for x in wa for y in wb])
            s, wf = _gauss(nfq, 0)
            one = np.ones_like(s)
            face_pts = [np.stack([s, -one], 1), np.stack([-s, s], 1), np.stack([-one, -s], 1)]
        B, D = _basis(d, p, pts)
        self.B, self.D, self.w, self.wf = t(B), t(D), t(w), t(wf)
        self.Bf = t(np.stack([_basis(d, p, q)[0] for q in face_pts]))  # (face, point, node)
        BE, DE = _basis(d, self.m3, pts)
        self.BE, self.DE = t(BE), t(DE)
        self.BEf = t(np.stack([_basis(d, self.m3, q)[0] for q in face_pts]))
        self.Minv = torch.linalg.inv(t((B * w[:, None]).T @ B))
        self.MEinv = torch.linalg.inv(t((BE * w[:, None]).T @ BE))
        self.avg = t((B * w[:, None]).sum(0) / w.sum())
        # geometry
        v = torch.from_numpy(inst.mesh[0]).to(dev)[torch.from_numpy(inst.mesh[1]).to(dev).long()]
        if d == 1:
            J = 0.5 * (v[:, 1, 0] - v[:, 0, 0])
            self.G = (1.0 / J)[:, None, None]
            self.n = t([[[-1.0], [1.0]]]).expand(len(J), 2, 1)
            self.sJ = torch.ones(len(J), 2, dtype=torch.float64, device=dev)
            self.dx = 2.0 * J
        else:
            r, s = 0.5 * (v[:, 1] - v[:, 0]), 0.5 * (v[:, 2] - v[:, 0])
            J = r[:, 0] * s[:, 1] - s[:, 0] * r[:, 1]
            self.G = torch.stack([torch.stack([s[:, 1], -s[:, 0]], 1), torch.stack([-r[:, 1], r[:, 0]], 1)], 1) / J[:, None, None]
            e = torch.roll(v, -1, dims=1) - v
            length = e.norm(dim=2)
            self.n = torch.stack([e[..., 1], -e[..., 0]], 2) / length[..., None]
            self.sJ, self.dx = 0.5 * length, 8.0 * J / length.sum(1)
        self.J = J
        self._connect(inst, dev)
        bed = inst.bed(dev)
        self.dH = None if bed is None else torch.einsum("kri,rqk->kqi", self.G, torch.einsum("rqa,ka->rqk", self.D, bed))
        c = inst.prm
        self.gc, self.gs = c["g"] * math.cos(c["alpha"]), c["g"] * math.sin(c["alpha"])

    def _connect(self, inst, dev):
        """Flat index (element * faces + face) of each face's other side (its own at the boundary)."""
        etov, tags = inst.mesh[1].astype(np.int64), inst.mesh[2]
        K, nf = etov.shape
        if self.dim == 1:
            key = etov.reshape(-1)
        else:
            a, b = etov.reshape(-1), np.roll(etov, -1, axis=1).reshape(-1)
            key = np.minimum(a, b) * (etov.max() + 1) + np.maximum(a, b)
        order = np.argsort(key, kind="stable")
        same = key[order][1:] == key[order][:-1]
        other = np.arange(K * nf)
        l, r = order[:-1][same], order[1:][same]
        other[l], other[r] = r, l
        self.other = torch.from_numpy(other).to(dev)
        rim = other == np.arange(K * nf)
        self.rim = torch.from_numpy(rim).to(dev).reshape(K, nf, 1)
        modes = np.array([b[0] for b in inst.bcs])[tags.reshape(-1)].reshape(K, nf, 1, 7)
        vals = np.array([b[1] for b in inst.bcs])[tags.reshape(-1)].reshape(K, nf, 1, 7)
        self.modes, self.vals = torch.from_numpy(modes).to(dev), torch.from_numpy(vals).to(dev)

    # ---- pieces of the scheme
    def _sides(self, tr, slot, wall=False):
        """Exterior values of traces tr (K, faces, points): the neighbour's, or the ghost value of the slot."""
        K, nf, m = tr.shape
        ext = torch.flip(tr.reshape(K * nf, m)[self.other], dims=[1]).reshape(K, nf, m)
        ghost = torch.where(self.modes[..., slot] == DIRICHLET, self.vals[..., slot], tr)
        return torch.where(self.rim, ghost, ext)

    def _vel_sides(self, um):
        up = [self._sides(u, 1 + j) for j, u in enumerate(um)]
        wall = self.rim & (self.modes[..., 1:1 + self.dim] == WALL).any(-1)
        un = sum(u * self.n[:, :, None, j] for j, u in enumerate(um))
        return [torch.where(wall, u - 2.0 * un * self.n[:, :, None, j], x) for j, (u, x) in enumerate(zip(um, up))]

    def gradient(self, V):
        """E[dim * i + j] = d u_j / d x_i, weakly with central fluxes: (nE, K, NpE)."""
        d = self.dim
        um = [torch.einsum("fma,ka->kfm", self.Bf, V[1 + j]) for j in range(d)]
        up = self._vel_sides(um)
        DEx = torch.einsum("kri,rqc,q->kiqc", self.G, self.DE, self.w)
        out = []
        for i in range(d):
            for j in range(d):
                g = 0.5 * (um[j] + up[j]) * self.n[:, :, None, i] * self.sJ[:, :, None] * self.wf
                r = torch.einsum("kfm,fmc->kc", g, self.BEf) / self.J[:, None]
                r = r - torch.einsum("kqc,kq->kc", DEx[:, i], V[1 + j] @ self.B.T)
                out.append(r @ self.MEinv.T)
        return torch.stack(out)

    def _stress(self, E):
        """sigma[i][j] of the gradient components E (list of nE tensors)."""
        c, d = self.i.prm, self.dim
        if d == 1:
            D = [[E[0]]]
            s2 = E[0] ** 2
        else:
            d12 = 0.5 * (E[1] + E[2])
            D = [[E[0], d12], [d12, E[3]]]
            s2 = 0.5 * (E[0] ** 2 + 2 * d12 ** 2 + E[3] ** 2 + (E[0] + E[3]) ** 2)
        s0, g, reg = c["sigma0"], c["gamma"], c["reg"]
        pos = s2 > 0
        s = torch.where(pos, torch.sqrt(torch.where(pos, s2, torch.ones_like(s2))), torch.zeros_like(s2))
        safe = torch.where(pos, s, torch.ones_like(s))
        coef = torch.zeros_like(s)
        if s0 > 0:
            e = 0.5 / c["beta"]
            if reg == 1:
                x = g * s - s0
                mb = torch.where(x >= e, x, torch.where(x <= -e, torch.zeros_like(x), 0.5 * c["beta"] * (x + e) ** 2))
                coef = s0 * g / (mb + s0)
            elif reg == 2:
                x = g * s
                mid = (2 * s0 - c["beta"] * (s0 - x + e) ** 2) / (2 * safe)
                coef = torch.where(x >= s0 + e, s0 / safe, torch.where(x <= s0 - e, torch.full_like(x, g), mid))
            elif reg == 3:
                coef = torch.where(g * s < 1e-8, torch.full_like(s, s0 * g), s0 * torch.tanh(g * s) / safe)
            elif reg == 4:
                x = c["pap_m"] * s
                coef = torch.where(x < 1e-12, torch.full_like(s, s0 * c["pap_m"]), -s0 * torch.expm1(-x) / safe)
            elif reg == 5:
                coef = torch.where(g * s < s0, torch.full_like(s, g), s0 / safe)
        mu = 2 * c["eta"] + coef
        tr = sum(D[k][k] for k in range(d))
        return [[mu * (D[i][j] + (tr if i == j else 0.0)) for j in range(d)] for i in range(d)]

    def residual(self, V, E):
        """r_V of the weak form, (nV, K, Np)."""
        d, c = self.dim, self.i.prm
        Q = [v @ self.B.T for v in V]
        sig = self._stress([e @ self.BE.T for e in E])
        h, u = Q[0], Q[1:]
        rows = []
        for i in range(d):
            f = [-h * u[i]] + [-h * u[i] * u[j] + h / c["rho"] * sig[j][i] for j in range(d)]
            f[1 + i] = f[1 + i] - 0.5 * self.gc * h * h
            rows.append(torch.stack(f))
        flux = torch.einsum("kri,ivkq->rvkq", self.G, torch.stack(rows))
        r = torch.einsum("rvkq,rqa,q->vka", flux, self.D, self.w)
        src = [torch.zeros_like(h)]
        for j in range(d):
            s = torch.zeros_like(h) if self.dH is None else -self.gc * h * self.dH[..., j]
            src.append(s - (self.gs * h if j == 0 else 0.0))
        r = (r - torch.einsum("vkq,qa,q->vka", torch.stack(src), self.B, self.w)) * self.J[None, :, None]
        # faces
        n = [self.n[:, :, None, i] for i in range(d)]
        tr = [torch.einsum("fma,ka->kfm", self.Bf, v) for v in V]
        hm, um = tr[0], tr[1:]
        hp, up = self._sides(hm, 0), self._vel_sides(um)
        em = [torch.einsum("fmc,kc->kfm", self.BEf, e) for e in E]
        ep = [self._sides(e, 1 + d + k) for k, e in enumerate(em)]
        unm, unp = sum(a * b for a, b in zip(um, n)), sum(a * b for a, b in zip(up, n))
        cm, cp = (torch.sqrt(self.gc * torch.clamp(x, min=c["h_floor"])) for x in (hm, hp))
        SL, SR = torch.minimum(unm - cm, unp - cp), torch.maximum(unm + cm, unp + cp)

        def side(hh, uu, un):
            p = 0.5 * self.gc * hh * hh
            return [hh * un] + [hh * uu[j] * un + p * n[j] for j in range(d)], [hh] + [hh * uu[j] for j in range(d)]

        (Fm, Um), (Fp, Up) = side(hm, um, unm), side(hp, up, unp)
        sm, sp = self._stress(em), self._stress(ep)
        tot = []
        for v in range(d + 1):
            f = (SR * Fm[v] - SL * Fp[v] + SL * SR * (Up[v] - Um[v])) / (SR - SL)
            f = torch.where(SL >= 0, Fm[v], torch.where(SR <= 0, Fp[v], f))
            if v:
                f = f - 0.5 / c["rho"] * sum((hm * sm[v - 1][i] + hp * sp[v - 1][i]) * n[i] for i in range(d))
            tot.append(f * self.sJ[:, :, None] * self.wf)
        return r + torch.einsum("vkfm,fma->vka", torch.stack(tot), self.Bf)

    def mass_solve(self, V, r):
        """x of M(V) x = r, M(V) the primitive-variable mass matrix dU/dV."""
        r = r / self.J[None, :, None]
        dh = r[0] @ self.Minv.T
        hq, dq = V[0] @ self.B.T, dh @ self.B.T
        Mh = self._mass_h(hq)
        rhs = [r[1 + j] - torch.einsum("kq,qa,q->ka", dq * (V[1 + j] @ self.B.T), self.B, self.w) for j in range(self.dim)]
        du = torch.linalg.solve(Mh, torch.stack(rhs, 2))
        return torch.cat([dh[None], du.permute(2, 0, 1)])

    def _mass_h(self, hq):
        """<psi, max(h, h_floor) psi> per element, reference scaling."""
        outer = torch.einsum("qa,qb,q->qab", self.B, self.B, self.w)
        return torch.einsum("kq,qab->kab", torch.clamp(hq, min=self.i.prm["h_floor"]), outer)

    def moments(self, V):
        """<psi, U(V)> in reference scaling."""
        Q = [v @ self.B.T for v in V]
        U = torch.stack([Q[0]] + [Q[0] * x for x in Q[1:]])
        return torch.einsum("vkq,qa,q->vka", U, self.B, self.w)

    def rate(self, V):
        E = self.gradient(V)
        return -self.mass_solve(V, self.residual(V, E)), E

    def step_bound(self, V):
        c, q = self.i.prm, 2 * self.p + 1
        speed = V[1:].square().sum(0).sqrt() + torch.sqrt(self.gc * torch.clamp(V[0], min=c["h_floor"]))
        slope = 0.0
        if c["sigma0"] > 0:
            slope = {0: 0.0, 1: 2 * c["gamma"], 2: 2 * c["gamma"], 3: 2 * c["sigma0"] * c["gamma"],
                     4: 2 * c["sigma0"] * c["pap_m"], 5: 2 * c["gamma"]}[c["reg"]]
        nu = (4 * c["eta"] + slope) / c["rho"]
        return (c["cfl"] * self.dx / (q * speed.amax(1) + q * q * 2 * nu / self.dx)).min()

    # ---- integrators
    def _wet_stage(self, V0, Vs, c0, c1, dt):
        r = self.residual(Vs, self.gradient(Vs)) / self.J[None, :, None]
        m = c0 * self.moments(V0) + c1 * (self.moments(Vs) - dt * r)
        h = c0 * V0[0] + c1 * (Vs[0] - dt * r[0] @ self.Minv.T)
        mean = (h @ self.avg)[:, None]
        low = torch.cat([h, h @ self.B.T, torch.einsum("fma,ka->kfm", self.Bf, h).flatten(1)], 1).amin(1, keepdim=True)
        squeezed = mean + mean / torch.where(mean > low, mean - low, torch.ones_like(low)) * (h - mean)
        h = torch.where(mean <= 0, torch.zeros_like(h), torch.where(low < 0, squeezed, h))
        u = torch.linalg.solve(self._mass_h(h @ self.B.T), m[1:].permute(1, 2, 0)).permute(2, 0, 1)
        return torch.cat([h[None], torch.where(mean < self.i.prm["h_floor"], torch.zeros_like(u), u)])

    def explicit(self, V, steps):
        for _ in range(steps):
            dt, V0, y = self.step_bound(V), V, V
            for c0, c1 in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
                y = self._wet_stage(V0, y, c0, c1, dt) if self.i.prm["positivity"] else c0 * V0 + c1 * (y + dt * self.rate(y)[0])
            V = y
        return V

    def backward_euler(self, V, dt, steps, dense):
        for _ in range(steps):
            old = self.moments(V)

            def R(x):
                return (self.moments(x) - old) * self.J[None, :, None] / dt + self.residual(x, self.gradient(x))

            r = R(V)
            first = last = r.norm()
            for _ in range(20):
                if dense:
                    n = V.numel()
                    eye = torch.eye(n, dtype=V.dtype, device=V.device).reshape(n, *V.shape)
                    jac = torch.func.vmap(lambda z: torch.func.jvp(R, (V,), (z,))[1])(eye).reshape(n, n).T
                    d = torch.linalg.solve(jac, -r.reshape(-1)).reshape(V.shape)
                else:
                    d = self._gmres(R, V, r, dt)
                V = V + d
                r = R(V)
                # to the rounding floor: the residual no longer falls
                if r.norm() <= 1e-13 * first or (r.norm() <= 1e-9 * first and r.norm() > 0.1 * last):
                    break
                last = r.norm()
        return V

    def _gmres(self, R, V, r, dt, m=60, tol=1e-7):
        """Step d of J d = -r, right preconditioned by dt M(V)^-1."""
        beta = r.norm()
        basis, H = [-r / beta], np.zeros((m + 1, m))
        for j in range(m):
            w = torch.func.jvp(R, (V,), (dt * self.mass_solve(V, basis[j]),))[1]
            for _ in range(2):
                for i, b in enumerate(basis):
                    dot = (w * b).sum()
                    H[i, j] += float(dot)
                    w = w - dot * b
            H[j + 1, j] = float(w.norm())
            basis.append(w / H[j + 1, j])
            e = np.zeros(j + 2)
            e[0] = float(beta)
            y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= tol * float(beta):
                break
        return dt * self.mass_solve(V, sum(float(c) * b for c, b in zip(y, basis)))


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "implicit":
            i = _instances(case)[0]
            x = _Exact(i, "cpu")
            V = x.backward_euler(i.state(seed, "cpu"), 1e-6, case["steps"], dense=True)
            return V.numpy(), x.gradient(V)[0].numpy()
        out = []
        for k, i in enumerate(_instances(case)):
            x, V = _Exact(i, "cuda"), i.state(seed + 7919 * k, "cuda")
            if case["kind"] == "residual":
                return x.rate(V)
            if case["kind"] == "newton":
                dt = case["dt_factor"] * float(x.step_bound(V))
                out.append(x.backward_euler(V, dt, case["steps"], dense=False))
            else:
                out.append(x.explicit(V, case["steps"]))
        return out
