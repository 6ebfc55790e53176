"""The work users have this framework do, as cases that can be timed and whose results can be compared.

A case is a relaxation that goes on (`kind` "relax": a handle advanced by some
steps, its positions read back in the precision it runs in), a sensitivity run (`kind`
"adjoint": forward and backward of `relax_fn`) or a batch of independent
instances (`kind` "batch"). Geometries, sizes, colour counts and step counts
are those of the repository's workloads (the 4,096-particle square, the circle
of Sec. 4.1, the graded hole, the graded inclusion, the polynomial field, the
batch of uneven instances) or lie between them.

`exact` runs the same steps in plain torch in 64 bits: pairs by direct search,
sums by index, gradients by torch's own differentiation.
"""
import math
from types import SimpleNamespace

import torch

from paper_1906_07925_gb300 import Batch, Relaxation, relax_fn

SPHERE, BOX = 0, 1
UNIFORM, LINEAR, TANH = 0, 1, 2


def listed():
    return [
        # the smallest use: a 4,096-particle square in FP64 (2D, four colours), a hundred short steps in one call
        dict(name="square_2d_4k_fp64", kind="relax", geometry="square", n=4096, colors=4, precision="fp64", gamma=2.0, steps=100),
        # the circle case of the paper at its smaller size, advanced a few steps at a time (a viewer, a convergence check)
        dict(name="circle_2d_4k_fp32", kind="relax", geometry="circle", n=4289, colors=6, precision="fp32", gamma=2.0, steps=10),
        # an odd middle size in 2D with an equation of state of its own (the density pass runs too)
        dict(name="hole_2d_100k_gamma_fp32", kind="relax", geometry="hole", n=99991, colors=16, precision="fp32", gamma=1.4, steps=10),
        # the square benchmark: a million particles in 2D
        dict(name="hole_2d_1m_fp32", kind="relax", geometry="hole", n=1 << 20, colors=64, precision="fp32", gamma=2.0, steps=10),
        # a body in 3D of the size of the paper's smaller volume meshes
        dict(name="ball_3d_240k_fp32", kind="relax", geometry="ball", n=240370, colors=20, precision="fp32", gamma=2.0, steps=10),
        # the throughput headline: eight million particles in 3D
        dict(name="inclusion_3d_8m_fp32", kind="relax", geometry="inclusion", n=1 << 23, colors=256, precision="fp32", gamma=2.0, steps=5),
        # double precision where a user wants it throughout, 3D and 2D
        dict(name="inclusion_3d_300k_fp64", kind="relax", geometry="inclusion", n=300007, colors=64, precision="fp64", gamma=2.0, steps=4),
        dict(name="hole_2d_200k_fp64", kind="relax", geometry="hole", n=200003, colors=32, precision="fp64", gamma=2.0, steps=4),
        # sensitivities of twenty steps with respect to positions, parameters and the target field, from an FP32 program
        dict(name="adjoint_2d_262k_fp32", kind="adjoint", geometry="poly", n=1 << 18, colors=32, precision="fp32", gamma=2.0, steps=20),
        # the same in 3D at a small odd size, FP64, with an equation of state of its own (density adjoints)
        dict(name="adjoint_3d_20k_gamma_fp64", kind="adjoint", geometry="ball", n=20011, colors=8, precision="fp64", gamma=1.4, steps=6),
        # many uneven instances at once, half 2D and half 3D
        dict(name="batch_48_fp32", kind="batch", instances=48, n_lo=2000, n_hi=100000, precision="fp32", steps=10),
    ]


def draw(rng):
    """A case of the same ranges: more adjoint and batch runs than chance among the sizes alone would give."""
    kind = rng.choice(["relax"] * 6 + ["adjoint"] * 2 + ["batch"])
    odd = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1  # noqa: E731
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "batch":
        n_lo = odd(2000, 8000)
        return dict(kind=kind, instances=rng.randrange(8, 49), n_lo=n_lo, n_hi=odd(2 * n_lo, 100000), precision="fp32", steps=rng.randrange(4, 11))
    geometry = rng.choice(["square", "circle", "hole", "poly", "ball", "inclusion"])
    gamma = rng.choice([2.0, 2.0, round(rng.uniform(1.2, 3.0), 2)])
    if kind == "adjoint":
        return dict(kind=kind, geometry=geometry, n=odd(4000, 12000 if precision == "fp64" else 100000), colors=rng.randrange(2, 33), precision=precision, gamma=gamma, steps=rng.randrange(4, 11))
    n = odd(4000, 200000 if precision == "fp64" else 4000000)
    return dict(kind=kind, geometry=geometry, n=n, colors=rng.randrange(2, 257), precision=precision, gamma=gamma, steps=rng.randrange(2, 11))


# ------------------------------------------------------------------ inputs

def _problem(geometry, colors, gamma, poly=()):
    """Geometry, target spacing and parameters as Relaxation takes them (rho_scale is set from the particle count below)."""
    p = SimpleNamespace(dim=2, lo=[0.0, 0.0, 0.0], hi=[1.0, 1.0, 0.0], shapes=[], field_kind=UNIFORM, s0=1.0, a=0.0, b=0.0, dist_shape=0, poly=list(poly),
                        rho_scale=1.0, P0=1.0, gamma=gamma, sigma0=3.0, tau=2.0, kappa=1.0, n_colors=colors)
    shape = lambda kind, inside, c, s: SimpleNamespace(kind=kind, keep_inside=inside, center=list(c), size=list(s))  # noqa: E731
    if geometry == "circle":  # a disk of radius 43 in [0, 100]^2 with a tanh-graded target size (Sec. 4.1)
        p.hi = [100.0, 100.0, 0.0]
        p.shapes = [shape(SPHERE, True, (50.0, 50.0, 0.0), (43.0, 0, 0))]
        p.field_kind, p.a, p.b, p.s0 = TANH, 0.391, (3.125 - 0.391) / math.tanh(2.5), 2.5 / 43.0
    elif geometry in ("hole", "poly"):  # the unit square less a disk, finer at the disk
        p.shapes = [shape(SPHERE, False, (0.5, 0.5, 0.0), (0.2, 0, 0))]
        p.field_kind, p.a, p.b = LINEAR, 0.002, 0.02
    elif geometry == "inclusion":  # the unit cube less a ball, finer at the ball
        p.dim, p.hi = 3, [1.0, 1.0, 1.0]
        p.shapes = [shape(SPHERE, False, (0.5, 0.5, 0.5), (0.25, 0, 0))]
        p.field_kind, p.a, p.b = LINEAR, 0.004, 0.03
    elif geometry == "ball":  # a ball, finer at its surface
        p.dim, p.hi = 3, [1.0, 1.0, 1.0]
        p.shapes = [shape(SPHERE, True, (0.5, 0.5, 0.5), (0.35, 0, 0))]
        p.field_kind, p.a, p.b = LINEAR, 0.01, 0.02
    p.copy = lambda **kw: SimpleNamespace(**{**vars(p), **kw})
    return p


def _inside_distance(s, x):
    d = x.shape[1]
    c = torch.tensor(s.center[:d], dtype=x.dtype, device=x.device)
    if s.kind == SPHERE:
        return s.size[0] - (x - c).norm(dim=1)
    q = (x - c).abs() - torch.tensor(s.size[:d], dtype=x.dtype, device=x.device)
    return -(q.clamp(min=0).norm(dim=1) + q.amax(dim=1).clamp(max=0))


def _spacing(p, x):
    if p.field_kind == UNIFORM:
        return torch.full_like(x[:, 0], p.s0)
    dist = _inside_distance(p.shapes[p.dist_shape], x).abs()
    return p.a + p.b * (torch.tanh(p.s0 * dist) if p.field_kind == TANH else dist)


def _poly_factor(p, x, coef):
    if coef is None or len(coef) == 0:
        return torch.ones_like(x[:, 0])
    lo, hi = (torch.tensor(v[:p.dim], dtype=x.dtype, device=x.device) for v in (p.lo, p.hi))
    t = 2 * (x - lo) / (hi - lo) - 1
    X, Y = t[:, 0], t[:, 1]
    if p.dim == 2:
        b = [X, Y, X * X, X * Y, Y * Y, X ** 3, X * X * Y, X * Y * Y]
    else:
        Z = t[:, 2]
        b = [X, Y, Z, X * X, Y * Y, Z * Z, X * Y, Y * Z]
    return 1 + sum(coef[k] * b[k] for k in range(len(coef)))


def _inside(p, x):
    m = torch.ones(len(x), dtype=torch.bool, device=x.device)
    for s in p.shapes:
        m &= (_inside_distance(s, x) > 0) == s.keep_inside
    return m


def _state(p, n, g):
    """n particles drawn in proportion to the target density (rejection), coloured by the nearest of n_colors
    generators in the region (the start of Sec. 4.2); sets p.rho_scale so that the region holds n unit masses."""
    d, dev = p.dim, torch.device("cuda")
    lo, hi = (torch.tensor(v[:d], dtype=torch.float64, device=dev) for v in (p.lo, p.hi))
    coef = torch.tensor(p.poly, dtype=torch.float64, device=dev) if p.poly else None

    def points(m):
        x = lo + (hi - lo) * torch.rand((m, d), dtype=torch.float64, device=dev, generator=g)
        return x[_inside(p, x)]

    weight = lambda x: _spacing(p, x) ** -d * _poly_factor(p, x, coef)  # noqa: E731
    res = 1024 if d == 2 else 128
    axes = [lo[k] + (hi[k] - lo[k]) * (torch.arange(res, dtype=torch.float64, device=dev) + 0.5) / res for k in range(d)]
    grid = torch.stack(torch.meshgrid(*axes, indexing="ij"), -1).reshape(-1, d)
    grid = grid[_inside(p, grid)]
    p.rho_scale = float(n / (weight(grid).sum() * (hi - lo).prod() / res ** d))
    wmax = float((p.s0 if p.field_kind == UNIFORM else p.a) ** -d * (1 + sum(abs(c) for c in p.poly)))
    gens = torch.empty((0, d), dtype=torch.float64, device=dev)
    while len(gens) < p.n_colors:
        gens = torch.cat([gens, points(4 * p.n_colors)])
    gens = gens[:p.n_colors]
    got, have = [], 0
    while have < n:
        x = points(4 * n if n < 1 << 20 else 2 * n)
        x = x[torch.rand(len(x), dtype=torch.float64, device=dev, generator=g) * wmax < weight(x)]
        got.append(x)
        have += len(x)
    x = torch.cat(got)[:n].contiguous()
    col = torch.cat([((c[:, None, :] - gens) ** 2).sum(-1).argmin(1) for c in x.split(1 << 18)]).to(torch.uint8)
    return x, col


def _inputs(case, seed):
    """One instance's problem, positions and colours, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    poly = ()
    if case["geometry"] == "poly":
        poly = [float(v) for v in (torch.rand(8, dtype=torch.float64, device="cuda", generator=g) * 0.1 - 0.05).cpu()]
    p = _problem(case["geometry"], case["colors"], case["gamma"], poly)
    if case["geometry"] == "square":  # a lattice with a jitter of 0.3 of its spacing, as far as it goes, for a uniform target
        p.s0 = 1.0 / math.isqrt(case["n"])
        side = math.isqrt(case["n"] - 1) + 1
        ij = torch.arange(side * side, device="cuda")[:case["n"]]
        x = (torch.stack([ij // side, ij % side], 1).double() + 0.5) / side
        x = x + (torch.rand(x.shape, dtype=torch.float64, device="cuda", generator=g) * 0.6 - 0.3) / side
        gens = torch.rand((case["colors"], 2), dtype=torch.float64, device="cuda", generator=g)
        return p, x.contiguous(), torch.cat([((c[:, None, :] - gens) ** 2).sum(-1).argmin(1) for c in x.split(1 << 18)]).to(torch.uint8)
    x, col = _state(p, case["n"], g)
    return p, x, col


def _instances(case, seed):
    """The batch's problems, positions and colours: half 2D and half 3D, sizes log-uniform, a sphere or a box, spacing graded from its surface."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    u = torch.rand((case["instances"], 12), dtype=torch.float64, device="cuda", generator=g).cpu()
    out = []
    for k in range(case["instances"]):
        v = [float(t) for t in u[k]]
        dim = 2 if k < case["instances"] // 2 else 3
        n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((k + 1) * 0.6180339887 % 1.0)))  # sizes are the case's, not the seed's
        p = _problem("square", 2 + int(63 * v[1]), 2.0)
        p.dim, p.hi = dim, [1.0, 1.0, 1.0 if dim == 3 else 0.0]
        c = [0.4 + 0.2 * v[2], 0.4 + 0.2 * v[3], 0.4 + 0.2 * v[4] if dim == 3 else 0.0]
        if v[5] < 0.5:
            p.shapes = [SimpleNamespace(kind=SPHERE, keep_inside=True, center=c, size=[0.3 + 0.1 * v[6], 0.0, 0.0])]
        else:
            p.shapes = [SimpleNamespace(kind=BOX, keep_inside=True, center=c, size=[0.25 + 0.1 * t for t in v[6:9]])]
        p.field_kind, p.a, p.b = LINEAR, 0.01, 0.005 + 0.025 * v[9]
        x, col = _state(p, n, g)
        out.append((p, x, col))
    return out


# --------------------------------------------------------------- the cases

def prepare(case, seed):
    if case["kind"] == "batch":
        inst = _instances(case, seed)
        b = Batch([p for p, _, _ in inst], [len(x) for _, x, _ in inst], [p.n_colors for p, _, _ in inst], precision=case["precision"], n_branches=32)
        for k, (_, x, col) in enumerate(inst):
            b.set_state(k, x.cpu().numpy(), col.cpu().numpy())
        return SimpleNamespace(case=case, batch=b)
    p, x, col = _inputs(case, seed)
    if case["kind"] == "adjoint":
        t = torch.float64 if case["precision"] == "fp64" else torch.float32
        leaf = lambda v: torch.tensor(v, dtype=t, device="cuda")  # noqa: E731
        f = relax_fn(p, col.cpu().numpy(), case["steps"], precision=case["precision"])
        args = [x.to(t), leaf(p.sigma0), leaf(p.gamma), leaf(p.P0), leaf(p.poly or [0.0] * 8)]
        # P0 stays a constant: with step sizes taken from the accelerations the run does not depend on it
        leaves = [a.requires_grad_() for k, a in enumerate(args) if k != 3]
        torch.cuda.synchronize()
        return SimpleNamespace(case=case, f=f, args=args, leaves=leaves)
    r = Relaxation(p, case["n"], case["colors"], precision=case["precision"])
    torch.cuda.synchronize()  # the handle has a stream of its own
    r.set_state(x, col)
    return SimpleNamespace(case=case, r=r, out=torch.empty_like(x))


def run(state):
    case = state.case
    if case["kind"] == "batch":
        state.batch.step(case["steps"])
        x = [state.batch.positions(k) for k in range(case["instances"])]
        return x if case["precision"] == "fp64" else [v.astype("float32") for v in x]
    if case["kind"] == "adjoint":
        # a training step's forward and backward: the loss in the program's type, a gradient for every input
        for a in state.leaves:
            a.grad = None
        x, loss = state.f(*state.args)
        loss = loss.to(state.args[0].dtype)
        loss.backward()
        return [x.detach().to(state.args[0].dtype), loss.detach()] + [a.grad for a in state.leaves]
    state.r.step(case["steps"])
    x = state.r.positions(out=state.out)
    return x if case["precision"] == "fp64" else x.float()


def work(case):
    """Positions and colours in, positions out; pair arithmetic of the two force sums (and the reverse pass's) per step."""
    if case["kind"] == "batch":
        n, d = case["instances"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"]), 2.5
    else:
        n, d = case["n"], 3 if case["geometry"] in ("ball", "inclusion") else 2
    pairs = 33.5 if d == 3 else 12.6 if d == 2 else 23.0
    flops = n * pairs * 90.0 * case["steps"]  # distance, kernel and force terms of both sums
    size = n * (16.0 * d + 1)
    if case["kind"] == "adjoint":
        return {"bytes": 2 * size, "flops": 3 * flops}
    return {"bytes": size, "flops": flops}


# ------------------------------------------------------------ 64-bit values

def _pairs(x, H, margin):
    """All ordered pairs i != j with r < (1 + margin) max(H_i, H_j): strips of the particles sorted along x."""
    order = x[:, 0].argsort()
    xs, Hs = x[order], H[order] * (1 + margin)
    reach = float(Hs.max())
    left = xs[:, 0].contiguous()
    out_i, out_j = [], []
    n, b = len(xs), 0
    while b < n:
        e = min(n, b + 1024)
        c0 = int(torch.searchsorted(left, left[b] - reach))
        c1 = int(torch.searchsorted(left, left[e - 1] + reach, right=True))
        r2 = 0
        for k in range(x.shape[1]):
            r2 = r2 + (xs[b:e, k, None] - xs[None, c0:c1, k]) ** 2
        i, j = torch.nonzero(r2 < torch.maximum(Hs[b:e, None], Hs[None, c0:c1]) ** 2, as_tuple=True)
        keep = i + b != j + c0
        out_i.append(order[i[keep] + b])
        out_j.append(order[j[keep] + c0])
        b = e
    return torch.cat(out_i), torch.cat(out_j)


class _Exact:
    """The relaxation step in torch, 64 bits, differentiable in everything."""

    def __init__(self, p, col, sigma0, gamma, P0, coef):
        self.p, self.col, self.sigma0, self.gamma, self.P0, self.coef = p, col.long(), sigma0, gamma, P0, coef
        self.alpha = 7 / math.pi if p.dim == 2 else 21 / (2 * math.pi)

    def h(self, x):
        p = self.p
        return p.tau * p.rho_scale ** (-1 / p.dim) * _spacing(p, x) * _poly_factor(p, x, self.coef) ** (-1 / p.dim)

    def add(self, n, i, v):
        return torch.zeros((n,) + tuple(v.shape[1:]), dtype=v.dtype, device=v.device).index_add(0, i, v)

    def density(self, h, i, r):
        H = self.p.kappa * h
        q = r / H[i]
        u = (1 - q).clamp(min=0)
        w = self.alpha * u ** 4 * (1 + 4 * q) / H[i] ** self.p.dim
        return self.add(len(h), i, w) + self.alpha / H ** self.p.dim

    def step(self, x, i, j):
        p, n, d = self.p, len(x), self.p.dim
        h = self.h(x)
        T = (h / p.tau) ** (2 * d)  # 1 / rho_t^2
        e = x[i] - x[j]
        r = e.norm(dim=1)
        Hij = p.kappa * (h[i] + h[j]) / 2
        F = -20 * self.alpha * (1 - r / Hij).clamp(min=0) ** 3 / Hij ** (d + 2)
        if float(self.gamma) == 2.0:  # P0 / rho_t^2 whatever the density: ln(rho / rho_t) only where gamma asks for it
            Q = self.P0 * T
            if torch.is_tensor(self.gamma):
                Q = Q * torch.exp((self.gamma - 2) * torch.log(self.density(h, i, r) * T.sqrt()).detach())
        else:
            rho = self.density(h, i, r)
            Q = self.P0 * (rho * T.sqrt()) ** self.gamma / rho ** 2
        beta = self.sigma0 * (self.col[i] != self.col[j])
        a = self.add(n, i, (-(Q[i] + Q[j] + beta * self.P0 * (T[i] + T[j])) * F)[:, None] * e)
        an = a.norm(dim=1)
        rc = p.kappa * h
        m = (rc / torch.where(an > 0, an, torch.full_like(an, 1e-300))).amin()
        dt1 = 0.25 * m.sqrt()
        dt2 = torch.minimum(dt1, torch.minimum(m / (20 * dt1), 2.5 * m / dt1))
        vt = 0.5 * dt1 * a
        eta = 0.1 * rc * vt.norm(dim=1) / T.sqrt()
        s = eta[i] + eta[j]
        hm = torch.where(s > 0, 2 * eta[i] * eta[j] / torch.where(s > 0, s, torch.ones_like(s)), torch.zeros_like(s))
        visc = self.add(n, i, (hm * (T[i] + T[j]) * F)[:, None] * (vt[i] - vt[j]))
        y = x + dt2 * (vt + 0.5 * dt2 * visc)
        lo, hi = (torch.tensor(v[:d], dtype=x.dtype, device=x.device) for v in (p.lo, p.hi))
        y = torch.minimum(torch.maximum(y, lo), hi)
        for sh in p.shapes:
            phi = _inside_distance(sh, y)
            out = phi < 0 if sh.keep_inside else phi > 0
            c = torch.tensor(sh.center[:d], dtype=x.dtype, device=x.device)
            if sh.kind == SPHERE:
                v = y - c
                q = c + sh.size[0] * v / v.norm(dim=1, keepdim=True)
            else:
                z = torch.tensor(sh.size[:d], dtype=x.dtype, device=x.device)
                q = torch.minimum(torch.maximum(y, c - z), c + z)
            y = torch.where(out[:, None], q, y)
        return y

    def run(self, x, steps):
        i = j = None
        for k in range(steps):
            if k % 5 == 0:  # a particle moves at most 0.025 of its support in a step
                with torch.no_grad():
                    i, j = _pairs(x.detach(), self.p.kappa * self.h(x.detach()), 0.3)
            x = self.step(x, i, j)
        return x

    def objective(self, x):
        p, d = self.p, self.p.dim
        with torch.no_grad():
            i, j = _pairs(x.detach(), p.kappa * self.h(x.detach()), 0.01)
        h = self.h(x)
        r = (x[i] - x[j]).norm(dim=1)
        T = (h / p.tau) ** (2 * d)
        H = p.kappa * (h[i] + h[j]) / 2
        q = r / H
        w = self.alpha * (1 - q).clamp(min=0) ** 4 * (1 + 4 * q) / H ** d
        return ((self.density(h, i, r) * T.sqrt() - 1) ** 2).sum() + 0.5 * (w * (self.col[i] != self.col[j])).sum()


def exact(case, seed):
    if case["kind"] == "batch":
        with torch.no_grad():
            return [_Exact(p, col, p.sigma0, p.gamma, p.P0, None).run(x, case["steps"]) for p, x, col in _instances(case, seed)]
    d = 3 if case["geometry"] in ("ball", "inclusion") else 2
    if case["n"] > (400000 if d == 3 else 2000000):
        return None  # the direct search takes too long
    p, x, col = _inputs(case, seed)
    if case["kind"] == "adjoint":
        t = torch.float64 if case["precision"] == "fp64" else torch.float32
        leaf = lambda v: torch.tensor(v, dtype=t, device="cuda").double().requires_grad_()  # noqa: E731
        x0, sigma0, gamma, coef = x.to(t).double().requires_grad_(), leaf(p.sigma0), leaf(p.gamma), leaf(p.poly or [0.0] * 8)
        p.poly = coef.tolist()
        ex = _Exact(p, col, sigma0, gamma, p.P0, coef)
        xk = ex.run(x0, case["steps"])
        loss = ex.objective(xk)
        return [xk.detach(), loss.detach()] + list(torch.autograd.grad(loss, [x0, sigma0, gamma, coef]))
    with torch.no_grad():
        return _Exact(p, col, p.sigma0, p.gamma, p.P0, torch.tensor(p.poly, dtype=torch.float64, device="cuda") if p.poly else None).run(x, case["steps"])
