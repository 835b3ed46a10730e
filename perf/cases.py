"""The work that users of the library have it do, as cases that can be timed and checked.

A case is a dict of plain values.  "kind" says which calls it makes:
  cycles    Forest.vcycle: a fixed number of V-cycles from u = 0
  solve     Forest.solve: cycles from u = 0 to a relative residual
  step      Forest.set_rhs with a new f and k, then Forest.solve
  gradient  MGSolveFn forward and backward: u, dL/df and dL/dk of L = 1/2 sum (u - target)^2
  operator  Forest.apply and Forest.apply_transpose
  batch     Batch.solve: many independent problems of different block sizes
and the other entries describe the forest (R roots per axis, n cells per block edge, how it is refined) and the
options it is built with.
"""
import itertools
import math

import numpy as np
import torch

from paper_2403_08063_gb300 import Batch, Forest, MGSolveFn

F64 = torch.float64
BASE = {"R": 2, "n": 16, "refine": "none", "depth": 0, "radius": 0.25, "box": 0, "k": False, "precision": 0, "inner": 1,
        "coarse": "k", "flux": True, "smoother": "rbgs", "boundary": False, "rtol": 1e-10, "cycles": 0, "problems": 0}


def _case(name=None, **kw):
    return {**({"name": name} if name else {}), **BASE, **kw}


def listed():
    return [
        # the smallest call: a 32^3 grid, exactly ten FP64 cycles (an inner solver of a larger program); latency-bound
        _case("small_cycles_f64", kind="cycles", R=2, n=16, cycles=10),
        # a small variable-coefficient solve with FP32 cycles, as one of many in a sweep over parameters
        _case("small_solve_mixed", kind="solve", R=2, n=16, k=True, precision=1, inner=5, coarse="faces"),
        # the plain method on an octree refined around a sphere (120 blocks of 32^3): interfaces on every level
        _case("sphere_solve_f64", kind="solve", R=2, n=32, refine="ball", depth=2),
        # the same forest with FP32 cycles inside FP64 defect correction
        _case("sphere_solve_mixed", kind="solve", R=2, n=32, refine="ball", depth=2, precision=1, inner=4),
        # a time or Newton step: the coefficient changes, so set-up and solve are both paid for
        _case("new_k_step_mixed", kind="step", R=4, n=32, k=True, precision=1, inner=5, coarse="faces"),
        # plain FP64 cycles with a variable coefficient and the library's default coarse operator, 256^3 cells
        _case("k_cycles_f64", kind="cycles", R=4, n=64, k=True, cycles=4),
        # the largest solve: 512^3 cells, rough coefficient, FP32 cycles inside FP64 defect correction
        _case("large_solve_mixed", kind="solve", R=8, n=64, k=True, precision=1, inner=5, coarse="faces"),
        # the paper's own cycle: damped Jacobi V(3,3), ghost-only interfaces, Jacobi coarsest sweeps, Dirichlet data
        _case("paper_cycles_f64", kind="cycles", R=1, n=64, refine="paper", depth=2, flux=False, smoother="jacobi",
              boundary=True, cycles=5),
        # matrix-free operator and its transpose, as an outer Krylov method calls them; odd root count
        _case("sphere_operator_f64", kind="operator", R=3, n=32, refine="ball", depth=1, k=True),
        # gradients on a small grid with an odd root count, FP64 cycles in both directions
        _case("odd_gradient_f64", kind="gradient", R=3, n=16, k=True, coarse="faces"),
        # one step of coefficient identification on a sphere-refined octree (31M cells), FP32 cycles both ways
        _case("sphere_gradient_mixed", kind="gradient", R=4, n=32, refine="ball", depth=2, k=True, precision=1, inner=4,
              coarse="faces"),
        # independent problems with mixed block sizes and refinement, solved together
        _case("batch_mixed", kind="batch", R=1, n=0, problems=24, box=1, k=True, precision=1, inner=5, coarse="faces",
              rtol=1e-8),
    ]


# Largest number of cells drawn per kind: below the cost of the largest listed cases.
MOST_CELLS = {"cycles": 3e7, "solve": 1.4e8, "step": 4e7, "gradient": 2e7, "operator": 3e7}


def draw(rng):
    kind = rng.choice(["cycles", "cycles", "solve", "solve", "step", "gradient", "gradient", "operator", "batch"])
    if kind == "batch":
        return _case(kind=kind, R=1, n=0, problems=int(round(4 * 8 ** rng.random())), box=rng.randrange(1, 10 ** 6), k=True,
                     precision=1, inner=rng.choice([3, 5]), coarse=rng.choice(["k", "faces"]), rtol=1e-8)
    k = kind in ("step", "gradient") or rng.random() < 0.6
    precision = 0 if kind == "cycles" else rng.choice([0, 1])
    most = MOST_CELLS[kind] if precision or kind == "operator" else min(MOST_CELLS[kind], 1e7 if kind == "gradient" else 2e7)
    want = math.exp(rng.uniform(math.log(3e4), math.log(most)))
    refine = rng.choice(["none", "ball", "box"])
    forests = []
    for R, n in itertools.product((1, 2, 3, 4, 6, 8), (8, 16, 32, 64)):
        c = _case(kind=kind, R=R, n=n, refine=refine, depth=0 if refine == "none" else rng.choice([1, 2]),
                  radius=round(rng.uniform(0.15, 0.35), 3), box=rng.randrange(1, 10 ** 6))
        if refine == "none" or R <= 4:
            cells = len(_leaves(c)) * n ** 3
            if cells <= most and R * n >= 16:
                forests.append((abs(math.log(cells / want)), len(forests), c))
    c = min(forests)[2]
    c.update(k=k, precision=precision, inner=rng.choice([4, 5]) if precision else 1,
             coarse="faces" if precision and k else rng.choice(["k", "faces"]) if k else "k",
             flux=rng.random() < 0.75, cycles=rng.randrange(2, 9) if kind == "cycles" else 0)
    return c


# ---------------------------------------------------------------------------------------------------------------------
# Forests: leaves (level, i, j, k) over the unit cube, 2:1 balanced across faces, edges and corners
# ---------------------------------------------------------------------------------------------------------------------
def _children(key):
    l, i, j, k = key
    return [(l + 1, 2 * i + a, 2 * j + b, 2 * k + c) for c in (0, 1) for b in (0, 1) for a in (0, 1)]


def _refined(R, depth, hit):
    done, todo = [], [(0, i, j, k) for k in range(R) for j in range(R) for i in range(R)]
    while todo:
        key = todo.pop(0)
        l, ijk = key[0], np.array(key[1:], float)
        e = 1.0 / (R * 2 ** l)
        if l < depth and hit(l, ijk * e, (ijk + 1) * e):
            todo.extend(_children(key))
        else:
            done.append(key)
    leaves = set(done)
    changed = depth > 1
    while changed:
        changed = False
        for l, i, j, k in sorted(leaves, reverse=True):
            if l < 2:
                break
            for a, b, c in itertools.product((-1, 0, 1), repeat=3):
                p = ((i + a) >> 2, (j + b) >> 2, (k + c) >> 2)  # the block two levels up next to this one
                if (l - 2, *p) in leaves:
                    leaves.remove((l - 2, *p))
                    leaves.update(_children((l - 2, *p)))
                    changed = True
    return sorted(leaves, key=lambda t: (t[0], t[3], t[2], t[1]))


def _box_hit(seed, index=0):
    r = np.random.RandomState((seed * 1009 + index) % (2 ** 31))
    side = r.uniform(0.1, 0.4, 3)
    lo = r.uniform(0, 1, 3) * (1 - side)
    return lambda l, a, b: bool(np.all(a < lo + side) and np.all(b > lo))


def _leaves(case):
    R, depth = case["R"], case["depth"]
    if case["refine"] == "none":
        return [(0, i, j, k) for k in range(R) for j in range(R) for i in range(R)]
    if case["refine"] == "ball":
        def hit(l, a, b):
            d = np.maximum(0, np.maximum(a - 0.5, 0.5 - b))
            return float(d @ d) < case["radius"] ** 2
    elif case["refine"] == "paper":  # every root once, a quarter of the domain (x and y below one half) once more
        def hit(l, a, b):
            return l == 0 or bool(a[0] < 0.5 and a[1] < 0.5)
    else:
        hit = _box_hit(case["box"])
    return _refined(R, depth, hit)


def _batch_problems(case):
    """Leaf rows (problem, level, i, j, k) and the block edge of every problem."""
    r = np.random.RandomState(case["box"])
    rows, edges = [], []
    for p in range(case["problems"]):
        edges.append(int(r.choice([16, 32, 64, 128])))
        depth = int(r.choice([0, 1, 2])) if edges[-1] < 128 else 0
        keys = _refined(case["R"], depth, _box_hit(case["box"], p + 1))
        rows += [(p, *key) for key in keys]
    return np.array(rows, np.int32), edges


# ---------------------------------------------------------------------------------------------------------------------
# Fields: (leaves, n^3), x fastest inside a leaf
# ---------------------------------------------------------------------------------------------------------------------
def _lines(R, n, leaves):
    """Cell-centre coordinates of every leaf along x, y and z, each (leaves, n)."""
    a = torch.tensor(np.array(leaves, np.float64).reshape(-1, 4), device="cuda")
    h = 1.0 / (R * n * 2.0 ** a[:, :1])
    t = torch.arange(n, dtype=F64, device="cuda") + 0.5
    return [(a[:, d + 1, None] * n + t) * h for d in range(3)]


def _rough_k(R, n, leaves, seed, waves=32):
    """exp of a Gaussian random field (unit variance, correlation length 0.1, never below two cells of a root block)."""
    g = torch.Generator().manual_seed(seed)
    length = max(0.1, 2.0 / (R * n))
    w = (torch.randn(3, waves, generator=g, dtype=F64) / length).cuda()
    phase = (2 * math.pi * torch.rand(waves, generator=g, dtype=F64)).cuda()
    x, y, z = _lines(R, n, leaves)
    a = x[:, :, None] * w[0] + phase
    b = (z[:, :, None, None] * w[2] + y[:, None, :, None] * w[1]).reshape(len(leaves), n * n, waves)
    field = torch.baddbmm(torch.bmm(b.cos(), a.cos().transpose(1, 2)), b.sin(), a.sin().transpose(1, 2), alpha=-1.0)
    return (math.sqrt(2.0 / waves) * field).exp_().reshape(len(leaves), n ** 3)


def _source(R, n, leaves, seed, rough):
    """Uniform noise in [-1, 1], or a Gaussian bump on a smooth background with noise of amplitude 1e-3."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.rand(len(leaves), n ** 3, generator=g, dtype=F64, device="cuda").mul_(2).sub_(1)
    if rough:
        return noise
    x, y, z = _lines(R, n, leaves)
    at = torch.rand(3, generator=torch.Generator().manual_seed(seed)) * 0.2 + 0.4
    bump, wave = [], []
    for c, v in zip(at.tolist(), (x, y, z)):
        bump.append(torch.exp(-(v - c) ** 2 / (2 * 0.05 ** 2)))
        wave.append(torch.sin(math.pi * v))
    for f, scale in ((bump, 1.0), (wave, 0.1)):
        noise.mul_(1e-3 if f is bump else 1.0)
        noise += scale * (f[2][:, :, None, None] * f[1][:, None, :, None] * f[0][:, None, None, :]).reshape(noise.shape)
    return noise


def _target(R, n, leaves, seed):
    m = [1 + (seed // 3 ** d) % 3 for d in range(3)]
    x, y, z = [torch.sin(math.pi * m[d] * v) for d, v in enumerate(_lines(R, n, leaves))]
    return (z[:, :, None, None] * y[:, None, :, None] * x[:, None, None, :]).reshape(len(leaves), n ** 3)


def _boundary(R, n, leaves, seed):
    """Dirichlet data sin(pi x) sin(pi y) sinh(sqrt(2) pi z) at the face centres, scaled by the seed."""
    scale = 1.0 + 0.01 * (seed % 97)
    x, y, z = _lines(R, n, leaves)
    fx, fy = (lambda v: scale * torch.sin(math.pi * v)), (lambda v: torch.sin(math.pi * v))
    fz = (lambda v: torch.sinh(math.sqrt(2) * math.pi * v))
    h = (x[:, 1] - x[:, 0])[:, None]
    out = torch.zeros(len(leaves), 6, n, n, dtype=F64, device="cuda")
    for side in (0, 1):
        ends = [(v[:, -1:] + h / 2) if side else (v[:, :1] - h / 2) for v in (x, y, z)]
        out[:, side] = (fx(ends[0]) * fz(z))[:, :, None] * fy(y)[:, None, :]
        out[:, 2 + side] = (fy(ends[1]) * fz(z))[:, :, None] * fx(x)[:, None, :]
        out[:, 4 + side] = (fz(ends[2]) * fy(y))[:, :, None] * fx(x)[:, None, :]
    return out.reshape(len(leaves), 6, n * n)


# ---------------------------------------------------------------------------------------------------------------------
def _inputs(case, seed):
    R, n, leaves = case["R"], case["n"], _leaves(case)
    d = {"f": _source(R, n, leaves, seed, case["k"] or case["smoother"] == "jacobi"), "k": None}
    if case["k"]:
        d["k"] = _rough_k(R, n, leaves, seed + 1)
    if case["kind"] == "gradient":
        d["target"] = _target(R, n, leaves, seed)
        d["f"] = _source(R, n, leaves, seed, False)
    if case["boundary"]:
        d["boundary"] = _boundary(R, n, leaves, seed)
    return leaves, d


def _prepare_batch(case, seed):
    rows, edges = _batch_problems(case)
    f, k = [], []
    for p, n in enumerate(edges):
        leaves = [tuple(r[1:]) for r in rows.tolist() if r[0] == p]
        f.append(_source(1, n, leaves, seed * 1000 + p, True).reshape(-1))
        k.append(_rough_k(1, n, leaves, seed * 1000 + p).reshape(-1))
    solver = Batch(rows, edges, R=1, coeff=True, inner_cycles=case["inner"], coarse_coef=case["coarse"])
    state = {"case": case, "solver": solver, "f": torch.cat(f), "k": torch.cat(k)}
    solver.set_rhs(state["f"], state["k"])
    return state


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    leaves, state = _inputs(case, seed)
    extra = {}
    if case["smoother"] == "jacobi":
        extra = {"smoother": "jacobi", "omega": 0.8, "coarse_iters": 256, "nu1": 3, "nu2": 3}
    solver = Forest(case["R"], case["n"], leaves, coeff=case["k"], interface_flux=case["flux"],
                    precision=case["precision"], inner_cycles=case["inner"], coarse_coef=case["coarse"], **extra)
    if "boundary" in state:
        solver.set_boundary(state["boundary"])
    solver.set_rhs(state["f"], state["k"])
    if case["kind"] == "gradient":  # the leaves of the user's graph
        state["f"].requires_grad_()
        state["k"].requires_grad_()
    return {**state, "case": case, "solver": solver}


def run(state):
    case, solver, f, k = state["case"], state["solver"], state["f"], state["k"]
    kind = case["kind"]
    if kind == "cycles":
        u = torch.zeros_like(f)
        solver.vcycle(u, case["cycles"])
        return {"u": u}
    if kind in ("solve", "step", "batch"):
        if kind == "step":
            solver.set_rhs(f, k)
        u = torch.zeros_like(f)
        cycles, _ = solver.solve(u, rtol=case["rtol"], max_cycles=100)
        return {"u": u, "cycles": cycles if isinstance(cycles, int) else np.array(cycles)}
    if kind == "operator":
        return {"Au": solver.apply(f), "ATu": solver.apply_transpose(f)}
    u = MGSolveFn.apply(f, k, solver, case["rtol"], 100)
    df, dk = torch.autograd.grad(0.5 * ((u - state["target"]) ** 2).sum(), (f, k))
    return {"u": u.detach(), "df": df, "dk": dk}


def work(case):
    """Bytes: every input read once and every output written once.  Flops: a V(2,2) cycle's four sweeps, residual and
    transfers on all levels (8/7 of the finest), times the cycles that are asked for or usual (10)."""
    if case["kind"] == "batch":
        rows, edges = _batch_problems(case)
        cells = sum(edges[p] ** 3 for p in rows[:, 0].tolist())
    else:
        cells = len(_leaves(case)) * case["n"] ** 3
    k = 1 if case["k"] else 0
    if case["kind"] == "operator":
        return {"bytes": 8.0 * cells * (3 + k), "flops": cells * (2 * (8.0 + 6 * k))}
    sweeps = 6 if case["smoother"] == "jacobi" else 4
    cycle = 8 / 7 * ((sweeps + 1) * (8.0 + 6 * k) + 6)
    if case["kind"] == "gradient":
        return {"bytes": 8.0 * cells * 6, "flops": cells * 20 * cycle}
    return {"bytes": 8.0 * cells * (2 + k), "flops": cells * (case["cycles"] or 10) * cycle}


# ---------------------------------------------------------------------------------------------------------------------
# The same results in plain torch, 64 bits
# ---------------------------------------------------------------------------------------------------------------------
# A forest that is not refined is one grid of (R n)^3 cells.
def _to_grid(v, R, n):
    return v.reshape(R, R, R, n, n, n).permute(0, 3, 1, 4, 2, 5).reshape(R * n, R * n, R * n)


def _from_grid(g, R, n):
    return g.reshape(R, n, R, n, R, n).permute(0, 2, 4, 1, 3, 5).reshape(R ** 3, n ** 3)


def _faces(k, N, device="cuda"):
    """Face coefficients over h^2 below and above every cell, per axis (z, y, x): harmonic means, k_i at the boundary."""
    if k is None:
        return [(N * N, N * N)] * 3
    out = []
    for d in range(3):
        lo, hi = k.narrow(d, 0, N - 1), k.narrow(d, 1, N - 1)
        inner = 2 * lo * hi / (lo + hi)
        out.append((torch.cat([k.narrow(d, 0, 1), inner], d) * (N * N), torch.cat([inner, k.narrow(d, N - 1, 1)], d) * (N * N)))
    return out


def _neighbours(u, d):
    """Values below and above every cell along an axis, the reflection -u outside."""
    N = u.shape[d]
    return (torch.cat([-u.narrow(d, 0, 1), u.narrow(d, 0, N - 1)], d),
            torch.cat([u.narrow(d, 1, N - 1), -u.narrow(d, N - 1, 1)], d))


def _sum_faces(u, T):
    s = 0
    for d in range(3):
        lo, hi = _neighbours(u, d)
        s = s + T[d][0] * lo + T[d][1] * hi
    return s


def _apply_grid(u, T, D):
    return D * u - _sum_faces(u, T)


def _mean8(v):
    h = v.shape[0] // 2
    return v.reshape(h, 2, h, 2, h, 2).mean((1, 3, 5))


class _Grid:
    """V(2,2) cycles with red-black Gauss-Seidel on one grid, coarse levels from the mean k of the eight children."""

    def __init__(self, R, n, k):
        self.levels = []
        N = R * n
        while True:
            T = _faces(k, N)
            D = sum(t[0] + t[1] for t in T)
            i = torch.arange(N, device="cuda")
            colour = (i[:, None, None] + i[:, None] + i) % 2
            self.levels.append((N, T, D, colour == 0))
            if N // R <= 4 and (N ** 3 <= 512 or N % 8):
                break
            N, k = N // 2, None if k is None else _mean8(k)
        eye = torch.eye(N ** 3, dtype=F64, device="cuda").reshape(-1, N, N, N)
        A = torch.stack([_apply_grid(e, T, D).reshape(-1) for e in eye], 1)
        self.inverse = torch.linalg.inv(A)

    def sweep(self, u, f, l):
        N, T, D, red = self.levels[l]
        for mask in (red, ~red):
            u = torch.where(mask, (f + _sum_faces(u, T)) / D, u)
        return u

    def cycle(self, u, f, l=0):
        N, T, D, _ = self.levels[l]
        if l == len(self.levels) - 1:
            return (self.inverse @ f.reshape(-1)).reshape(f.shape)
        u = self.sweep(self.sweep(u, f, l), f, l)
        e = self.cycle(torch.zeros(N // 2, N // 2, N // 2, dtype=F64, device="cuda"),
                       _mean8(f - _apply_grid(u, T, D)), l + 1)
        near = [_neighbours(e, d) for d in range(3)]
        u = u.clone()
        for a, b, c in itertools.product((0, 1), repeat=3):
            u[a::2, b::2, c::2] += 0.25 * (e + near[0][a] + near[1][b] + near[2][c])
        return self.sweep(self.sweep(u, f, l), f, l)

    def solve(self, f):
        N, T, D, _ = self.levels[0]
        u, last = torch.zeros_like(f), math.inf
        for _ in range(60):  # until rounding stops it
            u = self.cycle(u, f)
            now = float((f - _apply_grid(u, T, D)).norm() / f.norm())
            if now < 1e-14 or (now < 1e-11 and now > 0.7 * last):
                break
            last = now
        return u


# The quadratic coarse-to-fine rule of the paper's Sec. 3.3.2 in one tangential direction: the values at the n fine
# cells over half `seg` of a coarse block edge, from the n coarse cells along it.
def _tangential(n, seg):
    W = torch.zeros(n, n, dtype=F64)
    for i in range(n):
        c = seg * (n // 2) + i // 2
        at = (c, c + 1, c + 2) if c == 0 else (c - 2, c - 1, c) if c == n - 1 else (c - 1, c, c + 1)
        t = c + (0.25 if i % 2 else -0.25)
        for a in at:
            W[i, a] = math.prod((t - b) / (a - b) for b in at if b != a)
    return W.cuda()


def _operator(case, leaves, u, k):
    """A u on any forest, in torch operations that can be differentiated.  u, k: (leaves, n, n, n) as [z, y, x]."""
    n, h = case["n"], case["n"] // 2
    index = {key: b for b, key in enumerate(leaves)}
    W = [_tangential(n, s) for s in (0, 1)]
    N2 = torch.tensor([(case["R"] * n * 2.0 ** key[0]) ** 2 for key in leaves], dtype=F64, device="cuda")
    out = torch.zeros_like(u)
    mean = lambda v: v.reshape(-1, h, 2, h, 2).mean((2, 4))  # noqa: E731
    for axis in range(3):
        d = 3 - axis  # u's dimension of that axis; the other two keep their order (second, first)
        U, K = u.movedim(d, 1), k.movedim(d, 1)
        T = 2 * K[:, 1:] * K[:, :-1] / (K[:, 1:] + K[:, :-1])
        flow = T * (U[:, 1:] - U[:, :-1])
        row = torch.cat([-flow, torch.zeros_like(U[:, :1])], 1) + torch.cat([torch.zeros_like(U[:, :1]), flow], 1)
        for side in (0, 1):
            layer = lambda v, blocks, s, depth=0: v[blocks][:, n - 1 - depth if s else depth]  # noqa: E731
            kinds = {"boundary": [], "same": [], "fine": [], "coarse": []}
            for b, key in enumerate(leaves):
                l, p = key[0], list(key[1:])
                p[axis] += 1 if side else -1
                if not 0 <= p[axis] < case["R"] * 2 ** l:
                    kinds["boundary"].append((b, b))
                elif (l, *p) in index:
                    kinds["same"].append((b, index[(l, *p)]))
                elif (l - 1, *(q >> 1 for q in p)) in index:  # this block is the finer one
                    t = [q & 1 for i, q in enumerate(key[1:]) if i != axis]
                    kinds["fine"].append((b, index[(l - 1, *(q >> 1 for q in p))], t[0], t[1]))
            end = n - 1 if side else 0
            for kind in ("boundary", "same"):
                if kinds[kind]:
                    b, o = (torch.tensor(v, device="cuda") for v in zip(*kinds[kind]))
                    ui, ki = layer(U, b, side), layer(K, b, side)
                    ug, kg = (-ui, ki) if kind == "boundary" else (layer(U, o, 1 - side), layer(K, o, 1 - side))
                    term = 2 * ki * kg / (ki + kg) * (ui - ug)
                    row = row.index_put((b, torch.full_like(b, end)), term, accumulate=True)
            for s1, s2 in itertools.product((0, 1), repeat=2):
                group = [v[:2] for v in kinds["fine"] if v[2:] == (s1, s2)]
                if not group:
                    continue
                b, o = (torch.tensor(v, device="cuda") for v in zip(*group))
                normal = sum(w / 32 * layer(U, o, 1 - side, i) for i, w in enumerate((45.0, -18.0, 5.0)))
                ug = W[s2] @ normal @ W[s1].T
                quarter = lambda v: v[:, s2 * h:(s2 + 1) * h, s1 * h:(s1 + 1) * h]  # noqa: E731
                kC = quarter(layer(K, o, 1 - side))
                kg = kC.repeat_interleave(2, 1).repeat_interleave(2, 2)
                ui, ki = layer(U, b, side), layer(K, b, side)
                flux = 2 * ki * kg / (ki + kg) * (ui - ug)
                row = row.index_put((b, torch.full_like(b, end)), flux, accumulate=True)
                if case["flux"]:  # the coarse flux is the sum of the four fine ones (per coarse face area)
                    back = -2 * mean(flux)
                else:  # the coarse ghost is the mean of the eight fine cells behind it
                    uC = quarter(layer(U, o, 1 - side))
                    ghost = 0.5 * (mean(ui) + mean(layer(U, b, side, 1)))
                    kf = 0.5 * (mean(ki) + mean(layer(K, b, side, 1)))
                    back = 2 * kC * kf / (kC + kf) * (uC - ghost)
                full = torch.zeros(len(group), n, n, dtype=F64, device="cuda")
                full[:, s2 * h:(s2 + 1) * h, s1 * h:(s1 + 1) * h] = 1
                spread = torch.zeros_like(full).masked_scatter(full.bool(), back.reshape(-1))
                row = row.index_put((o, torch.full_like(o, n - 1 - end)), spread, accumulate=True)
        out = out + row.movedim(1, d)
    return out * N2[:, None, None, None]


def exact(case, seed):
    """None where plain torch has no direct way: solves on refined forests (the multigrid hierarchy itself would have to
    be written again) and batches of them."""
    if case["kind"] == "batch" or case["smoother"] != "rbgs":
        return None
    R, n = case["R"], case["n"]
    leaves, d = _inputs(case, seed)
    if case["kind"] == "operator":
        u = d["f"].reshape(-1, n, n, n).requires_grad_()
        k = d["k"].reshape(u.shape) if case["k"] else torch.ones_like(u).detach()
        Au = _operator(case, leaves, u, k)
        ATu, = torch.autograd.grad(Au, u, u.detach())
        return {"Au": Au.detach().reshape(d["f"].shape), "ATu": ATu.reshape(d["f"].shape)}
    if case["refine"] != "none" or (case["kind"] == "cycles" and case["coarse"] != "k"):
        return None
    f = _to_grid(d["f"], R, n)
    k = _to_grid(d["k"], R, n) if case["k"] else None
    grid = _Grid(R, n, k)
    if case["kind"] == "cycles":
        u = torch.zeros_like(f)
        for _ in range(case["cycles"]):
            u = grid.cycle(u, f)
        return {"u": _from_grid(u, R, n)}
    u = grid.solve(f)
    if case["kind"] != "gradient":
        return {"u": _from_grid(u, R, n), "cycles": None}
    lam = grid.solve(u - _to_grid(d["target"], R, n))  # A is symmetric on one grid
    k.requires_grad_()
    T = _faces(k, R * n)
    dk, = torch.autograd.grad(-(lam * _apply_grid(u, T, sum(t[0] + t[1] for t in T))).sum(), k)
    return {key: _from_grid(v, R, n) for key, v in (("u", u), ("df", lam), ("dk", dk))}
