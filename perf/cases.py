"""Cases for timing the library through its C ABI (paper_1908_08666_gb300.binding), and a plain
64-bit restatement of what each of them computes.

Meshes are boxes of nx x ny x nz cubes, each split into six Kuhn tetrahedra (1 x 1 x 1 is the
6-macro cube, 4 x 4 x 4 the 384-macro elastostatics mesh), refined to `level`; `skew` moves the
macro vertices so that no macro is axis-aligned.  The mesh, the problem and the coefficient
belong to the context, which a program sets up once; x, f and u come from the seed."""

import itertools
import math

import numpy as np
import torch

from paper_1908_08666_gb300 import binding as B

PERMS = tuple(itertools.permutations(range(3)))
DEV = "cuda"
LAM_STEPS = 15  # power iterations of the multigrid setup


def listed():
    return [
        # a coarse grid, or one call inside a solver's inner loop: launches and latency count
        dict(name="apply_small", op="apply", nx=1, ny=1, nz=1, skew=False, level=4, dt="f32", variant="physical", nu=0.3),
        # the benchmark's workload: one FP32 operator application on 129^3 nodes
        dict(name="apply_cube", op="apply", nx=1, ny=1, nz=1, skew=False, level=7, dt="f32", variant="physical", nu=0.3),
        # the same on 257^3 nodes (the size of the Carreau and learned-preconditioner runs)
        dict(name="apply_large", op="apply", nx=1, ny=1, nz=1, skew=False, level=8, dt="f32", variant="physical", nu=0.3),
        # an unstructured mesh of many macros (the elastostatics mesh, moved vertices)
        dict(name="apply_many_macros", op="apply", nx=4, ny=4, nz=4, skew=True, level=5, dt="f32", variant="physical", nu=0.3),
        # the outer residual of FP64 iterative refinement, with its norm
        dict(name="residual_f64", op="residual", nx=1, ny=1, nz=1, skew=False, level=7, dt="f64", variant="physical", nu=0.3),
        # the preconditioner of the FP32 solvers: one V(2,2) cycle with Chebyshev smoothing
        dict(name="vcycle_cheby", op="vcycle", nx=1, ny=1, nz=1, skew=False, level=7, dt="f32", smoother="cheby", steps=2, nu=0.3),
        # the paper's solver: one FP64 V(3,3) cycle with hybrid Gauss-Seidel smoothing
        dict(name="vcycle_gs", op="vcycle", nx=2, ny=2, nz=2, skew=False, level=5, dt="f64", smoother="gs", steps=3, nu=0.34),
        # the saddle operator that MINRES, the Uzawa cycle and GCR apply in every iteration
        dict(name="stokes_apply", op="stokes_apply", nx=1, ny=1, nz=1, skew=False, level=7, dt="f32", contrast=1e3),
        # a whole solve: FP64 refinement around multigrid-preconditioned FP32 CG
        dict(name="solve_elasticity", op="solve", nx=1, ny=1, nz=1, skew=False, level=6, nu=0.3),
        # one evaluation of the nonlinear residual of a Picard iteration: the viscosity of u, the
        # new coefficient, the FP64 saddle residual with it
        dict(name="picard_residual", op="picard_residual", nx=1, ny=1, nz=1, skew=False, level=6, kappa=1.0),
        # the learned preconditioner's network on the node grid of level 7
        dict(name="network_forward", op="forward", B=1, D=129, H=129, W=129),
        # one training step's loss and gradient: 8 crops of 32^3 voxels
        dict(name="network_gradient", op="gradient", B=8, D=32, H=32, W=32),
    ]


def _box(rng, lo, hi, least=3):
    """A mesh and level with lo..hi unique nodes, spread over the logarithm of that range."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    m = rng.choice([1, 1, 2, 3, 4])
    nx, ny, nz = (rng.randint(max(1, m - 1), m) for _ in range(3))
    level = int(round(math.log2(max(1.0, (want / (nx * ny * nz)) ** (1 / 3)))))
    level = max(least, min(8, level))
    while level > 2 and _nodes(dict(nx=nx, ny=ny, nz=nz, level=level)) > hi:
        level -= 1
    return dict(nx=nx, ny=ny, nz=nz, skew=rng.random() < 0.4, level=level)


def draw(rng):
    op = rng.choice(["apply"] * 4 + ["residual"] * 2 + ["vcycle"] * 3 + ["stokes_apply"] * 2 + ["solve", "picard_residual", "forward", "gradient"])
    nu = round(rng.uniform(0.1, 0.42), 4)
    if op == "apply":
        c = dict(op=op, **_box(rng, 700, 17e6), dt="f32", variant=rng.choice(["physical"] * 5 + ["unphysical", "bf16", "edge"]), nu=nu)
        if c["level"] < 8 and rng.random() < 0.2:
            c["variant"] = rng.choice(["nodal", "stored"])
        return c
    if op == "residual":
        return dict(op=op, **_box(rng, 700, 2.2e6), dt=rng.choice(["f64", "f64", "f32"]), variant=rng.choice(["physical", "physical", "edge"]), nu=nu)
    if op == "vcycle":
        if rng.random() < 0.6:
            return dict(op=op, **_box(rng, 4000, 2.2e6), dt=rng.choice(["f32", "f32", "f64"]), smoother="cheby", steps=rng.choice([1, 2, 3]), nu=nu)
        return dict(op=op, **_box(rng, 4000, 2.8e5), dt=rng.choice(["f32", "f64", "f64"]), smoother="gs", steps=rng.choice([1, 2, 3]), nu=nu)
    if op == "stokes_apply":
        return dict(op=op, **_box(rng, 700, 2.2e6), dt=rng.choice(["f32", "f32", "f64"]), contrast=round(10 ** rng.uniform(0, 3), 2))
    if op == "solve":
        return dict(dict(op=op, **_box(rng, 4000, 2.8e5), nu=nu), skew=False)
    if op == "picard_residual":
        return dict(op=op, **_box(rng, 700, 2.8e5), kappa=round(10 ** rng.uniform(-1, 1), 3))
    if op == "forward":
        want = math.exp(rng.uniform(math.log(1000), math.log(2.1e6)))
        s = want ** (1 / 3)
        d, h = max(1, int(s * rng.uniform(0.6, 1.4))), max(1, int(s * rng.uniform(0.6, 1.4)))
        return dict(op=op, B=1, D=d, H=h, W=max(1, int(want / d / h)))
    e = rng.choice([15, 16, 17, 24, 29, 31, 32])
    return dict(op=op, B=rng.randint(1, 8), D=e, H=e, W=rng.randint(11, 32))


def _nodes(c):
    n = 1 << c["level"]
    return (c["nx"] * n + 1) * (c["ny"] * n + 1) * (c["nz"] * n + 1)


def work(case):
    op = case["op"]
    if op in ("forward", "gradient"):
        v = case["B"] * case["D"] * case["H"] * case["W"]
        net = 27 * 2 * (7 * 16 + 2 * 16 * 16 + 16 * 3) * v
        if op == "forward":
            return {"bytes": v * 4.0 * (7 + 3), "flops": float(net)}
        return {"bytes": v * 4.0 * (7 + 3), "flops": 3.0 * net}
    w = 8 if case.get("dt", "f64") == "f64" else 4
    u = _nodes(case)
    row = 723.0  # flops of one scaled-stencil row (14 directions, FMA = 2)
    if op == "apply":
        return {"bytes": 7.0 * w * u, "flops": row * u}
    if op == "residual":
        return {"bytes": 10.0 * w * u, "flops": row * u}
    if op == "stokes_apply":
        return {"bytes": 9.0 * w * u, "flops": (row + 14 * 16) * u}
    # levels of a cycle hold 1 + 1/8 + 1/64 + ... of the finest level's nodes
    if op == "vcycle":
        sweeps = 2 * case["steps"]
        return {"bytes": 8 / 7 * w * u * (10.0 * (sweeps + 1) + 6), "flops": 8 / 7 * row * u * (sweeps + 1)}
    if op == "solve":  # about 10 inner iterations of one cycle, one apply and the CG vectors; 4 FP64 residuals
        return {"bytes": u * (10 * 4.0 * (8 / 7 * 56 + 7 + 30) + 4 * 80.0), "flops": row * u * (10 * (8 / 7 * 5 + 1) + 4)}
    return {"bytes": 8.0 * u * (3 + 1 + 1 + 9 + 4), "flops": (row + 14 * 16 + 14 * 3 * 9) * u}  # picard_residual


# ---------------------------------------------------------------------------- meshes and fields


def _vertices(nx, ny, nz, skew):
    """Vertex coordinates over the integer grid of the box, [nx+1, ny+1, nz+1, 3]."""
    g = np.stack(np.meshgrid(*(np.arange(m + 1.0) for m in (nx, ny, nz)), indexing="ij"), axis=-1)
    v = g / max(nx, ny, nz)
    if skew:
        s = 0.13 / max(nx, ny, nz)
        v = v + s * np.sin(g @ np.array([[2.1, 1.3, 3.7], [0.9, 2.9, 1.9], [3.1, 0.7, 2.3]]) + np.array([0.3, 1.1, 2.0]))
        v = v @ np.array([[1.0, 0.15, -0.05], [0.1, 0.95, 0.2], [0.0, 0.1, 1.05]])
    return v


def _macro_mesh(nx, ny, nz, skew):
    """(xyz, tets): the tetrahedra (c, c+e_a, c+e_a+e_b, c+(1,1,1)) of every cube, in that order."""
    v = _vertices(nx, ny, nz, skew)
    ident = lambda p: (p[0] * (ny + 1) + p[1]) * (nz + 1) + p[2]  # noqa: E731
    tets = []
    for c in itertools.product(range(nx), range(ny), range(nz)):
        for a, b, _ in PERMS:
            p1 = list(c)
            p1[a] += 1
            p2 = list(p1)
            p2[b] += 1
            tets.append([ident(c), ident(p1), ident(p2), ident((c[0] + 1, c[1] + 1, c[2] + 1))])
    return v.reshape(-1, 3), np.array(tets, dtype=np.int64)


class Grid:
    """The refined mesh as a global lattice of (nx n + 1)(ny n + 1)(nz n + 1) points, and the
    library's entries on it (macro by macro; k slices, j rows, i; see include/hhg.h)."""

    def __init__(self, c, level):
        n = 1 << level
        self.n, self.box, self.skew = n, (c["nx"], c["ny"], c["nz"]), c["skew"]
        self.shape = tuple(m * n + 1 for m in self.box)
        r = torch.arange(n + 1, device=DEV)
        k, j, i = torch.nonzero(r[:, None, None] + r[None, :, None] + r[None, None, :] <= n, as_tuple=True)
        kuhn = (i + j + k, j + k, k)
        gid = []
        for cube in itertools.product(*(range(m) for m in self.box)):
            for perm in PERMS:
                g = [None] * 3
                for axis, q in zip(perm, kuhn):
                    g[axis] = q + cube[axis] * n
                gid.append((g[0] * self.shape[1] + g[1]) * self.shape[2] + g[2])
        self.gid = torch.cat(gid)  # global point of every entry
        self.points = self.shape[0] * self.shape[1] * self.shape[2]

    def entries(self, field):
        """[comps, points] -> the library's component-major entries."""
        return field.reshape(-1, self.points)[:, self.gid].reshape(-1).contiguous()

    def field(self, entries):
        """The inverse: every copy of a point holds the same value."""
        v = entries.reshape(-1, self.gid.numel())
        out = torch.zeros((v.shape[0], self.points), dtype=v.dtype, device=DEV)
        out[:, self.gid] = v
        return out.reshape(-1, *self.shape)

    def unit_coords(self):
        """Coordinates in the unmoved box, scaled to its longest side, [3, *shape]."""
        axes = [torch.arange(s, device=DEV, dtype=torch.float64) / (self.n * max(self.box)) for s in self.shape]
        return torch.stack(torch.meshgrid(*axes, indexing="ij"))

    def boundary(self):
        b = torch.zeros(self.shape, dtype=torch.bool, device=DEV)
        b[0] = b[-1] = True
        b[:, 0] = b[:, -1] = True
        b[:, :, 0] = b[:, :, -1] = True
        return b


def _uniform(points, comps, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.rand((comps, points), generator=g, device=DEV, dtype=torch.float64) * 2 - 1


def _lognormal(x):
    """A smooth lognormal modulus: exp of 32 random cosines of correlation length about 0.1."""
    rng = np.random.default_rng(2)
    s = torch.zeros_like(x[0])
    for f, p in zip(rng.normal(0.0, 1.125, (32, 3)), rng.uniform(0, 2 * math.pi, 32)):
        s += torch.cos(2 * math.pi * (f[0] * x[0] + f[1] * x[1] + f[2] * x[2]) + p)
    return torch.exp(s / 4.0)


def _sphere(x, contrast):
    """Viscosity 1 inside a sphere, `contrast` outside."""
    r = ((x - 0.5) ** 2).sum(0).sqrt()
    return 1.0 + (contrast - 1.0) * 0.5 * (1.0 + torch.tanh((r - 0.25) / 0.02))


def _smooth_velocity(x, seed):
    """A smooth velocity field of magnitude 1 (plus 1e-3 noise), as an iterate of a flow solver is."""
    rng = np.random.default_rng(seed)
    u = torch.zeros_like(x)
    for c in range(3):
        for f, p, a in zip(rng.normal(0.0, 1.5, (6, 3)), rng.uniform(0, 2 * math.pi, 6), rng.uniform(-1, 1, 6)):
            u[c] += a * torch.sin(2 * math.pi * (f[0] * x[0] + f[1] * x[1] + f[2] * x[2]) + p)
    return u + 1e-3 * _uniform(x[0].numel(), 3, seed).reshape(u.shape)


# ---------------------------------------------------------------------------- contexts

CARREAU = dict(eta0=10.0, eta_inf=0.1, r=-0.3)


def _coarsest(c):
    """The coarsest level: the direct coarse solve takes at most 3000 degrees of freedom."""
    return 2 if c["nx"] * c["ny"] * c["nz"] <= 8 else 1


class Context:
    """A library context with its mesh, problem and coefficient."""

    def __init__(self, c):
        self.h = B.hhg_create(0, torch.cuda.current_stream().cuda_stream)
        self.level = c.get("level", 2)
        op, variant = c["op"], c.get("variant", "physical")
        if op in ("forward", "gradient"):
            B.hhg_set_macro_mesh(self.h, *_macro_mesh(1, 1, 1, False))
            B.hhg_refine(self.h, 2)
            B.hhg_set_problem(self.h)
            return
        B.hhg_set_macro_mesh(self.h, *_macro_mesh(c["nx"], c["ny"], c["nz"], c["skew"]))
        B.hhg_set_coarsest_level(self.h, _coarsest(c))
        B.hhg_refine(self.h, self.level)
        self.grid = Grid(c, self.level)
        stokes = op in ("stokes_apply", "picard_residual")
        B.hhg_set_problem(
            self.h,
            kind=B.STOKES if stokes else B.ELASTICITY,
            nu=c.get("nu", 0.3),
            variant={"unphysical": B.UNPHYSICAL, "nodal": B.NODAL, "stored": B.STORED}.get(variant, B.PHYSICAL),
            khat=B.KHAT_EDGE if variant == "edge" else B.KHAT_PATCH,
        )
        if op == "picard_residual":
            return
        x = self.grid.unit_coords()
        k = self.grid.entries(_sphere(x, c["contrast"]) if stokes else _lognormal(x))
        if variant == "bf16":
            B.hhg_set_coefficient(self.h, k.to(torch.bfloat16), B.BF16)
        else:
            B.hhg_set_coefficient(self.h, k, B.F64)
        if op in ("vcycle", "solve"):
            gs, steps = c.get("smoother") == "gs", c.get("steps", 2)
            B.hhg_set_mg_params(self.h, smoother=B.SMOOTH_HYBRID_GS if gs else B.SMOOTH_CHEBYSHEV, pre=steps, post=steps, power_iters=LAM_STEPS)
            B.hhg_mg_setup(self.h)
        torch.cuda.synchronize()

    def __del__(self):
        if getattr(self, "h", None):
            torch.cuda.synchronize()
            B.hhg_destroy(self.h)
            self.h = None


_last = {}


def _context(case):
    """The context of the case's mesh and problem; the last one used is kept."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name" and not (case["op"] in ("forward", "gradient") and k in "BDHW")))
    if key not in _last:
        _last.clear()
        _last[key] = Context(case)
    return _last[key]


# ---------------------------------------------------------------------------- prepare and run


def _net_params(seed):
    """BF16-representable weights and biases of the 4 layers, in the library's layout."""
    rng = np.random.default_rng(seed)
    parts = []
    for fan, out in ((7, 16), (16, 16), (16, 16), (16, 3)):
        w = np.zeros((27, 16, 16))
        w[:, :fan, :out] = rng.normal(0.0, math.sqrt(2.0 / (27 * fan)), (27, fan, out))
        b = np.zeros(16)
        b[:out] = 0.05 * rng.normal(size=out)
        parts += [torch.as_tensor(w).to(torch.bfloat16).float().numpy().reshape(-1), b.astype(np.float32)]
    return np.concatenate(parts).astype(np.float32)


def _net_input(case, seed, channels):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = torch.randn((case["B"], case["D"], case["H"], case["W"], channels), generator=g, device=DEV)
    return x.to(torch.bfloat16).float()


def prepare(case, seed):
    ctx = _context(case)
    op = case["op"]
    s = dict(op=op, ctx=ctx, h=ctx.h, level=ctx.level)
    if op in ("forward", "gradient"):
        B.hhg_learn_set_params(ctx.h, _net_params(1))
        s["shape"] = (case["B"], case["D"], case["H"], case["W"])
        s["x"] = _net_input(case, seed, 7)
        if op == "forward":
            s["y"] = torch.empty((*s["shape"], 3), dtype=torch.float32, device=DEV)
        else:
            s["target"] = _net_input(case, seed + 1000003, 3)
        return s
    g = ctx.grid
    s["dt"] = B.F64 if case.get("dt", "f64") == "f64" else B.F32
    t = torch.float64 if s["dt"] == B.F64 else torch.float32
    if op == "picard_residual":
        s["kappa"] = case["kappa"]
        x = g.unit_coords()
        u = torch.cat([_smooth_velocity(x, seed).reshape(3, -1), 0.1 * _uniform(g.points, 1, seed + 1)])
        s["x"], s["f"] = g.entries(u), g.entries(_uniform(g.points, 4, seed + 2) / g.n**3)
        s["mu"], s["y"] = torch.empty(g.gid.numel(), dtype=t, device=DEV), torch.empty_like(s["x"])
        return s
    comps = 4 if op == "stokes_apply" else 3
    x = _uniform(g.points, comps, seed).reshape(comps, *g.shape)
    if op in ("vcycle", "solve"):
        x[:, g.boundary()] = 0.0
    if op != "solve":
        s["x"] = g.entries(x).to(t)
    if op in ("apply", "residual", "stokes_apply"):
        s["y"] = torch.empty_like(s["x"])
    if op in ("residual", "vcycle"):
        s["f"] = g.entries(_uniform(g.points, 3, seed + 1)).to(t)
    if op == "solve":
        s["f"] = g.entries(x) / g.n**3
        s["x"] = torch.empty_like(s["f"])
    return s


def run(s):
    op, h = s["op"], s["h"]
    if op == "apply":
        B.hhg_apply(h, s["level"], s["dt"], s["x"], s["y"])
        return s["y"]
    if op == "residual":
        return s["y"], B.hhg_residual(h, s["level"], s["dt"], s["f"], s["x"], s["y"], want_norm=True)
    if op == "vcycle":  # x is updated in place, as an iterate is
        B.hhg_vcycle(h, s["level"], s["dt"], s["f"], s["x"])
        return s["x"]
    if op == "stokes_apply":
        B.hhg_stokes_apply(h, s["level"], s["dt"], s["x"], s["y"])
        return s["y"]
    if op == "solve":
        s["x"].zero_()
        B.hhg_solve(h, s["f"], s["x"], method=B.SOLVE_IR_MG_CG, level=s["level"], dt=B.F64, rtol=1e-11, max_iter=30)
        return s["x"]
    if op == "picard_residual":
        B.hhg_carreau_viscosity(h, s["level"], s["x"], s["mu"], kappa=s["kappa"], **CARREAU)
        B.hhg_set_coefficient(h, s["mu"], B.F64)
        B.hhg_stokes_residual(h, s["level"], s["dt"], s["f"], s["x"], s["y"])
        return s["mu"], s["y"]
    if op == "forward":
        B.hhg_learn_forward(h, s["x"], 7, *s["shape"], s["y"])
        return s["y"]
    loss, grad = B.hhg_learn_loss_grad(h, s["x"], 7, s["target"], *s["shape"])
    return loss, grad


# ---------------------------------------------------------------------------- 64-bit restatement

DIRS = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1))


def _cells(shape, corner):
    """The view of a lattice array that holds vertex `corner` of every cell."""
    return tuple(slice(c, s - 1 + c) for c, s in zip(corner, shape))


def _shifted(shape, d):
    """Views of the lattice points p and p + d of every edge in direction d."""
    return tuple(slice(0, s - q) for s, q in zip(shape, d)), tuple(slice(q, s) for s, q in zip(shape, d))


class Elements:
    """The mesh's elements: 6 per lattice cell, each the affine image of a Kuhn simplex under the
    map of its macro."""

    def __init__(self, c, level):
        self.g = g = Grid(c, level)
        v = torch.as_tensor(_vertices(*g.box, g.skew), device=DEV)
        maps = []  # d position / d lattice coordinate of every macro
        for cube in itertools.product(*(range(m) for m in g.box)):
            for perm in PERMS:
                p, J = list(cube), torch.zeros((3, 3), dtype=torch.float64, device=DEV)
                for axis in perm:
                    q = list(p)
                    q[axis] += 1
                    J[:, axis] = (v[tuple(q)] - v[tuple(p)]) / g.n
                    p = q
                maps.append(J)
        self.J = torch.stack(maps)
        self.cells = tuple(s - 1 for s in g.shape)
        at = [torch.arange(s, device=DEV) for s in self.cells]
        cube = [a // g.n for a in at]
        self.cube = ((cube[0][:, None, None] * g.box[1] + cube[1][None, :, None]) * g.box[2] + cube[2][None, None, :]) * 6
        self.local = [(a % g.n).double().reshape([-1 if q == ax else 1 for q in range(3)]) for ax, a in enumerate(at)]

    def each(self):
        """(macro of every cell, corners of the simplex, gradients [macro, 4, 3], volume [macro])."""
        inv = torch.linalg.inv(self.J)
        vol = torch.linalg.det(self.J).abs() / 6
        for perm in PERMS:
            corners = [(0, 0, 0)]
            for axis in perm:
                q = list(corners[-1])
                q[axis] += 1
                corners.append(tuple(q))
            mid = [self.local[ax] + sum(cn[ax] for cn in corners) / 4 for ax in range(3)]
            macro = torch.zeros(self.cells, dtype=torch.int64, device=DEV)
            for m, (a, b, c) in enumerate(PERMS):
                macro = torch.where((mid[a] > mid[b]) & (mid[b] > mid[c]), m, macro)
            ref = torch.zeros((4, 3), dtype=torch.float64, device=DEV)  # gradients in lattice coordinates
            for q, axis in enumerate(perm):
                ref[q, axis] -= 1
                ref[q + 1, axis] += 1
            yield self.cube + macro, corners, torch.einsum("ax,mxy->may", ref, inv), vol


def _operator(c, level, k, ce, cd):
    """The operator as 3x3 blocks of the lattice's edges: {direction: [3, 3, *edges]}, the block of
    (p, p + d); that of (p + d, p) is its transpose, the centre blocks are minus the row sums."""
    E = Elements(c, level)
    g, variant = E.g, c.get("variant", "physical")
    n = g.n
    ah = {d: torch.zeros((3, 3, *g.shape), dtype=torch.float64, device=DEV) for d in DIRS}
    ref = {d: torch.zeros_like(ah[d]) for d in DIRS}
    ks = {d: torch.zeros((2, *g.shape), dtype=torch.float64, device=DEV) for d in DIRS}
    for macro, corners, grad, vol in E.each():
        kb = sum(k[_cells(g.shape, cn)] for cn in corners) / 4
        for a in range(4):
            for b in range(a + 1, 4):
                d = tuple(q - p for p, q in zip(corners[a], corners[b]))
                ga, gb = grad[:, a], grad[:, b]
                eye = torch.eye(3, dtype=torch.float64, device=DEV) * (ga * gb).sum(1)[:, None, None]
                K = vol[:, None, None] * (ce * 0.5 * (eye + gb[:, :, None] * ga[:, None, :]) + cd * ga[:, :, None] * gb[:, None, :])
                at = _cells(g.shape, corners[a])
                for m in range(3):
                    for l in range(3):
                        Kc = K[:, m, l][macro]
                        ref[d][m, l][at] += Kc
                        ah[d][m, l][at] += kb * Kc
                ks[d][0][at] += kb
                ks[d][1][at] += 1
    inner = torch.ones(g.shape, dtype=torch.bool, device=DEV)  # macro-interior points
    loc = [(torch.arange(s, device=DEV) % n).reshape([-1 if q == ax else 1 for q in range(3)]) for ax, s in enumerate(g.shape)]
    for q in range(3):
        inner &= (loc[q] != 0) & (loc[q] != loc[(q + 1) % 3])
    out = {}
    for d in DIRS:
        lo, hi = _shifted(g.shape, d)
        blk = ah[d][(slice(None), slice(None), *lo)].clone()
        if variant != "nodal":
            kh = 0.5 * (k[lo] + k[hi]) if variant == "edge" else (ks[d][0] / ks[d][1].clamp(min=1))[lo]
            sc = kh * ref[d][(slice(None), slice(None), *lo)]
            if variant != "unphysical":
                sc = sc + 0.5 * (blk - blk.transpose(0, 1))
            blk = torch.where(inner[lo] | inner[hi], sc, blk)
        del ah[d], ref[d], ks[d]
        out[d] = blk
    return g, out, inner


def _apply(g, blocks, x):
    y = torch.zeros_like(x)
    for d, blk in blocks.items():
        lo, hi = _shifted(g.shape, d)
        dx = [x[m][hi] - x[m][lo] for m in range(3)]
        for m in range(3):
            y[m][lo] += blk[m, 0] * dx[0] + blk[m, 1] * dx[1] + blk[m, 2] * dx[2]
            y[m][hi] -= blk[0, m] * dx[0] + blk[1, m] * dx[1] + blk[2, m] * dx[2]
    return y


def _diagonal(g, blocks):
    y = torch.zeros((3, *g.shape), dtype=torch.float64, device=DEV)
    for d, blk in blocks.items():
        lo, hi = _shifted(g.shape, d)
        for m in range(3):
            y[m][lo] -= blk[m, m]
            y[m][hi] -= blk[m, m]
    return y


def _saddle(c, level, k, x):
    """[[A, B^T], [B, C]] x on (u, v, w, p); velocity rows on the boundary are x."""
    g, blocks, _ = _operator(c, level, k, 2.0, 0.0)
    y = torch.zeros_like(x)
    y[:3] = _apply(g, blocks, x[:3])
    E = Elements(c, level)
    vol_macro = torch.linalg.det(E.J).abs() * g.n**3  # 6 |T|
    h2 = (vol_macro ** (1 / 3) / g.n) ** 2
    for macro, corners, grad, vol in E.each():
        at = [_cells(g.shape, cn) for cn in corners]
        for a in range(4):
            for b in range(4):
                lc = (-(h2 / 12) * vol * (grad[:, a] * grad[:, b]).sum(1))[macro]
                y[3][at[a]] += lc * x[3][at[b]]
                for l in range(3):
                    y[3][at[a]] += (-0.25 * vol * grad[:, b, l])[macro] * x[l][at[b]]
                    y[l][at[a]] += (-0.25 * vol * grad[:, a, l])[macro] * x[3][at[b]]
    bd = g.boundary()
    y[:3, bd] = x[:3, bd]
    return g, y


def _halves(shape):
    """For the 8 parities e of a fine lattice point: (its points, the coarse points p - e, p + e)."""
    for e in itertools.product(range(2), repeat=3):
        fine = tuple(slice(q, None, 2) for q in e)
        coarse = tuple((s + 1) // 2 for s in shape)
        yield fine, tuple(slice(0, cs - q) for cs, q in zip(coarse, e)), tuple(slice(q, cs) for cs, q in zip(coarse, e))


def _vcycle(case, level, f, x, ops, lam):
    g, blocks, inner, dia = ops[level]
    bd = g.boundary()
    if level == _coarsest(case):
        free = (~bd).flatten().nonzero().flatten()
        N = free.numel()
        M = torch.zeros((3 * N, 3 * N), dtype=torch.float64, device=DEV)
        for col in range(3 * N):
            e = torch.zeros((3, g.points), dtype=torch.float64, device=DEV)
            e[col // N, free[col % N]] = 1.0
            M[:, col] = _apply(g, blocks, e.reshape(3, *g.shape)).reshape(3, -1)[:, free].reshape(-1)
        sol = torch.linalg.solve(M, f.reshape(3, -1)[:, free].reshape(-1))
        out = torch.zeros((3, g.points), dtype=torch.float64, device=DEV)
        out[:, free] = sol.reshape(3, N)
        return out.reshape(3, *g.shape)

    def residual(x):
        r = f - _apply(g, blocks, x)
        r[:, bd] = 0
        return r

    def smooth(x):
        if case["smoother"] == "cheby":
            a, b = lam[level] / 8, 1.1 * lam[level]
            theta, delta = (a + b) / 2, (b - a) / 2
            sigma = theta / delta
            rho, d = 1 / sigma, None
            for _ in range(case["steps"]):
                if d is None:
                    d = residual(x) / dia / theta
                else:
                    rn = 1 / (2 * sigma - rho)
                    d = rn * rho * d + 2 * rn / delta * residual(x) / dia
                    rho = rn
                x = x + d
            return x
        loc = [(torch.arange(s, device=DEV) % g.n).reshape([-1 if q == ax else 1 for q in range(3)]) for ax, s in enumerate(g.shape)]
        hi = torch.maximum(torch.maximum(loc[0], loc[1]), loc[2]).expand(g.shape)
        lo = torch.minimum(torch.minimum(loc[0], loc[1]), loc[2]).expand(g.shape)
        mid = loc[0] + loc[1] + loc[2] - hi - lo
        colour = 4 * ((hi - mid) % 2) + 2 * ((mid - lo) % 2) + lo % 2  # of (i, j, k) = (hi - mid, mid - lo, lo)
        for _ in range(case["steps"]):
            x = torch.where(inner, x, x + 2 / 3 * residual(x) / dia)
            for q in range(8):
                x = torch.where(inner & (colour == q), x + residual(x) / dia, x)
        return x

    x = smooth(x)
    r = residual(x)
    gc = ops[level - 1][0]
    rc = torch.zeros((3, *gc.shape), dtype=torch.float64, device=DEV)
    for fine, p, q in _halves(g.shape):
        rc[(slice(None), *p)] += 0.5 * r[(slice(None), *fine)]
        rc[(slice(None), *q)] += 0.5 * r[(slice(None), *fine)]
    rc[:, gc.boundary()] = 0
    xc = _vcycle(case, level - 1, rc, torch.zeros_like(rc), ops, lam)
    x = x.clone()
    for fine, p, q in _halves(g.shape):
        x[(slice(None), *fine)] += 0.5 * (xc[(slice(None), *p)] + xc[(slice(None), *q)])
    return smooth(x)


def _positions(g):
    """Node positions, [3, *shape]: affine in every macro."""
    v = torch.as_tensor(_vertices(*g.box, g.skew), device=DEV)
    idx = [torch.arange(s, device=DEV) for s in g.shape]
    cube = [torch.clamp(a // g.n, max=m - 1) for a, m in zip(idx, g.box)]
    loc = [(a - q * g.n).double() / g.n for a, q in zip(idx, cube)]
    base = torch.meshgrid(*cube, indexing="ij")
    t = torch.stack(torch.meshgrid(*loc, indexing="ij"), -1)
    order = torch.argsort(t, dim=-1, descending=True, stable=True)
    at = [b.clone() for b in base]
    pos = v[at[0], at[1], at[2]].clone()
    for q in range(3):
        axis = order[..., q]
        for m in range(3):
            at[m] = at[m] + (axis == m)
        nxt = v[at[0], at[1], at[2]]
        before = v[at[0] - (axis == 0).long(), at[1] - (axis == 1).long(), at[2] - (axis == 2).long()]
        pos += torch.gather(t, -1, axis[..., None]) * (nxt - before)
    return pos.movedim(-1, 0)


def _viscosity(g, u, kappa):
    """Carreau viscosity of the affine least-squares velocity gradient over the mesh neighbours."""
    pos = _positions(g)
    cnt = torch.ones(g.shape, dtype=torch.float64, device=DEV)
    s1 = torch.zeros((3, *g.shape), dtype=torch.float64, device=DEV)
    t0, s2, t1 = torch.zeros_like(s1), torch.zeros((3, 3, *g.shape), dtype=torch.float64, device=DEV), torch.zeros((3, 3, *g.shape), dtype=torch.float64, device=DEV)
    for d in DIRS:
        lo, hi = _shifted(g.shape, d)
        dx, du = pos[(slice(None), *hi)] - pos[(slice(None), *lo)], u[(slice(None), *hi)] - u[(slice(None), *lo)]
        for at, sign in ((lo, 1.0), (hi, -1.0)):
            w = (slice(None), *at)
            cnt[at] += 1
            s1[w] += sign * dx
            t0[w] += sign * du
            s2[(slice(None), *w)] += dx[:, None] * dx[None, :]
            t1[(slice(None), *w)] += dx[:, None] * du[None, :]
    cov = (s2 - s1[:, None] * s1[None, :] / cnt).movedim((0, 1), (-2, -1))
    cross = (t1 - s1[:, None] * t0[None, :] / cnt).movedim((0, 1), (-2, -1))
    adj = torch.stack([torch.linalg.cross(cov[..., 1, :], cov[..., 2, :]), torch.linalg.cross(cov[..., 2, :], cov[..., 0, :]), torch.linalg.cross(cov[..., 0, :], cov[..., 1, :])], -1)
    det = (cov[..., 0, :] * adj[..., :, 0]).sum(-1)
    grad = adj @ cross / det[..., None, None]
    e = 0.5 * (grad + grad.transpose(-1, -2))
    e2 = (e * e).sum((-1, -2))
    p = CARREAU
    return p["eta_inf"] + (p["eta0"] - p["eta_inf"]) * (1 + kappa * e2) ** p["r"]


def _network(params, x, grad=False):
    """The 4 layers in 64 bits, as 27 shifted products per layer; x [B, D, H, W, 7]."""
    p = torch.as_tensor(params, dtype=torch.float64, device=DEV).requires_grad_(grad)
    a = torch.nn.functional.pad(x.double(), (0, 9))
    for layer in range(4):
        w, b = p[layer * 6928:layer * 6928 + 6912].reshape(27, 16, 16), p[layer * 6928 + 6912:(layer + 1) * 6928]
        z = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1, 1, 1))
        D, H, W = a.shape[1:4]
        y = b
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            y = y + z[:, dz:dz + D, dy:dy + H, dx:dx + W] @ w[t]
        a = torch.relu(y) if layer < 3 else y
    return a[..., :3], p


def exact(case, seed):
    op = case["op"]
    if op == "forward":
        with torch.no_grad():
            return _network(_net_params(1), _net_input(case, seed, 7))[0]
    if op == "gradient":
        y, p = _network(_net_params(1), _net_input(case, seed, 7), grad=True)
        loss = ((y - _net_input(case, seed + 1000003, 3).double()) ** 2).mean()
        loss.backward()
        return torch.as_tensor(loss.item(), dtype=torch.float64), p.grad
    level = case["level"]
    g = Grid(case, level)
    x0 = g.unit_coords()
    t = torch.float64 if case.get("dt", "f64") == "f64" else torch.float32
    if op == "picard_residual":
        u = torch.cat([_smooth_velocity(x0, seed).reshape(3, -1), 0.1 * _uniform(g.points, 1, seed + 1)]).reshape(4, *g.shape)
        f = (_uniform(g.points, 4, seed + 2) / g.n**3).reshape(4, *g.shape)
        mu = _viscosity(g, u[:3], case["kappa"])
        r = f - _saddle(case, level, mu, u)[1]
        r[:3, g.boundary()] = 0
        return g.entries(mu[None]), g.entries(r)
    stokes = op == "stokes_apply"
    x = _uniform(g.points, 4 if stokes else 3, seed).reshape(-1, *g.shape)
    if stokes:
        x = x.to(t).double()
        return g.entries(_saddle(case, level, _sphere(x0, case["contrast"]), x)[1])
    bd = g.boundary()
    k = _lognormal(x0)
    if case.get("variant") == "bf16":
        k = k.to(torch.bfloat16).double()
    nu = case["nu"]
    ce, cd = 1 / (1 + nu), nu / ((1 + nu) * (1 - 2 * nu))
    if op == "vcycle":
        x[:, bd] = 0
        f = _uniform(g.points, 3, seed + 1).to(t).double().reshape(3, *g.shape)
        h = _context(case).h
        ops, lam = {}, {}
        for l in range(_coarsest(case), level + 1):
            st = 1 << (level - l)
            gl, blocks, inner = _operator(case, l, k[::st, ::st, ::st].contiguous(), ce, cd)
            dia = _diagonal(gl, blocks)
            dia[:, gl.boundary()] = 1
            ops[l] = (gl, blocks, inner, dia)
            if case["smoother"] == "cheby" and l > _coarsest(case):
                lam[l] = B.hhg_get_lambda_max(h, l)  # the smoother's interval is set from the setup's estimate
        return g.entries(_vcycle(case, level, f, x.to(t).double(), ops, lam))
    _, blocks, _ = _operator(case, level, k, ce, cd)
    if op == "apply":
        x = x.to(t).double()
        y = _apply(g, blocks, x)
        y[:, bd] = x[:, bd]
        return g.entries(y)
    if op == "residual":
        f = _uniform(g.points, 3, seed + 1).to(t).double().reshape(3, *g.shape)
        r = f - _apply(g, blocks, x.to(t).double())
        r[:, bd] = 0
        return g.entries(r), torch.as_tensor((r * r).sum().item(), dtype=torch.float64)
    # solve: Jacobi-preconditioned CG to the limit of 64 bits
    x[:, bd] = 0
    f = x / g.n**3
    dia = _diagonal(g, blocks)
    dia[:, bd] = 1
    sol, r = torch.zeros_like(f), f.clone()
    z = r / dia
    p, rz = z.clone(), (r * z).sum()
    r0 = (r * r).sum()
    for _ in range(4000):
        q = _apply(g, blocks, p)
        q[:, bd] = 0
        alpha = rz / (p * q).sum()
        sol += alpha * p
        r -= alpha * q
        if (r * r).sum() < 1e-30 * r0:
            break
        z = r / dia
        rz, old = (r * z).sum(), rz
        p = z + rz / old * p
    return g.entries(sol)
