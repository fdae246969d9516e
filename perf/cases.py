"""What this library's users run it for, as cases that can be timed.

A program builds a hierarchy for a triangle mesh once and keeps it; then it assembles, projects
right-hand sides, and smooths, cycles or solves, many times, on new data.  A case names a mesh, a
grid depth, a number of right-hand sides, a precision and what one pass does:

  smooth    `sweeps` Gauss-Seidel sweeps of the finest level (a smoother inside the caller's own solver)
  transfer  residual, restriction and prolongation of the finest level (the caller's own two-grid method)
  cycle     `cycles` V(2,2) cycles from zero (the caller's own outer iteration, fixed cost)
  step      one implicit step: assembly, projection of vertex values, solve to `tol`, vertex evaluation
  flow      one step of conformalized mean-curvature flow from given vertex positions
  batch     a projected right-hand side solved on many meshes at once

The hierarchy (and, where a pass does not assemble, its matrices) belongs to the plan that a program
keeps; vertex values, positions, right-hand sides and starts are the inputs, made from the seed.  Mixed
precision carries single-precision accuracy (its cycles run in FP32 and its solves stop at 1e-6), so a
program takes its results as float32; FP64 results stay float64.
"""
import math
import sys

import numpy as np
import torch

import meshgen
import paper_1505_03615_gb300 as lb

F64 = torch.float64


# ---- the cases -------------------------------------------------------------------------------------

def listed():
    sphere = dict(mesh="sphere", a=3, b=0, depth=5, t=1e-3)        # 1,280 triangles
    torus = dict(mesh="torus", a=361, b=111, depth=7, t=1e-3)      # 80,142 triangles
    knot = dict(mesh="knot23", a=1000, b=100, depth=8, t=1e-4)     # 200,000 triangles
    sheet = dict(mesh="sheet", a=500, b=0, depth=9, t=1e-3)        # 1,000,000 triangles
    fine = dict(mesh="knot35", a=5000, b=100, depth=10, t=1e-4)    # 1,000,000 triangles
    return [
        # a small scan kept in double precision, a scalar field smoothed to full accuracy
        dict(name="sphere_step_f64_r1", kind="step", nrhs=1, fp64=True, solver="cg", tol=1e-10, **sphere),
        # a few cycles on the same small surface inside an interactive tool: all latency
        dict(name="sphere_cycle_mixed_r1", kind="cycle", nrhs=1, fp64=False, cycles=4, **sphere),
        # smoothing two-component texture coordinates on a mid-sized surface with odd counts
        dict(name="torus_smooth_mixed_r2", kind="smooth", nrhs=2, fp64=False, sweeps=2, **torus),
        # positions of a 200k-triangle model through one implicit mean-curvature step, the paper's cycles
        dict(name="knot200k_step_mixed_r3", kind="step", nrhs=3, fp64=False, solver="cycles", tol=1e-6, **knot),
        # the same model's double-precision cycle as a preconditioner of the caller's own solver
        dict(name="knot200k_cycle_f64_r3", kind="cycle", nrhs=3, fp64=True, cycles=4, **knot),
        # one flow step of that model, conjugate gradients
        dict(name="knot200k_flow_mixed_r3", kind="flow", nrhs=3, fp64=False, solver="cg", tol=1e-6, **knot),
        # a caller's own two-grid method on four fields (colour and alpha)
        dict(name="knot200k_transfer_f64_r4", kind="transfer", nrhs=4, fp64=True, **knot),
        # a scalar field on two nearly touching sheets of a million triangles
        dict(name="sheet1m_cycle_mixed_r1", kind="cycle", nrhs=1, fp64=False, cycles=4, **sheet),
        # many uneven meshes solved together
        dict(name="batch12_mixed_r1", kind="batch", nrhs=1, fp64=False, tol=1e-6, count=12, lo=10_000, hi=60_000,
             mesh="mix", mseed=7, t=1e-3),
        # double-precision smoothing of positions on the deepest grid
        dict(name="knot1m_smooth_f64_r3", kind="smooth", nrhs=3, fp64=True, sweeps=2, **fine),
        # the fixed-cost mixed iteration on the deepest grid
        dict(name="knot1m_cycle_mixed_r3", kind="cycle", nrhs=3, fp64=False, cycles=8, **fine),
        # a whole implicit step there, the largest call
        dict(name="knot1m_step_mixed_r3", kind="step", nrhs=3, fp64=False, solver="cg", tol=1e-6, **fine),
    ]


def _depth(tris):
    """The grid depth a mesh of that many triangles is given (finest voxels about as wide as a few triangles)."""
    return 5 if tris < 3_000 else 6 if tris < 15_000 else 7 if tris < 100_000 else 8 if tris < 400_000 else 9


def draw(rng):
    kind = rng.choice(["smooth", "smooth", "cycle", "cycle", "cycle", "transfer", "step", "step", "flow", "batch"])
    fp64 = rng.random() < 0.4
    nrhs = rng.randint(1, 4)
    if kind == "batch":
        return dict(kind=kind, nrhs=nrhs, fp64=fp64, tol=1e-6, count=rng.randint(2, 10), lo=2_000, hi=40_000,
                    mesh="mix", mseed=rng.randint(1, 10_000), t=1e-3)
    tris = math.exp(rng.uniform(math.log(1_500), math.log(600_000)))
    mesh = rng.choice(["torus", "knot23", "knot35", "sheet", "bumpy"])
    if mesh == "bumpy":
        a, b = max(3, min(6, round(math.log(tris / 20) / math.log(4)))), rng.randint(1, 1000)
        tris = 20 * 4 ** a
    elif mesh == "sheet":
        a, b = max(20, round(math.sqrt(tris / 4))), 0
        tris = 4 * a * a
    else:
        b = rng.randint(12, 120)
        a = max(40, round(tris / (2 * b)))
        tris = 2 * a * b
    case = dict(kind=kind, mesh=mesh, a=a, b=b, depth=_depth(tris) - (1 if mesh == "sheet" and tris >= 400_000 else 0),
                t=rng.choice([1e-4, 1e-3, 1e-2]), nrhs=3 if kind == "flow" else nrhs, fp64=fp64)
    if kind == "smooth":
        case["sweeps"] = rng.randint(1, 4)
    elif kind == "transfer":
        case["fp64"] = True   # the transfers are FP64 calls
    elif kind == "cycle":
        case["cycles"] = rng.randint(1, 6)
    elif kind in ("step", "flow"):
        case.update(solver="cg", tol=1e-9 if fp64 else 1e-6)
    return case


# ---- plans: the hierarchy a program keeps ----------------------------------------------------------

def _mesh(case):
    m, a, b = case["mesh"], case["a"], case["b"]
    if m == "sphere":
        return meshgen.icosphere(a, 1.0, 1e-3, 1)
    if m == "bumpy":
        return meshgen.bumpy_sphere(a, seed=b)
    if m == "torus":
        return meshgen.torus(1.0, 0.3, a, b)
    if m == "knot23":
        return meshgen.torus_knot_tube(2, 3, 1.0, 0.04, a, b, 1e-6, 2)
    if m == "knot35":
        return meshgen.torus_knot_tube(3, 5, 1.0, 0.02, a, b, 1e-7, 6)
    return meshgen.double_sheet(a, 0.05, case["depth"], 0.5, 1e-6, 4)


class _Plan:
    """A built and once assembled hierarchy, destroyed with its last user."""

    def __init__(self, case):
        if case["kind"] == "batch":
            meshes = meshgen.batch_mix(case["count"], case["lo"], case["hi"], case["mseed"])
            self.V = np.concatenate([v for v, _, _ in meshes])
            self.h = lb.lbmg_build_batch(meshes)
        else:
            self.V, F = _mesh(case)
            self.h = lb.lbmg_build_hierarchy(self.V, F, case["depth"])
        self.d0, self.D = lb.lbmg_levels(self.h)
        self.sizes = {d: lb.lbmg_level_info(self.h, d)[:2] for d in range(self.d0, self.D + 1)}
        self.n = self.sizes[self.D][0]
        self.nv = self.V.shape[0]
        lb.lbmg_assemble(self.h, case["t"])

    def __del__(self, destroy=lb.lbmg_destroy, leaving=sys.is_finalizing):
        if getattr(self, "h", None) is not None and not leaving():
            destroy(self.h)


_kept = {}


def _plan(case):
    """The plan of this mesh; a program that moves to another mesh gives the last one back."""
    key = tuple((k, case[k]) for k in sorted(case) if k not in ("name", "nrhs", "fp64", "solver", "tol", "sweeps", "cycles"))
    if key not in _kept:
        _kept.clear()
        _kept[key] = _Plan(case)
    return _kept[key]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _values(plan, nrhs, g, positions):
    """Vertex values.  For a whole step a rotated, noisy copy of the coordinates (and noise alone in a single
    or fourth column), as positions, texture coordinates and measured fields are; else noise, as the
    residuals are that a caller's own iteration smooths and cycles on."""
    V = torch.tensor(plan.V, dtype=F64, device="cuda")
    noise = torch.rand((plan.nv, nrhs), dtype=F64, device="cuda", generator=g) * 2 - 1
    if nrhs == 1 or not positions:
        return noise
    q, _ = torch.linalg.qr(torch.randn((3, 3), dtype=F64, device="cuda", generator=g))
    f = 0.3 * noise
    k = min(nrhs, 3)
    f[:, :k] += (V @ q)[:, :k]
    return f.contiguous()


def prepare(case, seed):
    plan = _plan(case)
    g = _gen(seed)
    nrhs, kind = case["nrhs"], case["kind"]
    s = dict(case=dict(case), plan=plan, prec=lb.LBMG_FP64 if case["fp64"] else lb.LBMG_MIXED)

    def vec(n=plan.n):
        return torch.zeros((n, nrhs), dtype=F64, device="cuda")

    def project():
        rhs = vec()
        lb.lbmg_project_rhs(plan.h, _values(plan, nrhs, g, False), rhs)
        return rhs

    if kind == "flow":
        V = torch.tensor(plan.V, dtype=F64, device="cuda")
        q, _ = torch.linalg.qr(torch.randn((3, 3), dtype=F64, device="cuda", generator=g))
        stretch = 0.9 + 0.2 * torch.rand(3, dtype=F64, device="cuda", generator=g)
        s.update(X=((V * stretch) @ q).contiguous(), x=vec(), X_next=torch.zeros((plan.nv, 3), dtype=F64, device="cuda"))
    elif kind == "step":
        s.update(f=_values(plan, nrhs, g, True), rhs=vec(), x=vec(), u=torch.zeros((plan.nv, nrhs), dtype=F64, device="cuda"))
    elif kind == "transfer":
        s.update(rhs=project(), x0=torch.rand((plan.n, nrhs), dtype=F64, device="cuda", generator=g), r=vec(),
                 rc=vec(plan.sizes[plan.D - 1][0]), x=vec())
    elif kind == "smooth":
        s.update(rhs=project(), x0=torch.rand((plan.n, nrhs), dtype=F64, device="cuda", generator=g), x=vec())
    else:
        s.update(rhs=project(), x=vec())
    return s


def _out(s, v):
    return v if s["case"]["fp64"] else v.float()


def run(s):
    c, p, prec = s["case"], s["plan"], s["prec"]
    h, kind = p.h, c["kind"]
    if kind == "smooth":
        s["x"].copy_(s["x0"])
        lb.lbmg_smooth(h, p.D, s["rhs"], s["x"], c["sweeps"], prec)
        return _out(s, s["x"])
    if kind == "transfer":
        lb.lbmg_residual(h, p.D, s["rhs"], s["x0"], s["r"])
        lb.lbmg_restrict(h, p.D, s["r"], s["rc"])
        s["x"].copy_(s["x0"])
        lb.lbmg_prolong_add(h, p.D, s["rc"], s["x"])
        return [s["r"], s["rc"], s["x"]]
    if kind == "cycle":
        s["x"].zero_()
        lb.lbmg_vcycles(h, s["rhs"], s["x"], c["cycles"], prec)
        return _out(s, s["x"])
    if kind == "batch":
        s["x"].zero_()
        lb.lbmg_solve_pcg(h, s["rhs"], s["x"], c["tol"], 500, prec)
        return _out(s, s["x"])
    s["x"].zero_()
    if kind == "flow":
        lb.lbmg_cmcf_step(h, s["X"], c["t"], s["x"], c["tol"], 500, prec, s["X_next"], solver=1)
        return [_out(s, s["x"]), _out(s, s["X_next"])]
    lb.lbmg_assemble(h, c["t"])
    lb.lbmg_project_rhs(h, s["f"], s["rhs"])
    solve = lb.lbmg_solve_pcg if c["solver"] == "cg" else lb.lbmg_solve
    solve(h, s["rhs"], s["x"], c["tol"], 2000, prec)
    lb.lbmg_eval_vertices(h, s["x"], s["u"])
    return [s["rhs"], _out(s, s["x"]), _out(s, s["u"])]


# ---- the work of a pass ----------------------------------------------------------------------------

# iterations that a solve of the seeded meshes takes to its tolerance (about): they set its work
_ITERS = dict(cg=45, cycles=110, flow=25, batch=150)


def work(case):
    """Bytes and operations of one pass.  Each sweep, residual and transfer reads its matrix or stencil
    entries once (value and column: 8 bytes in FP32, 12 in FP64) and its vectors once, and writes its
    result once; the grids are 1/3 of the finest one below it, taken together.  An assembly reads one mass
    and one stiffness integral per piece and pair of functions and writes both matrices."""
    p = _plan(case)
    n, nnz = p.sizes[p.D]
    R, w = case["nrhs"], 8 if case["fp64"] else 4
    sweep = (nnz * (4 + w) + 3 * n * R * w, 2 * nnz * R)
    outer = (nnz * 12 + 3 * n * R * 8, 2 * nnz * R)
    kind = case["kind"]
    rows = sum(v[0] for v in p.sizes.values()) / n
    cyc = (rows * (5 * sweep[0] + 4 * n * R * w) + outer[0], rows * (5 * sweep[1] + 32 * n * R) + outer[1])
    if kind == "smooth":
        k = case["sweeps"]
        return {"bytes": k * sweep[0], "flops": k * sweep[1]}
    if kind == "transfer":
        return {"bytes": outer[0] + 2 * (n + p.sizes[p.D - 1][0]) * R * 8 + n * R * 8, "flops": outer[1] + 32 * n * R}
    if kind == "cycle":
        k = case["cycles"]
        return {"bytes": k * cyc[0], "flops": k * cyc[1]}
    iters = _ITERS[kind if kind in _ITERS else case["solver"]]
    b, f = iters * cyc[0], iters * cyc[1]
    if kind in ("step", "flow"):
        nfrag = lb.lbmg_level_info(p.h, p.D)[2]
        b += nfrag * 36 * 16 + rows * nnz * 28 + nfrag * 27 * 8 + p.nv * R * 16
        f += nfrag * 72 * 2 + nfrag * 8 * R * 8
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, in plain torch -----------------------------------------------------------

def _csr(plan, case, d):
    """A_d = M_d + t L_d of the plan as a torch CSR matrix, and its diagonal."""
    rp, ci, M, L = lb.lbmg_get_matrix(plan.h, d)
    n = len(rp) - 1
    rp = torch.tensor(rp, dtype=torch.int64, device="cuda")
    ci = torch.tensor(ci, dtype=torch.int64, device="cuda")
    v = torch.tensor(M, device="cuda") + case["t"] * torch.tensor(L, device="cuda")
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    dg = torch.zeros(n, dtype=F64, device="cuda")
    on = row == ci
    dg[row[on]] = v[on]
    return rp, ci, v, n, dg


def _mat(rp, ci, v, r0, r1, n):
    k0, k1 = int(rp[r0]), int(rp[r1])
    return torch.sparse_csr_tensor(rp[r0:r1 + 1] - k0, ci[k0:k1], v[k0:k1], size=(r1 - r0, n))


class _Level:
    def __init__(self, plan, case, d, transfer=True):
        rp, ci, v, n, dg = _csr(plan, case, d)
        self.n, self.dg = n, dg
        self.A = _mat(rp, ci, v, 0, n, n)
        # functions that meet the surface in slivers only are not relaxed
        keep = (dg > 0) & (dg >= 1e-20 * dg.mean())
        self.dinv = torch.where(keep, 1 / torch.where(keep, dg, torch.ones_like(dg)), torch.zeros_like(dg))[:, None]
        corner = torch.tensor(lb.lbmg_get_dofs(plan.h, d)[0], device="cuda")
        colour = (corner[:, 0] & 1) | ((corner[:, 1] & 1) << 1) | ((corner[:, 2] & 1) << 2)
        at = torch.searchsorted(colour, torch.arange(9, device="cuda", dtype=colour.dtype)).tolist()   # rows come by colour
        self.colours = [(at[c], at[c + 1], _mat(rp, ci, v, at[c], at[c + 1], n)) for c in range(8) if at[c + 1] > at[c]]
        self.P = self.PT = None
        if transfer and d > plan.d0:
            par, w = lb.lbmg_get_prolongation(plan.h, d)
            i, k = np.nonzero(par >= 0)
            nc = plan.sizes[d - 1][0]
            ij = torch.tensor(np.stack([i, par[i, k]]).astype(np.int64), device="cuda")
            P = torch.sparse_coo_tensor(ij, torch.tensor(w[i, k], device="cuda"), (n, nc)).coalesce()
            self.P, self.PT = P.to_sparse_csr(), P.t().coalesce().to_sparse_csr()

    def sweep(self, b, x, forward=True):
        for r0, r1, A in self.colours if forward else reversed(self.colours):
            x[r0:r1] += self.dinv[r0:r1] * (b[r0:r1] - A @ x)


def _vcycle(levels, d, d0, b):
    L = levels[d]
    if d == d0:
        A = L.A.to_dense()
        return torch.linalg.solve(A + 1e-12 * L.dg.mean() * torch.eye(L.n, dtype=F64, device="cuda"), b)
    x = torch.zeros_like(b)
    for _ in range(2):
        L.sweep(b, x)
    x += L.P @ _vcycle(levels, d - 1, d0, L.PT @ (b - L.A @ x))
    for _ in range(2):
        L.sweep(b, x, False)
    return x


def exact(case, seed):
    """`run`'s result in 64 bits from the plan's matrices and transfer weights.  None for solves: at their
    tolerance the coefficients of nearly dependent functions are undetermined (only the sum of the functions
    is), and projected and evaluated values need the functions themselves."""
    kind = case["kind"]
    if kind in ("step", "flow", "batch"):
        return None
    s = prepare(case, seed)
    p = s["plan"]
    if kind == "smooth":
        L = _Level(p, case, p.D, transfer=False)
        x = s["x0"].clone()
        for _ in range(case["sweeps"]):
            L.sweep(s["rhs"], x)
        return x
    if kind == "transfer":
        L = _Level(p, case, p.D)
        r = s["rhs"] - L.A @ s["x0"]
        rc = L.PT @ r
        return [r, rc, s["x0"] + L.P @ rc]
    levels = {d: _Level(p, case, d) for d in range(p.d0, p.D + 1)}
    x = torch.zeros_like(s["rhs"])
    for _ in range(case["cycles"]):
        x += _vcycle(levels, p.D, p.d0, s["rhs"] - levels[p.D].A @ x)
    return x
