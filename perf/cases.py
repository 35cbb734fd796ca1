"""The work a user of the solver has it do, as cases that can be timed.

Every case goes through the package's public entry points (`Solver`, `Batch`)
on meshes of its own generator: cloth grids and jittered or regular hex
blocks split into five tetrahedra per cell, with the compliances, pins and
parameters of the named workloads and of the serving trace.

Kinds of cases:

  frame      one frame of Alg. 1 on a resident instance: state in, `max_iter`
             global iterations (evaluate, assemble, re-form the hierarchy,
             factor the coarsest level, MGPCG, update), state out
  vcycle     the preconditioner alone: one V-cycle z = V(r)
  apply      the level-0 operator alone: y = A x, matrix-free or assembled
  reform     C, grad C, the values of A, the Galerkin products of every level
             and the coarsest factorisation at a new state
  setup      the lazy AMG setup at a new state (near-kernel, strength,
             aggregation, prolongators, Galerkin patterns and values)
  serve      a session of the service: instances admitted, created, set up and
             stepped side by side, their states read back

Solves run to the workloads' relative residual of 1e-6; where that would take
seconds (`cap` below a thousand) they stop at `cap` PCG iterations, the time
budget of an interactive user.  A frame's state is returned as the vertex
buffers that a renderer takes, and the FP32 V-cycle's z in the precision it
has: both 32 bits.  Everything else is returned as it is.
"""
import math

import numpy as np
import torch

from paper_2505_13390_gb300.meshgen import cloth, default_params, hex_block
from paper_2505_13390_gb300.mgpbd import Batch, Solver

MIXED = {"precision": 1, "level0_op": 1, "use_graphs": 1}
FP64 = {"precision": 0, "level0_op": 0, "use_graphs": 0}


def listed():
    return [
        # the 32 x 32 cloth in FP64 with the library's default path (assembled
        # matrix, plain launches), two levels, part of a frame: the smallest
        # whole call, all latency
        dict(name="frame-cloth32-fp64", kind="frame", mesh="cloth", n=32, log_alpha=-8.0, max_levels=2, max_iter=5,
             cap=20000, **FP64),
        # a cloth of the serving trace in the served form (mixed precision,
        # matrix-free level 0, captured graphs); odd size
        dict(name="frame-cloth129", kind="frame", mesh="cloth", n=129, log_alpha=-7.0, max_iter=4, cap=20000, **MIXED),
        # a beam of the serving trace in the served form
        dict(name="frame-beam26", kind="frame", mesh="beam", n=26, log_alpha=-8.0, max_iter=2, cap=20000, **MIXED),
        # the beam of 40 x 10 x 10 cells with one ARAP row per tetrahedron
        dict(name="frame-beam40-arap", kind="frame", mesh="arap", n=40, log_alpha=0.0, max_iter=3, cap=200, **MIXED),
        # the 512 x 512 cloth with bend edges and per-row compliance
        dict(name="frame-cloth512-bend", kind="frame", mesh="bend", n=512, log_alpha=-6.0, max_iter=1, cap=400, **MIXED),
        # a large cloth with the smoother meant for cloth, Chebyshev
        dict(name="frame-cloth256-chebyshev", kind="frame", mesh="cloth", n=256, log_alpha=-8.0, max_iter=1, cap=400,
             smoother=2, **MIXED),
        # the 1.65M-tet block: one global iteration between two lazy setups
        dict(name="frame-block100", kind="frame", mesh="block", n=100, ny=33, nz=100, log_alpha=-10.0, max_iter=1,
             cap=300, **MIXED),
        # the preconditioner in mixed precision on a mid-sized block
        dict(name="vcycle-block40", kind="vcycle", mesh="block", n=40, ny=33, nz=40, log_alpha=-10.0, **MIXED),
        # the recurrence's FP64 product on the 1.65M-tet block
        dict(name="apply-block100", kind="apply", mesh="block", n=100, ny=33, nz=100, log_alpha=-10.0, form=1, **MIXED),
        # what each global iteration does before its solve, on a mid-sized block
        dict(name="reform-block40", kind="reform", mesh="block", n=40, ny=33, nz=40, log_alpha=-10.0, **MIXED),
        # the lazy setup of the beam workload
        dict(name="setup-beam40", kind="setup", mesh="beam", n=40, log_alpha=-9.0, **MIXED),
        # a serving session: uneven instances side by side on their own streams
        dict(name="serve-6", kind="serve", n=6, log_alpha=-6.5, max_iter=1, cap=20000, **MIXED),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def alpha(lo, hi):
        return round(rng.uniform(lo, hi), 2)

    kind = rng.choice(["frame", "frame", "frame", "vcycle", "vcycle", "apply", "reform", "setup", "serve"])
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(2, 6), log_alpha=alpha(-7.0, -6.0), max_iter=1, cap=20000, **MIXED)
    mesh = rng.choice(["cloth", "cloth", "beam", "beam", "block", "bend"] + (["arap"] if kind == "frame" else []))
    frame = kind == "frame"
    c = dict(kind=kind, mesh=mesh)
    if mesh == "cloth":
        c.update(n=log_int(16, 256), log_alpha=alpha(-8.0 if frame else -9.0, -6.0))
    elif mesh == "bend":
        c.update(n=log_int(200 if frame else 32, 512), log_alpha=-6.0)
    elif mesh == "beam":
        c.update(n=log_int(10, 40 if frame else 80), log_alpha=alpha(-8.0 if frame else -9.0, -6.0))
    elif mesh == "arap":
        c.update(n=log_int(10, 60), log_alpha=0.0)
    else:
        most = 12 if frame else 60
        c.update(n=log_int(5, most), ny=rng.randint(5, most // 2), nz=log_int(5, most), log_alpha=alpha(-8.0 if frame else -10.0, -7.0))
    c.update(MIXED if rng.random() < 0.75 or mesh in ("bend", "arap") else dict(FP64, level0_op=rng.randint(0, 1), use_graphs=1))
    if frame:
        c.update(max_iter=1, cap=400 if mesh == "bend" else 200 if mesh == "arap" else 20000)
        if mesh == "cloth" and rng.random() < 0.3:
            c.update(smoother=2)
    if kind == "apply":
        c.update(form=c["level0_op"])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _mesh(case, seed):
    """The case's mesh: rest shape, compliance and start from the seed."""
    kind, n, alpha = case["mesh"], case["n"], 10.0 ** case["log_alpha"]
    if kind == "cloth":
        m = cloth(n, plane="xz", alpha=alpha, pin="corners", noise=1e-4, seed=seed)
    elif kind == "bend":  # per-row compliance over the four decades below log_alpha
        m = cloth(n, plane="xy", bend=True, alpha_log_range=(case["log_alpha"] - 4.0, case["log_alpha"]), pin="top",
                  noise=1e-4, seed=seed)
    elif kind == "beam":
        m = hex_block(n, 10, 10, h=0.01, alpha=alpha, pin="x0", seed=seed)
    elif kind == "arap":
        m = hex_block(n, 10, 10, h=0.01, arap_mu=1e7, pin="x0", seed=seed)
    else:
        m = hex_block(n, case["ny"], case["nz"], h=0.005, jitter=0.1, alpha=alpha, pin="y0", seed=seed)
    return _moving(m, seed)


def _moving(m, seed):
    """An affine velocity field of about 0.01 m/s, drawn from the seed."""
    rng = np.random.default_rng(seed + 100)
    size = np.abs(m.rest_pos).max()
    m.v0 = rng.uniform(-0.01, 0.01, 3) + m.rest_pos @ (rng.uniform(-0.01, 0.01, (3, 3)) / size)
    m.v0[m.inv_mass == 0] = 0.0
    return m


def _params(case):
    soft = case.get("mesh") not in ("cloth", "bend")
    keep = ("precision", "level0_op", "use_graphs", "smoother", "max_levels", "max_iter")
    return default_params(omega_x=0.1 if soft else 0.25, pcg_maxiter=case.get("cap", 400), setup_interval=0,
                          **{k: case[k] for k in keep if k in case})


def _sessions(case, seed):
    """Instances of a serving session: cloths and beams of uneven sizes (the
    sizes are the case's, the states the seed's)."""
    rng = np.random.default_rng(1000 * case["n"])
    out = []
    for k in range(case["n"]):
        alpha = 10.0 ** (case["log_alpha"] + rng.uniform(-0.5, 0.5))
        if k % 2 == 0:
            m = cloth(int(rng.integers(16, 161)), plane="xz", alpha=alpha, pin="corners", seed=seed + k)
            p = dict(_params(case), omega_x=0.25)
        else:
            m = hex_block(int(rng.integers(10, 41)), 10, 10, h=0.01, alpha=alpha, pin="x0", seed=seed + k)
            p = dict(_params(case), omega_x=0.1)
        out.append((_moving(m, seed + k), p))
    return out


def _vector(m, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(m, dtype=torch.float64, device="cuda", generator=g)


def prepare(case, seed):
    if case["kind"] == "serve":
        return {"case": case, "instances": _sessions(case, seed)}
    mesh = _mesh(case, seed)
    stream = torch.cuda.Stream()
    g = Solver(mesh, _params(case), stream=stream)
    s = {"case": case, "g": g, "stream": stream}
    s["x"], s["v"] = (torch.from_numpy(a).cuda() for a in (mesh.x0, mesh.v0))
    if case["kind"] in ("frame", "reform"):  # the resident instance has its hierarchy
        g.begin_frame()
    g.eval_assemble()
    g.prepare_solve()
    if case["kind"] in ("vcycle", "apply"):
        s["r"] = _vector(mesh.n_rows, seed)
    if case["kind"] in ("reform", "setup"):  # a later state of the same instance
        s["x"] += 1e-3 * s["v"]
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    if case["kind"] == "serve":
        return _serve(s)
    g, mixed = s["g"], case["precision"] == 1
    with torch.cuda.stream(s["stream"]):
        if case["kind"] == "frame":
            g.set_state(s["x"], s["v"])
            g.step(1)
            x, v = torch.empty_like(s["x"]), torch.empty_like(s["v"])
            g.get_state_device(x, v)
            return {"x": x.float(), "v": v.float()}
        if case["kind"] == "vcycle":
            z = g.vcycle(s["r"])
            return z.float() if mixed else z
        if case["kind"] == "apply":
            return g.apply(s["r"], case["form"])
        g.set_state(s["x"], s["v"])
        g.eval_assemble()
        if case["kind"] == "reform":
            g.prepare_solve()
            return [g.matrix(0, device=True)[2], _coarse(g)]
        g.setup()
        agg, _, P, _ = g.level_agg(0)[1:]
        return [_coarse(g), agg, P]


def _coarse(g):
    """The coarse matrices' values, one after the other in a buffer of a
    quarter of A's size (their number of entries depends on the state)."""
    out, at = torch.zeros(g.level_info(0)["nnz"] // 4, dtype=torch.float64, device="cuda"), 0
    for level in range(1, g.levels):
        val = g.matrix(level, device=True)[2]
        out[at:at + len(val)] = val
        at += len(val)
    return out


def _serve(s):
    b = Batch(64 << 30, 4)
    ids = [b.add(m, p) for m, p in s["instances"]]
    status, results = b.run([(k, i, 1, 0.0) for k, i in enumerate(ids)])
    if status < 0:
        raise RuntimeError(b.error())
    out = [b.state(i)[0].astype(np.float32) for i in ids]
    b.close()
    return out


# ---------------------------------------------------------------------------
# the least that a pass moves and computes
# ---------------------------------------------------------------------------
def _sizes(case):
    """(vertices, distance rows, tetrahedra, nonzeros of A)."""
    n = case["n"]
    if case["mesh"] in ("cloth", "bend"):
        e = 2 * n * (n - 1) + (n - 1) ** 2 + (2 * n * (n - 2) if case["mesh"] == "bend" else 0)
        return n * n, e, 0, e * (19 if case["mesh"] == "bend" else 11)
    a, b, c = (n, case["ny"], case["nz"]) if case["mesh"] == "block" else (n, 10, 10)
    cells, verts = a * b * c, (a + 1) * (b + 1) * (c + 1)
    if case["mesh"] == "arap":
        return verts, 0, 5 * cells, 5 * cells * 70
    # axis edges and one diagonal per face of every cell
    e = (a * (b + 1) * (c + 1) + b * (a + 1) * (c + 1) + c * (a + 1) * (b + 1)
         + a * b * (c + 1) + b * c * (a + 1) + a * c * (b + 1))
    return verts, e, 5 * cells, (e + 5 * cells) * 95


def _iterations(case):
    """PCG iterations of one solve, about (cond(A) grows as alpha falls)."""
    if case["cap"] < 1000:
        return case["cap"]
    if case["mesh"] == "cloth":
        return int(90 * 10 ** (0.45 * (-6.0 - case["log_alpha"])))
    return int(1000 * (case["n"] / 26) ** 0.55 * 10 ** (0.12 * (-6.0 - case["log_alpha"])))


def work(case):
    """Per product with A: the constraint gradients and vertex indices once,
    the row vectors it takes and gives; two multiply-adds per gradient value."""
    if case["kind"] == "serve":
        each = [dict(case, kind="frame", mesh=m, n=n) for k in range(case["n"]) for m, n in ((("cloth", 88), ("beam", 25))[k % 2],)]
        parts = [work(c) for c in each]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    verts, e, t, nnz = _sizes(case)
    m = e + t
    grads, index = 3 * e + 12 * t, 4 * (2 * e + 4 * t)
    flops = 4 * (6 * e + 12 * t) + 4 * m
    wide = 8 * grads + index + 8 * 3 * m
    low = (4 if case["precision"] == 1 else 8)
    # two sweeps before and after the coarse correction, the first of them
    # from zero, and the residual: four products
    cycle = 4 * (low * grads + index) + 4 * 5 * low * m + 8 * 2 * m
    if case["kind"] == "apply":
        return {"bytes": wide, "flops": flops}
    if case["kind"] == "vcycle":
        return {"bytes": cycle, "flops": 4 * flops}
    # new values of A and one pass over them for the coarse operator
    values = 24 * 2 * verts + index + 8 * grads + nnz * (8 + 4 + 2) + 12 * nnz
    if case["kind"] == "reform":
        return {"bytes": values, "flops": 12 * nnz}
    if case["kind"] == "setup":  # near-kernel sweeps and power method as well
        return {"bytes": values + (3 + 15) * 12 * nnz, "flops": 12 * nnz + 18 * 2 * nnz}
    per_iteration = wide + cycle + 8 * 9 * m
    its = case["max_iter"] * _iterations(case)
    return {"bytes": case["max_iter"] * values + its * per_iteration,
            "flops": case["max_iter"] * 12 * nnz + its * 5 * flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, plainly
# ---------------------------------------------------------------------------
class _Plain:
    """Distance and volume rows at given positions, in float64."""

    def __init__(self, m, dt):
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.m, self.dist, self.tet, self.w = m, to(m.dist).long(), to(m.tet).long(), to(m.inv_mass)
        self.at = to(m.alpha) / dt ** 2
        self.rest = self.values(to(m.rest_pos))

    def values(self, x):
        d = x[self.dist[:, 0]] - x[self.dist[:, 1]]
        e = x[self.tet[:, 1:]] - x[self.tet[:, :1]]
        return torch.cat([d.norm(dim=1), (e[:, 0] * torch.linalg.cross(e[:, 1], e[:, 2])).sum(1) / 6])

    def gradients(self, x):
        d = x[self.dist[:, 0]] - x[self.dist[:, 1]]
        n = d / d.norm(dim=1, keepdim=True)
        e = x[self.tet[:, 1:]] - x[self.tet[:, :1]]
        g = torch.stack([torch.linalg.cross(e[:, (k + 1) % 3], e[:, (k + 2) % 3]) / 6 for k in range(3)], 1)
        return torch.stack([n, -n], 1), torch.cat([-g.sum(1, keepdim=True), g], 1)

    def jt(self, grads, y):
        e = len(self.dist)
        u = torch.zeros(self.m.n_verts, 3, dtype=torch.float64, device="cuda")
        u.index_add_(0, self.dist.reshape(-1), (grads[0] * y[:e, None, None]).reshape(-1, 3))
        u.index_add_(0, self.tet.reshape(-1), (grads[1] * y[e:, None, None]).reshape(-1, 3))
        return u * self.w[:, None]

    def apply(self, grads, y):
        u = self.jt(grads, y)
        rows = torch.cat([(grads[0] * u[self.dist]).sum((1, 2)), (grads[1] * u[self.tet]).sum((1, 2))])
        return rows + self.at * y

    def dense(self, grads):
        e, rows, n3 = len(self.dist), self.m.n_rows, 3 * self.m.n_verts
        j = torch.zeros(rows, n3, dtype=torch.float64, device="cuda")
        k = torch.arange(3, device="cuda")
        for verts, g, first in ((self.dist, grads[0], 0), (self.tet, grads[1], e)):
            for s in range(verts.shape[1]):
                j[first + torch.arange(len(verts), device="cuda")[:, None], 3 * verts[:, s, None] + k] = g[:, s]
        return (j * self.w.repeat_interleave(3)) @ j.T + torch.diag(self.at)


def _exact_frame(case, seed):
    """Alg. 1 with a direct solve of each system."""
    m, p = _mesh(case, seed), _params(case)
    a = _Plain(m, p["dt"])
    x0, v = torch.from_numpy(m.x0).cuda(), torch.from_numpy(m.v0).cuda()
    free = (a.w > 0)[:, None].double()
    v = (v + p["dt"] * torch.tensor(p["gravity"], dtype=torch.float64, device="cuda")) * free
    x, lam = x0 + p["dt"] * v, torch.zeros(m.n_rows, dtype=torch.float64, device="cuda")
    for _ in range(case["max_iter"]):
        grads = a.gradients(x)
        b = a.rest - a.values(x) - a.at * lam
        dl = torch.linalg.solve(a.dense(grads), b)
        lam, x = lam + dl, x + p["omega_x"] * a.jt(grads, dl)
    return {"x": x, "v": (x - x0) / p["dt"]}


def _exact_vcycle(case, seed):
    """The V-cycle in float64 on the instance's hierarchy (matrices,
    aggregates, prolongators and weights are its data)."""
    s = prepare(case, seed)
    g, levels = s["g"], s["g"].levels
    mats = []
    for level in range(levels):
        ptr, col, val = g.matrix(level, device=True)
        n = len(ptr) - 1
        mats.append((torch.sparse_csr_tensor(ptr, col.long(), val, (n, n)), val[ptr[1:] - 1]))

    def cycle(level, b):
        a, diag = mats[level]
        if level == levels - 1:
            return torch.linalg.solve(a.to_dense(), b)
        _, agg, _, weight, _ = g.level_agg(level)
        agg, weight = torch.from_numpy(agg).long().cuda(), torch.from_numpy(weight).cuda()
        omega = g.level_omega(level)[1]
        x = torch.zeros_like(b)
        for _ in range(2):
            x = x + omega * (b - a @ x) / diag
        r = weight * (b - a @ x)
        bc = torch.zeros(len(mats[level + 1][1]), dtype=torch.float64, device="cuda")
        bc.index_add_(0, agg.clamp(min=0), torch.where(agg >= 0, r, torch.zeros_like(r)))
        x = x + torch.where(agg >= 0, weight * cycle(level + 1, bc)[agg.clamp(min=0)], torch.zeros_like(b))
        for _ in range(2):
            x = x + omega * (b - a @ x) / diag
        return x

    return cycle(0, s["r"])


def _exact_values(case, seed):
    """The values of A in the library's order (ascending, diagonal last)."""
    m, p = _mesh(case, seed), _params(case)
    a = _Plain(m, p["dt"])
    x = torch.from_numpy(m.x0 + 1e-3 * m.v0).cuda()
    grads, rows, e = a.gradients(x), m.n_rows, len(a.dist)
    vert = torch.cat([a.dist.reshape(-1), a.tet.reshape(-1)])
    row = torch.cat([torch.arange(e, device="cuda").repeat_interleave(2),
                     e + torch.arange(rows - e, device="cuda").repeat_interleave(4)])
    grad = torch.cat([grads[0].reshape(-1, 3), grads[1].reshape(-1, 3)])
    order = torch.argsort(vert, stable=True)
    vert, row, grad = vert[order], row[order], grad[order]
    count = torch.bincount(vert, minlength=m.n_verts)
    first = torch.cumsum(count, 0) - count
    # every pair of rows at a vertex
    left = torch.arange(len(vert), device="cuda").repeat_interleave(count[vert])
    start = torch.cumsum(count[vert], 0) - count[vert]
    right = first[vert[left]] + torch.arange(len(left), device="cuda") - start[left]
    i, j = row[left], row[right]
    key = i * (rows + 1) + torch.where(i == j, torch.full_like(j, rows), j)
    key, at = torch.unique(key, return_inverse=True)
    val = torch.zeros(len(key), dtype=torch.float64, device="cuda")
    val.index_add_(0, at, a.w[vert[left]] * (grad[left] * grad[right]).sum(1))
    diag = key % (rows + 1) == rows
    val[diag] += a.at[key[diag] // (rows + 1)]
    return [val, None]


def exact(case, seed):
    if case["kind"] == "frame" and case["mesh"] == "cloth" and case["n"] <= 37 and case["cap"] >= 1000:
        return _exact_frame(case, seed)
    if case["kind"] == "vcycle":
        return _exact_vcycle(case, seed)
    if case["kind"] == "apply":
        m, p = _mesh(case, seed), _params(case)
        a = _Plain(m, p["dt"])
        return a.apply(a.gradients(torch.from_numpy(m.x0).cuda()), _vector(m.n_rows, seed))
    if case["kind"] == "reform" and case["mesh"] != "arap":
        return _exact_values(case, seed)
    return None
