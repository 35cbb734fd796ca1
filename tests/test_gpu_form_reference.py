"""The kernel forms a solve picks by size, against plain FP64 references.

The products and V-cycles on both sides of every size rule are compared with
the same formulas in torch, in FP64, from the instance's matrices, aggregates,
prolongators and weights (which the setup tests pin to the oracle bit for bit).
The meshes are soft (alpha 1e-4), so that the V-cycle is well conditioned: its
FP64 sums in another order stay within 1e-9 of each other and its FP32 bulk
within 1e-4, as for the V-cycle tests against the oracle.  A product's row is a
sum of at most a few hundred terms: 1e-13 of the sum of their magnitudes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2505_13390_gb300.meshgen import Mesh, cloth, default_params, hex_block  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def cut_cloth(rows):
    """A soft cloth with exactly `rows` distance rows."""
    m = cloth(int((rows / 3) ** 0.5) + 3, alpha=1e-4, noise=1e-3, seed=3)
    return Mesh("cut", m.rest_pos, m.inv_mass, m.dist[:rows], m.tet, m.alpha[:rows], m.x0, m.v0)


def cut_block(rows, ny, nz):
    """A soft block, pinned at one end, with exactly `rows` rows: all of its
    edges and as many of its tets."""
    n = 1
    while len((m := hex_block(n, ny, nz, h=0.01, jitter=0.1, alpha=1e-4, pin="x0", seed=2)).alpha) < rows:
        n = max(n + 1, int(n * rows / len(m.alpha)))
    tets = rows - len(m.dist)
    assert 0 < tets
    return Mesh("cut", m.rest_pos, m.inv_mass, m.dist, m.tet[:tets], m.alpha[:rows], m.x0, m.v0)


def ready(mesh, **over):
    from paper_2505_13390_gb300.mgpbd import Solver
    g = Solver(mesh, default_params(**over))
    g.begin_frame()
    g.eval_assemble()
    g.prepare_solve()
    torch.cuda.synchronize()
    return g


def matrices(g):
    out = []
    for level in range(g.levels):
        ptr, col, val = g.matrix(level, device=True)
        n = len(ptr) - 1
        out.append((torch.sparse_csr_tensor(ptr, col.long(), val, (n, n)), val[ptr[1:] - 1]))
    return out


def vcycle(g, mats, level, b):
    a, diag = mats[level]
    if level == len(mats) - 1:
        return torch.linalg.solve(a.to_dense(), b)
    _, agg, _, weight, _ = g.level_agg(level)
    agg, weight = torch.from_numpy(agg).long().cuda(), torch.from_numpy(weight).cuda()
    omega, take, keep = g.level_omega(level)[1], agg.clamp(min=0), agg >= 0
    x = torch.zeros_like(b)
    for _ in range(2):
        x = x + omega * (b - a @ x) / diag
    r = torch.where(keep, weight * (b - a @ x), 0.0)
    bc = torch.zeros(len(mats[level + 1][1]), dtype=torch.float64, device="cuda")
    bc.index_add_(0, take, r)
    x = x + torch.where(keep, weight * vcycle(g, mats, level + 1, bc)[take], 0.0)
    for _ in range(2):
        x = x + omega * (b - a @ x) / diag
    return x


def rel(a, b):
    return float((a - b).norm() / b.norm())


def check_forms(mesh, op, prec):
    with torch.cuda.stream(torch.cuda.Stream()):  # graphs need a stream of their own
        _check_forms(mesh, op, prec)


def _check_forms(mesh, op, prec):
    g = ready(mesh, level0_op=op, precision=prec, pcg_rtol=1e-14, pcg_maxiter=9)
    mats = matrices(g)
    gen = torch.Generator(device="cuda").manual_seed(4)
    r = torch.randn(g.m, dtype=torch.float64, device="cuda", generator=gen)
    a = mats[0][0]
    size = torch.sparse_csr_tensor(a.crow_indices(), a.col_indices(), a.values().abs(), a.shape) @ r.abs()
    if op:  # the matrix-free terms: at most |A| with its diagonal's magnitudes
        size = size + mats[0][1] * r.abs()
    y = g.apply(r, op)
    assert float(((y - a @ r).abs() / size).max()) <= 1e-13
    assert rel(g.vcycle(r), vcycle(g, mats, 0, r)) <= (1e-4 if prec else 1e-9)
    # nine iterations, one chunk of eight replayed from a graph, bit for bit
    # the plain launches
    x, info = g.solve(r)
    assert info["pcg_iters"] == 9 or g.levels == 1  # (a direct solve ends sooner)
    g.close()
    g = ready(mesh, level0_op=op, precision=prec, pcg_rtol=1e-14, pcg_maxiter=9, use_graphs=1)
    x2, info2 = g.solve(r)
    assert torch.equal(x, x2) and info2 == info
    g.close()


# entries: 2^18 and 3 * 2^18 (fused prolongation), 2^22 and 3 * 2^22 (early
# form); rows of 11 entries (cloth) and of about 90 (beam)
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("make", [
    *(lambda n=n: cut_cloth(n) for n in (23500, 24100, 71000, 72000, 379000, 383000, 1135000, 1150000)),
    *(lambda n=n: cut_block(n, 10, 10) for n in (3000, 30000, 48000, 141000))],
    ids=["c23500", "c24100", "c71000", "c72000", "c379000", "c383000", "c1135000", "c1150000",
         "b3000", "b30000", "b48000", "b141000"])
def test_csr_forms(make, prec):
    check_forms(make(), 0, prec)


# rows: 2^17 (FP64 early form), 524,288 (its FP32 passes with a dot product) and
# 2^20 (FP32); distance rows alone, and with tets, whose row pass gathers four
# vertices and whose lists are long enough for eight FP64 lanes up to 2^17 rows
@pytest.mark.parametrize("make,prec", [
    *((lambda n=n: cut_cloth(n), p) for p, ns in ((0, (129, 131072, 131073)),
                                                  (1, (129, 524288, 524289, 1048576, 1048577)))
      for n in ns),
    *((lambda n=n: cut_block(n, 33, 33), p) for p, ns in ((0, (131072, 131073)),
                                                          (1, (524288, 524289)))
      for n in ns),
    (lambda: cut_block(3000, 10, 10), 0), (lambda: cut_block(3000, 10, 10), 1)],
    ids=["c129-0", "c131072-0", "c131073-0", "c129-1", "c524288-1", "c524289-1", "c1048576-1",
         "c1048577-1", "b131072-0", "b131073-0", "b524288-1", "b524289-1", "b3000-0", "b3000-1"])
def test_matrix_free_forms(make, prec):
    check_forms(make(), 1, prec)


# the places of the test on r.r: a large level 0's first pass in each form
# (matrix-free and CSR, Jacobi with one and two sweeps, Chebyshev), the x/r update
# (Gauss-Seidel on a large matrix) and the p update (small instances)
@pytest.mark.parametrize("rows,over", [
    (1100000, dict(precision=1, level0_op=1)), (200000, dict(precision=0, level0_op=1)),
    (1100000, dict(precision=1, level0_op=1, smoother=2)), (390000, dict(precision=0)),
    (1200000, dict(precision=1)), (390000, dict(precision=0, smooth_sweeps=1)),
    (390000, dict(precision=0, smoother=2)), (390000, dict(precision=0, smoother=1)),
    (9000, dict(precision=1, level0_op=1)), (9000, dict(precision=0, smoother=1))])
@pytest.mark.parametrize("graphs", [0, 1])
def test_solve_ends_where_it_should(rows, over, graphs):
    """A solve to a tolerance ends in the first iteration at or below it, with
    the solution and residual of a solve capped there; one iteration less is
    above the tolerance and says so."""
    mesh = cut_cloth(rows)
    got = {}
    with torch.cuda.stream(torch.cuda.Stream()):
        gen = torch.Generator(device="cuda").manual_seed(5)
        b = torch.randn(rows, dtype=torch.float64, device="cuda", generator=gen)
        k = None
        for case in ("tolerance", "before", "at"):
            tol = 1e-2 if case != "at" else 1e-300
            cap = {"tolerance": 5000, "before": (k or 1) - 1, "at": k}[case]
            if cap == 0:
                continue
            g = ready(mesh, pcg_rtol=tol, pcg_maxiter=cap, use_graphs=graphs, **over)
            x, info = g.solve(b)
            got[case] = x, info
            k = k or info["pcg_iters"]
            g.close()
    x, info = got["tolerance"]
    assert info["status"] == 0 and info["pcg_iters"] == k and info["rel_res"] <= 1e-2
    x2, info2 = got["at"]
    assert torch.equal(x, x2) and info2["pcg_iters"] == k and info2["status"] == 1
    assert info2["rel_res"] == info["rel_res"]
    if k > 1:
        _, info3 = got["before"]
        assert info3["status"] == 1 and info3["pcg_iters"] == k - 1 and info3["rel_res"] > 1e-2


def test_last_iteration_leaves_the_vcycle_out():
    """One FP64 iteration on an assembled block of 0.6M rows: a V-cycle, a
    product and the vector updates, not a second V-cycle (which would be 0.5
    V-cycles above the line, and its absence is as far below it)."""
    import time
    mesh = hex_block(40, 33, 40, h=0.005, jitter=0.1, alpha=1e-10, pin="y0", seed=1)

    def best(f):
        ts = []
        for _ in range(15):
            torch.cuda.synchronize()
            t = time.perf_counter()
            f()
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t)
        return min(ts)

    g = ready(mesh, precision=0, pcg_maxiter=1, pcg_rtol=1e-300)
    r = torch.randn(g.m, dtype=torch.float64, device="cuda")
    cycle, product, solve = best(lambda: g.vcycle(r)), best(lambda: g.apply(r)), best(lambda: g.solve(r))
    g.close()
    assert solve <= 1.5 * cycle + 2 * product, (solve, cycle, product)


@pytest.mark.parametrize("rows,per_cycle", [(9000, 1), (80000, 2)])
def test_profile_times_plain_sweeps_only(rows, per_cycle):
    """The sweep channel's bytes per launch are those of a plain CSR sweep, so
    the sweep that takes the prolongation along (up to 786,432 entries) and the
    one that writes z are not timed: of the three sweeps behind the one from
    zero, one and two are."""
    g = ready(cut_cloth(rows), precision=1, pcg_rtol=1e-300, pcg_maxiter=10)
    b = torch.ones(rows, dtype=torch.float64, device="cuda")
    g.profile(True)
    _, info = g.solve(b)
    assert info["pcg_iters"] == 10
    # the cycles before each iteration's end but the last one's
    assert g.profile_read()["launches"] == 10 * per_cycle
    g.close()


def test_autotuner_times_sixteen_fp64_lanes():
    """On a beam of 6,125 rows the FP64 vertex pass is fastest with sixteen
    lanes per vertex (its lists hold about thirty rows), and so are whole
    solves: the autotuner has to try them."""
    mesh = hex_block(5, 10, 10, h=0.01, alpha=1e-8, pin="x0", seed=1)
    g = ready(mesh, precision=0, level0_op=1, autotune=1)
    assert g.lanes(0)["vert64"] == 16
    g.close()
