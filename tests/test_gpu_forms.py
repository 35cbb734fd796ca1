"""The edges of the kernel forms that a solve picks by size.

* The matrix-free passes have an early form up to 2^20 rows, and 524,288 rows
  (4096 partials) where they end in a dot product; the CSR level-0 sweep takes
  the prolongation with it up to 65,536 rows.  Three PCG iterations are compared
  with the same three iterations put together from the solver's own A.p and
  V-cycle: a dropped partial or an unwritten row changes alpha or beta.  In FP64
  the dot products of up to 2^20 terms differ by their summation order only (a
  tree of depth 20 and block chains of at most a few hundred terms: below 1e-12
  relative), which three iterations do not raise past 1e-9; in mixed precision a
  residual that differs in its last bit can round to another FP32 value, so z
  differs as two FP32 V-cycles do (1e-4, as for the V-cycle against FP64).
* The setup and assembly kernels that work on several rows per warp or block
  have to give the oracle's bits on ragged row counts.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle  # noqa: E402
from paper_2505_13390_gb300.meshgen import Mesh, cloth, default_params, hex_block  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def solver(mesh, params):
    from paper_2505_13390_gb300.mgpbd import Solver
    return Solver(mesh, params)


def cut_cloth(rows):
    """A soft cloth with exactly `rows` distance rows."""
    n = 3
    while len((m := cloth(n, alpha=1e-4, noise=1e-3, seed=3)).dist) < rows:
        n = n + 1 if n < 12 else int(n * 1.1)
    return Mesh("cut", m.rest_pos, m.inv_mass, m.dist[:rows], m.tet, m.alpha[:rows], m.x0, m.v0)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("op,rows", [
    (1, 129), (1, 131073), (1, 524288), (1, 524289), (1, 1048576), (1, 1048577),
    (0, 129), (0, 65536), (0, 65537)])
def test_three_iterations_at_form_edges(op, rows, prec):
    mesh = cut_cloth(rows)
    g = solver(mesh, default_params(level0_op=op, precision=prec, pcg_maxiter=3, pcg_rtol=1e-14))
    g.begin_frame()
    g.eval_assemble()
    g.prepare_solve()
    b = torch.tensor(np.random.default_rng(4).standard_normal(rows), device="cuda")
    got, info = g.solve(b)
    x, r = torch.zeros_like(b), b.clone()
    p = z = g.vcycle(r)
    rz = r @ z
    for _ in range(info["pcg_iters"]):  # (a one-level hierarchy converges earlier)
        q = g.apply(p, op)
        a = rz / (p @ q)
        x, r = x + a * p, r - a * q
        z = g.vcycle(r)
        rz, old = r @ z, rz
        p = z + (rz / old) * p
    rel = float((got - x).norm() / x.norm())
    assert 1 <= info["pcg_iters"] <= 3 and rel <= (1e-4 if prec else 1e-9), rel


def test_more_vertices_than_a_grid_of_groups():
    """Forty rows on the last of 8.5 million vertices: 8 lanes per vertex in
    blocks of 64 threads would be more blocks than a launch gets."""
    nv, rows = 8_500_000, 40
    x = np.zeros((nv, 3))
    x[:, 0] = 0.01 * np.arange(nv)
    e = np.stack([np.arange(nv - rows - 1, nv - 1), np.arange(nv - rows, nv)], 1).astype(np.int32)
    mesh = Mesh("tail", x, np.ones(nv), e, np.zeros((0, 4), np.int32), np.full(rows, 1e-6),
                x.copy(), np.zeros((nv, 3)))
    r = torch.tensor(np.random.default_rng(5).standard_normal(rows), device="cuda")
    z = []
    for op in (0, 1):
        g = solver(mesh, default_params(level0_op=op, precision=1, coarse_max=10, max_levels=3,
                                        gravity=(0.0, 0.0, 0.0)))
        g.begin_frame()
        g.eval_assemble()
        g.prepare_solve()
        z.append(g.vcycle(r))
        ref = g.apply(r, 0)
        if op:  # A in FP64: at most five products per entry
            assert float((g.apply(r, 1) - ref).norm() / ref.norm()) <= 1e-13
        g.close()
    assert float((z[1] - z[0]).norm() / z[0].norm()) <= 1e-4


def block(x, y, z):
    return hex_block(x, y, z, h=0.01, jitter=0.1, alpha=1e-8, pin="x0", seed=2)


@pytest.mark.parametrize("make", [
    lambda: block(1, 1, 1), lambda: block(2, 1, 1), lambda: block(5, 3, 2), lambda: block(9, 7, 4),
    lambda: block(21, 16, 13), lambda: cloth(2, alpha=1e-6, noise=1e-3),
    lambda: cloth(17, alpha=1e-8, noise=1e-3), lambda: cloth(150, alpha=1e-8, noise=1e-3)],
    ids=["b1", "b2", "b5", "b9", "b21", "c2", "c17", "c150"])
def test_setup_bits_on_ragged_sizes(make):
    mesh = make()
    p = default_params(coarse_max=6 if mesh.n_rows < 2000 else 400)
    o, g = Oracle(mesh, p, omp=True), solver(mesh, p)
    for s in (o, g):
        s.begin_frame()
        s.eval_assemble()
        s.prepare_solve()
    assert o.levels == g.levels
    for l in range(o.levels):
        for a, b in zip(o.matrix(l), g.matrix(l)):
            assert np.array_equal(a, b), l
        if l + 1 < o.levels:
            for a, b in zip(o.level_agg(l)[1:], g.level_agg(l)[1:]):
                assert np.array_equal(a, b), l
            assert g.level_omega(l) == pytest.approx(o.level_omega(l), rel=1e-10)


@pytest.mark.parametrize("rows", [1, 3, 4, 5, 31, 4095, 4096, 4097, 65535, 65536, 65537])
def test_near_kernel_bits_at_rows_per_warp(rows):
    """4 rows per warp up to 4,096, 8 up to 65,536, then 32: the near-kernel
    vector is the oracle's, bit for bit, on every side."""
    mesh = cut_cloth(rows)
    p = default_params(coarse_max=400)
    o, g = Oracle(mesh, p, omp=True), solver(mesh, p)
    for s in (o, g):
        s.begin_frame()
        s.eval_assemble()
        s.prepare_solve()
    assert np.array_equal(o.level_agg(0)[4], g.level_agg(0)[4])
