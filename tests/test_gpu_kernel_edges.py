"""Kernels that work in tiles, at the sizes where a tile is short, exact or one
past full, against the FP64 oracle (tolerances as in test_gpu_parity)."""
import numpy as np
import pytest

import mhfp_inputs as mi
import oracle
from oracle import precond, system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _solver(prob, **opts):
    from paper_2002_09603_gb300 import default_options, prepare
    o = default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    return prepare(prob, o)


def _close(got, ref, sizes, rtol):
    o = 0
    for n in sizes:
        g, r = got[o:o + n], ref[o:o + n]
        assert np.abs(g - r).max() <= rtol * max(np.abs(r).max(), 1e-300), o
        o += n


# element kernels: 32 cells per block of the displacement kernel
@pytest.mark.parametrize("dims", [(1, 1, 1), (31, 1, 1), (8, 4, 1), (11, 3, 1), (5, 13, 1), (3, 5, 7)])
def test_element_kernels_at_tile_edges(dims):
    prob = mi.random_small(*dims, seed=7, jitter=0.2)
    B = oracle.assemble(prob)
    pc = precond.build(B, "amg")
    s = _solver(prob, autotune=0)
    x = np.random.default_rng(3).standard_normal(s.n)
    y = s.apply_operator(torch.from_numpy(x).cuda()).cpu().numpy()
    _close(y, system.system_matrix(B) @ x, B.sizes, 1e-12)
    bt, ds = s.scalings()
    assert np.allclose(bt.cpu().numpy(), pc.Bt, rtol=1e-12, atol=0)
    assert np.allclose(ds.cpu().numpy(), precond.equilibration(B, pc.Bt, pc.C), rtol=1e-12, atol=0)
    s.close()


# FP64 rows of the displacement level: 32 nodes per block (operator, sweeps,
# residual), 256 per block in the allocation-free norm; at most 300,000 nodes
# here (the form above that runs in the 128^3 test)
# (the lines are U64_SPLIT_ROWS, U64_SPLIT_NODES and NA_SPLIT_NODES, 60,000 to
# 120,000; the form between runs in test_gpu_size_rules)
@pytest.mark.parametrize("dims", [(7, 1, 1), (10, 1, 2), (1, 3, 15), (15, 3, 3), (4, 5, 9)])
def test_fp64_rows_at_tile_edges(dims):
    prob = mi.random_small(*dims, seed=11, jitter=0.2)
    B = oracle.assemble(prob)
    pc = precond.build(B, "amg", coarse_max=8)
    s = _solver(prob, autotune=0, coarse_max=8)
    rng = np.random.default_rng(4)
    x, b = rng.standard_normal(s.n), rng.standard_normal(s.n)
    xd, bd = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    A = system.system_matrix(B)
    _close(s.apply_operator(xd).cpu().numpy(), A @ x, B.sizes, 1e-12)
    nU = B.sizes[0]
    v = s.vcycle(0, bd[:nU].contiguous()).cpu().numpy()
    ref = precond.vcycle(pc.u_levels, b[:nU])
    assert np.abs(v - ref).max() <= 1e-10 * np.abs(ref).max()
    ds = precond.equilibration(B, pc.Bt, pc.C)
    r, n0 = s.residual_norm_noalloc(bd, xd).cpu().numpy()
    assert np.isclose(r, np.linalg.norm(ds * (b - A @ x)), rtol=1e-12)
    assert np.isclose(n0, np.linalg.norm(ds * b), rtol=1e-12)
    s.close()


# Gram-Schmidt: the basis columns in groups of eight and chunks of four, rows
# in blocks of 256, reductions by the last block, both numbers of passes;
# restart 1, 7, 9 and 63 (column counts 1..63) and vectors of one block up
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("dims,restart", [((1, 1, 1), 7), ((3, 2, 2), 9), ((6, 5, 4), 63), ((7, 6, 5), 1)])
def test_arnoldi_vectors_at_edges(dims, restart, reorth, precision):
    prob = mi.random_small(*dims, seed=5, jitter=0.1)
    B = oracle.assemble(prob)
    s = _solver(prob, autotune=0, restart=restart, reorth=reorth, precision=precision, coarse_max=8, cheb_degree=3,
                maxit=3000)
    x, st = s.solve(s.build_rhs(), tol=1e-10)
    ref = oracle.solve_direct(B, oracle.rhs(B))
    # energy-norm-like check at the residual tolerance (1e-8, as test_gpu_parity's solves)
    ds = s.scalings()[1].cpu().numpy()
    err = np.linalg.norm((x.cpu().numpy() - ref) / ds) / np.linalg.norm(ref / ds)
    assert st["converged"] and err < 1e-7, (st, err)
    s.close()


# (through the library's vectors; the functions alone, over every branch: test_gpu_kernel_units)
def test_conversions_match_the_instructions():
    """The integer-pipe FP32 <-> FP64 conversions (vectors that the mixed form
    rounds and widens) bit for bit, over every exponent, ties, signed zeros,
    subnormals, infinities and NaN."""
    s = _solver(mi.random_small(6, 5, 4, seed=2), autotune=0, precision=1)
    rng = np.random.default_rng(0)
    n = s.n
    v = rng.standard_normal(n) * 2.0 ** rng.integers(-160, 140, n)
    v[:8] = [0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -149, 3.4028235677973366e38, -2.0 ** -126 * (1 - 2.0 ** -25)]
    m = rng.integers(0, 1 << 23, n - 8).astype(np.float64) / (1 << 23) + 1.0  # FP32 values plus an exact half ulp
    v[8:n // 2] = (m + 2.0 ** -24)[: n // 2 - 8] * 2.0 ** rng.integers(-120, 120, n // 2 - 8)
    x = torch.from_numpy(v).cuda()
    s.apply_operator_ff(x)  # rounds x; the operator itself is tested elsewhere
    # apply_precond rounds its input the same way: equal for x and fl32(x)
    ok = torch.isfinite(x) & (x.abs() < 1e30)
    x = torch.where(ok, x, torch.zeros_like(x))
    a, b = s.apply_precond(x), s.apply_precond(x.float().double())
    assert torch.equal(a, b) and torch.equal(a, a.float().double())
    s.close()


# the float-float operator's five row families share one launch, a block row
# per family: sizes where the families need different numbers of blocks
@pytest.mark.parametrize("dims", [(1, 1, 1), (15, 15, 1), (1, 16, 16), (40, 2, 3), (2, 3, 40), (7, 6, 5)])
def test_float_float_operator_row_families(dims):
    prob = mi.random_small(*dims, seed=9, jitter=0.2)
    s = _solver(prob, autotune=0, precision=1)
    x = torch.from_numpy(np.random.default_rng(6).standard_normal(s.n).astype(np.float32).astype(np.float64)).cuda()
    y, ref = s.apply_operator_ff(x), s.apply_operator(x)
    # 2^-40 of the row's sum of |terms|, bounded by the operator on |x| with
    # the largest coefficient sum of the block (test_gpu_parity's bound, coarser)
    nU, nP, _ = s.sizes
    for a, b in ((0, nU), (nU, nU + nP), (nU + nP, s.n)):
        scale = ref[a:b].abs().max()
        assert (y[a:b] - ref[a:b]).abs().max() <= 2.0 ** -38 * scale
    s.close()


# row-major sweeps and residuals (a warp or eight lanes per point) as the
# autotuner and the size rule pick them: box levels of 1 to a few thousand
# points (a last block that is not full), 1, 3 and 6 unknowns per point
# (every schedule by itself, eight lanes among them: test_gpu_kernel_units)
@pytest.mark.parametrize("near_kernel", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dims,autotune", [((12, 10, 4), 0), ((12, 10, 4), 1), ((45, 7, 7), 0)])
def test_row_major_levels_against_the_oracle(dims, autotune, precision, near_kernel):
    prob = mi.random_small(*dims, seed=13, jitter=0.15)
    B = oracle.assemble(prob)
    from oracle import rbm
    pc = precond.build(B, "amg_rbm" if near_kernel else "amg", coarse_max=4)
    s = _solver(prob, autotune=autotune, coarse_max=4, precision=precision, near_kernel=near_kernel)
    if not autotune:
        assert 32 in s.hierarchy(0)["schedule"] and 32 in s.hierarchy(1)["schedule"]
    rng = np.random.default_rng(8)
    nU, _, nPi = B.sizes
    tol = 1e-5 if precision else 1e-10
    for which, n, levels in ((0, nU, pc.u_levels), (1, nPi, pc.pi_levels)):
        b = rng.standard_normal(n)
        ref = rbm.vcycle(levels, b) if near_kernel and which == 0 else precond.vcycle(levels, b)
        got = s.vcycle(which, torch.from_numpy(b).cuda()).cpu().numpy()
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
    if not precision:
        for which, levels in ((0, pc.u_levels), (1, pc.pi_levels)):
            for l, lev in enumerate(levels):
                x = rng.standard_normal(lev.A.shape[0])
                y = s.level_apply(which, l, torch.from_numpy(x).cuda()).cpu().numpy()
                assert np.abs(y - lev.A @ x).max() <= 1e-11 * np.abs(lev.A @ x).max()
    s.close()


@pytest.mark.parametrize("precision,degree", [(0, 1), (0, 3), (1, 1), (1, 2)])
def test_update_keeps_the_captured_solves(precision, degree):
    """Solves (both directions) captured before a permeability update give,
    after it, bit for bit what a handle updated before its first solve gives."""
    prob = mi.random_small(9, 8, 7, seed=21, jitter=0.1)
    logk = np.log(prob.kappa[:, 0]) + np.random.default_rng(1).uniform(-2, 2, prob.n_cells)
    lk = torch.from_numpy(logk).cuda()
    opts = dict(autotune=0, coarse_max=30, restart=9, precision=precision, cheb_degree=degree)
    used, fresh = _solver(prob, **opts), _solver(prob, **opts)
    b = used.build_rhs()
    used.solve(b, tol=1e-9)
    used.adjoint_solve(b, tol=1e-6)
    used.update_logk(lk)
    fresh.update_logk(lk)
    for f in ("solve", "adjoint_solve"):
        (x, sx), (y, sy) = (getattr(s, f)(b, tol=1e-9) for s in (used, fresh))
        assert torch.equal(x, y) and sx["iterations"] == sy["iterations"]
    used.close()
    fresh.close()


# dense coarsest level, eliminated in blocks of 32 columns and updated in
# tiles of 32: one level of 6 to 420 unknowns, the last block short
@pytest.mark.parametrize("dims", [(1, 1, 1), (4, 1, 1), (2, 2, 2), (5, 3, 1), (3, 3, 3), (6, 4, 3)])
def test_dense_level_is_the_inverse(dims):
    prob = mi.random_small(*dims, seed=17, jitter=0.1)
    s = _solver(prob, autotune=0, coarse_max=400)
    rng = np.random.default_rng(2)
    for which, n in ((0, s.sizes[0]), (1, s.sizes[2])):
        assert s.hierarchy(which)["levels"] == 1
        x = torch.from_numpy(rng.standard_normal(n)).cuda()
        y = s.vcycle(which, s.level_apply(which, 0, x))
        assert (y - x).abs().max() <= 1e-9 * x.abs().max()  # condition number up to 1.4e4
    s.close()


# the second interface-pressure level's Galerkin product, by rows of slots from
# 2,432 cells on: one line, the first size past it, each residue mod 3 along x
@pytest.mark.parametrize("dims", [(2600, 1, 1), (19, 16, 8), (23, 9, 12), (45, 8, 7), (20, 13, 10)])
def test_galerkin_products_by_rows_of_slots(dims):
    prob = mi.random_small(*dims, seed=29, jitter=0.15)
    levels = precond.build(oracle.assemble(prob), "amg", coarse_max=60).pi_levels
    s = _solver(prob, autotune=0, coarse_max=60)
    rng = np.random.default_rng(4)
    for l, lev in enumerate(levels[1:-1], 1):
        x = rng.standard_normal(lev.A.shape[0])
        y = s.level_apply(1, l, torch.from_numpy(x).cuda()).cpu().numpy()
        assert np.abs(y - lev.A @ x).max() <= 1e-11 * np.abs(lev.A @ x).max()
    s.close()
