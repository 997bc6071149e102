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
