"""The forms that the rules on sizes choose above the other tests' meshes,
against the FP64 oracle (tolerances as in test_gpu_parity): one mesh of 68,880
nodes and 63,960 cells with odd sides."""
import numpy as np
import pytest

import mhfp_inputs as mi
import oracle
from oracle import precond, rbm, system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(scope="module")
def mesh(_built):
    prob = mi.random_small(41, 40, 39, seed=11, jitter=0.2)
    return prob, oracle.assemble(prob)


@pytest.fixture(scope="module")
def oracle_pc(mesh):
    return precond.build(mesh[1], "amg")


@pytest.fixture(scope="module")
def oracle_rbm_levels(mesh):
    return rbm.build_u_hierarchy(mesh[1])


def _solver(prob, **opts):
    from paper_2002_09603_gb300 import default_options, prepare
    o = default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    return prepare(prob, o)


def _vcycle_close(s, which, ref, b, tol):
    got = s.vcycle(which, torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


# FP64 displacement rows: both operators by a thread per row, the V-cycle's steps
# and residual by nine threads per node (its steps by a thread per row: the 64^3
# V-cycle of test_gpu_fullsize)
def test_fp64_rows_by_a_thread_per_row(mesh, oracle_pc):
    prob, B = mesh
    s = _solver(prob, autotune=0)
    A = system.system_matrix(B)
    rng = np.random.default_rng(4)
    x, b = rng.standard_normal(s.n), rng.standard_normal(s.sizes[0])
    xd = torch.from_numpy(x).cuda()
    for f, M in ((s.apply_operator, A), (s.apply_operator_t, A.T)):
        y, ref, o = f(xd).cpu().numpy(), M @ x, 0
        for n in B.sizes:
            assert np.abs(y[o:o + n] - ref[o:o + n]).max() <= 1e-12 * np.abs(ref[o:o + n]).max()
            o += n
    _vcycle_close(s, 0, precond.vcycle(oracle_pc.u_levels, b), b, 1e-10)
    s.close()


# The schedules that the size rule takes without the autotuner (coarse levels of
# 2,744 and 2,548 points: past the warp-per-point size), and with them both
# V-cycles: from 65,536 fine points on the prolongation of the finest levels
# takes its wide forms (3 x 3, with the rigid-body modes 3 x 6, and scalar).
@pytest.mark.parametrize("precision,near_kernel,u_sched", [(0, 0, 8), (0, 1, 64), (1, 0, 32), (1, 1, 32)])
def test_size_rule_and_wide_transfers(mesh, oracle_pc, oracle_rbm_levels, precision, near_kernel, u_sched):
    prob, _ = mesh
    s = _solver(prob, autotune=0, precision=precision, near_kernel=near_kernel)
    assert s.hierarchy(0)["points"] == [68880, 2744, 125] and s.hierarchy(0)["schedule"][1] == u_sched
    assert s.hierarchy(1)["points"] == [196679, 63960, 2548, 125] and s.hierarchy(1)["schedule"][2] == 64
    rng = np.random.default_rng(6)
    tol = 1e-5 if precision else 1e-10
    b = rng.standard_normal(s.sizes[0])
    ref = rbm.vcycle(oracle_rbm_levels, b) if near_kernel else precond.vcycle(oracle_pc.u_levels, b)
    _vcycle_close(s, 0, ref, b, tol)
    b = rng.standard_normal(s.sizes[2])
    _vcycle_close(s, 1, precond.vcycle(oracle_pc.pi_levels, b), b, tol)
    s.close()
