"""What a set-up leaves behind: device memory after one that fails, and the
buffers that a permeability update has to rewrite."""
import numpy as np
import pytest

import mhfp_inputs as mi
import oracle
from oracle import precond

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


# A cell whose Lame parameter overflows gives an operator that is not finite,
# which the dense elimination of the coarsest displacement level reports.  The
# handle then holds the displacement hierarchy; the Galerkin scratch (441 or,
# with the rigid-body modes, 882 MB here) is given back.
@pytest.mark.parametrize("formulation,near_kernel", [(0, 0), (0, 1), (1, 0)])
def test_failed_setup_gives_its_scratch_back(formulation, near_kernel):
    from paper_2002_09603_gb300 import MhfpError, Solver, default_options
    o = default_options()
    o.autotune, o.restart, o.formulation, o.near_kernel = 0, 1, formulation, near_kernel

    def held(spoil):
        prob = mi.terzaghi_cube(nx=60, ny=60, nz=60)
        if spoil:
            prob.E[prob.n_cells // 2], prob.nu[prob.n_cells // 2] = 1e308, 0.4999
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s = Solver(prob)
        s.assemble_condense()
        if spoil:
            with pytest.raises(MhfpError, match="coarsest"):
                s.setup_precond(o)
        else:
            s.setup_precond(o)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
        s.close()
        return used

    held(False)  # the context's own growth
    whole = held(False)
    failed = held(True)
    assert failed < whole, (failed, whole)


# Every buffer of the interface-pressure hierarchy that follows from kappa: the
# face level, the 25-point cell level (its prolongator in the cycles' layout),
# and a 125-point level of 140 points, which the cycles read row by row (a copy
# of its own, in FP32 another).  After an update the levels and the V-cycle are
# the oracle's for the new field (tolerances as in test_gpu_parity).
@pytest.mark.parametrize("precision", [0, 1])
def test_update_rewrites_the_row_major_level(precision):
    from paper_2002_09603_gb300 import default_options, prepare
    prob = mi.random_small(20, 13, 10, seed=23, jitter=0.1)
    prob.kappa[:] = prob.kappa[:, :1]  # isotropic, as the update's field
    o = default_options()
    o.autotune, o.coarse_max, o.precision = 0, 30, precision
    s = prepare(prob, o)
    assert s.hierarchy(1)["points"][2:] == [140, 12] and s.hierarchy(1)["schedule"][2] == 32
    rng = np.random.default_rng(9)
    logk = np.log(prob.kappa[:, 0]) + rng.uniform(-2, 2, prob.n_cells)
    s.update_logk(torch.from_numpy(logk).cuda())
    prob.kappa[:] = np.exp(logk)[:, None]
    levels = precond.build(oracle.assemble(prob), "amg", coarse_max=30).pi_levels
    # the residual of a field in the 125-point level's range: there the old
    # values of that level alone would change the result by 6e-2 of its largest
    # entry, the old prolongator onto it by 6e-3
    b = levels[0].A @ (levels[0].P @ (levels[1].P @ rng.standard_normal(140)))
    ref = precond.vcycle(levels, b)
    got = s.vcycle(1, torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.abs(got - ref).max() <= (1e-5 if precision else 1e-10) * np.abs(ref).max()
    for l, lev in enumerate(levels):
        x = rng.standard_normal(lev.A.shape[0])
        y = s.level_apply(1, l, torch.from_numpy(x).cuda()).cpu().numpy()
        assert np.abs(y - lev.A @ x).max() <= 1e-11 * np.abs(lev.A @ x).max()
    s.close()
