"""What a set-up leaves behind."""
import pytest

import mhfp_inputs as mi

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
