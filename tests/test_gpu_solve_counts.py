"""dlz_stats.mvps of the FP32 defect-correction solves on a single right-hand side without a
deflation set: the applications of D and D^dagger that were made.  From x = 0 the first residual
is the right-hand side itself and takes none; every later pass of the outer loop takes one, an
inner MinRes iteration one, an inner CG iteration two."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver,per_iteration", [("dminres", 1), ("dcg", 2)])
@pytest.mark.parametrize("zero", [False, True])
def test_mvps(solver, per_iteration, zero):
    from paper_0901_3163_gb300 import dlz
    dims = (4, 4, 4, 6)
    op = dlz.create_operator(dims, torch.from_numpy(synth.su3_links(dims, 2)).cuda(), 0.18)
    b = torch.from_numpy(synth.gaussian_spinors(dims, [1])).cuda()
    if zero:
        b.zero_()
    _, (st,) = getattr(dlz, solver)(op, None, b, dlz.params_default(tol=1e-10, precision=dlz.F32))
    assert st.converged == 1 and (st.cycles > 1 or zero)
    assert st.mvps == per_iteration * st.iterations + st.cycles
