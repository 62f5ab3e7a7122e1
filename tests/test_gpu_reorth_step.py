"""The FP32 Lan-DR step with re-orthogonalisation, at site counts that fill no block of 128 or
256 sites and numbers of kept vectors around the groups of four of its multi-dot.  The first
right-hand side's solution is checked with the FP64 oracle's operator (the stopping rule is the
FP64 residual, so the oracle's may exceed tol only by the rounding of its own sum, 1%).  A kept
pair's vector has unit norm, its Rayleigh quotient is the value, and |A v - theta v| is the
residual that the library reports: sums of at most 27648 FP64 terms of order one, so 1e-10
leaves four digits of margin."""
import numpy as np
import pytest
import torch

import synth
from oracle import wilson

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.mark.parametrize("dims,m,k", [((3, 5, 2, 7), 20, 1), ((3, 5, 2, 7), 24, 5), ((4, 6, 6, 8), 30, 12)])
def test_landr_f32(dims, m, k):
    from paper_0901_3163_gb300 import dlz
    U = synth.su3_links(dims, 11)
    b = synth.gaussian_spinor(dims, 0)
    op = dlz.create_operator(dims, torch.from_numpy(U).to("cuda:0"), 0.18, -1)
    p = dlz.params_default(m=m, k=k, tol=TOL, precision=dlz.F32, finish=1)
    x, defl, st = dlz.landr(op, torch.from_numpy(b).to("cuda:0"), p)
    D = wilson.operator(U, 0.18, dims, "D", bc_t=-1)
    A = wilson.operator(U, 0.18, dims, "DdagD", bc_t=-1)
    bb = b.reshape(-1)
    assert st.converged == 1
    assert np.linalg.norm(bb - D(x.cpu().numpy().reshape(-1))) <= 1.01 * TOL * np.linalg.norm(bb)
    for i in range(k):
        v = torch.empty((int(np.prod(dims)), 4, 3), dtype=torch.complex128, device="cuda:0")
        theta, res = dlz.defl_get(defl, i, v)
        v = v.cpu().numpy().reshape(-1)
        Av = A(v)
        assert abs(np.linalg.norm(v) - 1.0) <= 1e-10
        assert abs(np.vdot(v, Av).real - theta) <= 1e-10
        assert abs(np.linalg.norm(Av - theta * v) - res) <= 1e-10
