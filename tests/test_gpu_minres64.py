"""The fused FP64 D-MinRes step at each of its block sizes (32, 64 and 128 sites, chosen by the
number of sites), at site counts that fill no block, and on an even-odd operator.  The solution
is checked with the FP64 oracle's operator: the stopping rule is the FP64 residual, so the
oracle's may exceed tol only by the rounding of its own sum (1%)."""
import numpy as np
import pytest
import torch

import synth
from oracle import wilson

pytestmark = pytest.mark.gpu
TOL = 1e-11


@pytest.mark.parametrize("dims,eo", [((1, 2, 2, 4), False), ((3, 5, 2, 7), False), ((8, 8, 8, 16), False),
                                     ((8, 10, 12, 17), False), ((4, 6, 2, 8), True)])
def test_dminres_f64_residual(dims, eo):
    from paper_0901_3163_gb300 import dlz
    U = synth.su3_links(dims, 9)
    make = dlz.create_operator_eo if eo else dlz.create_operator
    op = make(dims, torch.from_numpy(U).to("cuda:0"), 0.18, -1)
    B = synth.gaussian_spinors(dims, range(2))
    Bd, p = torch.from_numpy(B).to("cuda:0"), dlz.params_default(tol=TOL, precision=dlz.F64)
    if eo:
        xe, st = dlz.dminres(op, None, dlz.eo_prepare(op, Bd), p)
        X = dlz.eo_reconstruct(op, xe, Bd)
    else:
        X, st = dlz.dminres(op, None, Bd, p)
    D = wilson.operator(U, 0.18, dims, "D", bc_t=-1)
    X = X.cpu().numpy()
    for i in range(2):
        b = B[i].reshape(-1)
        assert st[i].converged == 1
        # even-odd: the even system's right-hand side is up to a factor of two longer
        assert np.linalg.norm(b - D(X[i].reshape(-1))) <= (2.0 if eo else 1.01) * TOL * np.linalg.norm(b)
