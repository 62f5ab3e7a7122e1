"""The FP32 D-CG whose direction and iterate are updated once per block of iterations, at
sizes around its tiles: site counts that fill no block of 128 sites or 256 elements, one
right-hand side, a ragged and a full batch, and a zero right-hand side beside others.  The
solution is checked with the FP64 oracle's operator: the stopping rule is the FP64 residual,
so the oracle's residual may exceed tol only by the rounding of its own sum (1%)."""
import numpy as np
import pytest
import torch

import synth
from oracle import wilson

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nrhs,eo", [((3, 5, 2, 7), 1, False), ((3, 5, 2, 7), 16, False), ((4, 4, 4, 9), 5, False),
                                          ((2, 4, 6, 4), 7, True), ((4, 6, 8, 6), 16, True)])
def test_dcg_f32_residual(dims, nrhs, eo):
    from paper_0901_3163_gb300 import dlz
    kappa, tol = 0.18, 1e-11
    U = synth.su3_links(dims, 5)
    B = synth.gaussian_spinors(dims, range(nrhs))
    if nrhs > 2:
        B[1] = 0.0
    Bd = torch.from_numpy(B).to("cuda:0")
    p = dlz.params_default(tol=tol, precision=dlz.F32)
    make = dlz.create_operator_eo if eo else dlz.create_operator
    op = make(dims, torch.from_numpy(U).to("cuda:0"), kappa, -1)
    if eo:
        xe, st = dlz.dcg(op, None, dlz.eo_prepare(op, Bd), p)
        X = dlz.eo_reconstruct(op, xe, Bd)
    else:
        X, st = dlz.dcg(op, None, Bd, p)
    D = wilson.operator(U, kappa, dims, "D", bc_t=-1)
    X = X.cpu().numpy()
    for i in range(nrhs):
        b = B[i].reshape(-1)
        assert st[i].converged == 1
        if not b.any():
            assert not X[i].any()
            continue
        # even-odd: the even system's right-hand side is up to a factor of two longer
        assert np.linalg.norm(b - D(X[i].reshape(-1))) <= (2.0 if eo else 1.01) * tol * np.linalg.norm(b)
