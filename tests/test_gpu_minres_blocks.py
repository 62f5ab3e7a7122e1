"""The FP32 D-MinRes whose directions and iterate are updated once per block of iterations,
at sizes around its tiles: site counts that fill no block of 128 sites or 256 elements, one
right-hand side (whose sums are taken inside the kernels), a ragged and a full batch, a zero
right-hand side beside others, and several lattices in one call in both launch forms.  The
solution is checked with the FP64 oracle's operator: the stopping rule is the FP64 residual,
so the oracle's residual may exceed tol only by the rounding of its own sum (1%)."""
import numpy as np
import pytest
import torch

import synth
from oracle import wilson

pytestmark = pytest.mark.gpu
TOL = 1e-11


def _check(U, kappa, dims, B, X, st):
    D = wilson.operator(U, kappa, dims, "D", bc_t=-1)
    X = X.cpu().numpy()
    for i in range(len(B)):
        b = B[i].reshape(-1)
        assert st[i].converged == 1
        if not b.any():
            assert not X[i].any()
            continue
        assert np.linalg.norm(b - D(X[i].reshape(-1))) <= 1.01 * TOL * np.linalg.norm(b)


def _problem(dims, nrhs, seed):
    from paper_0901_3163_gb300 import dlz
    U = synth.su3_links(dims, seed)
    B = synth.gaussian_spinors(dims, range(nrhs))
    if nrhs > 2:
        B[1] = 0.0
    op = dlz.create_operator(dims, torch.from_numpy(U).to("cuda:0"), 0.18, -1)
    return dlz, U, B, op


@pytest.mark.parametrize("dims,nrhs", [((3, 5, 2, 7), 1), ((3, 5, 2, 7), 16), ((4, 4, 4, 9), 5), ((8, 4, 6, 8), 11)])
def test_dminres_f32_residual(dims, nrhs):
    dlz, U, B, op = _problem(dims, nrhs, 5)
    X, st = dlz.dminres(op, None, torch.from_numpy(B).to("cuda:0"), dlz.params_default(tol=TOL, precision=dlz.F32))
    _check(U, 0.18, dims, B, X, st)


@pytest.mark.parametrize("form", ["graph", "persistent"])
def test_batch_dminres_residual(form, monkeypatch):
    monkeypatch.setenv("DLZ_MULTI_FORM", form)
    shapes = [((3, 5, 2, 7), 2), ((4, 4, 4, 4), 5), ((6, 4, 5, 8), 1)]
    ps = [_problem(d, n, 7 + i) for i, (d, n) in enumerate(shapes)]
    dlz = ps[0][0]
    Xs, sts = dlz.batch_dminres([p[3] for p in ps], [None] * 3, [torch.from_numpy(p[2]).to("cuda:0") for p in ps],
                                dlz.params_default(tol=TOL, precision=dlz.F32))
    for (dims, _), p, X, st in zip(shapes, ps, Xs, sts):
        _check(p[1], 0.18, dims, p[2], X, st)
