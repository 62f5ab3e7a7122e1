"""dlz_apply over the routes it chooses between, at the sizes where they change: blocks of 32,
64 and 128 sites with remainders, one and several right-hand sides in a launch, and FP32
vectors that are only 8-byte aligned, which must give the bits of the aligned call.  FP64
elements against the FP64 oracle to 1e-14 of the largest element, FP32 to 3e-6 (rounding of
the input and 24-bit arithmetic over a sum of about 100 terms)."""
import numpy as np
import pytest
import torch

import synth
from oracle import wilson

pytestmark = pytest.mark.gpu
REFS = {"D": wilson.apply_D, "DDAG": wilson.apply_Ddag, "Q": wilson.apply_Q, "DDAGD": wilson.apply_DdagD}


# sites x right-hand sides below, at and above 152 * 64 (32-thread blocks)
@pytest.mark.parametrize("dims,nrhs", [((1, 3, 1, 5), 1), ((3, 5, 7, 9), 1), ((3, 5, 7, 9), 11), ((8, 8, 8, 9), 3),
                                       ((10, 10, 10, 8), 5), ((7, 9, 11, 13), 5), ((12, 10, 14, 6), 4)])
def test_apply_routes(dims, nrhs):
    from paper_0901_3163_gb300 import dlz
    U = synth.su3_links(dims, 3)
    psi = synth.gaussian_spinors(dims, range(nrhs))
    op = dlz.create_operator(dims, torch.from_numpy(U).cuda(), 0.137, -1)
    x64 = torch.from_numpy(psi).cuda()
    x32 = x64.to(torch.complex64)
    n = x32.numel()
    odd_in = torch.zeros(n + 1, dtype=torch.complex64, device="cuda")[1:].reshape(x32.shape)
    odd_out = torch.empty(n + 1, dtype=torch.complex64, device="cuda")[1:].reshape(x32.shape)
    odd_in.copy_(x32)
    for name, ref in REFS.items():
        which = getattr(dlz, name)
        want = ref(U, psi, 0.137, dims, -1)
        top = np.abs(want).max()
        assert np.abs(dlz.apply(op, which, x64).cpu().numpy() - want).max() <= 1e-14 * top, name
        got = dlz.apply(op, which, x32)
        assert np.abs(got.cpu().numpy() - want).max() <= 3e-6 * top, name
        assert torch.equal(dlz.apply(op, which, odd_in, odd_out), got), name
        assert torch.equal(dlz.apply(op, which, x32[nrhs - 1:]), got[nrhs - 1:]), name
