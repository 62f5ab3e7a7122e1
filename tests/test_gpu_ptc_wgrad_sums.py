"""The tensor-core weight gradient where every term of its sums has the same sign and the largest
remainders that its bfloat16 parts can have: on unit links every entry is 48 v^2 per 16 sites.
The values are of 24 bits and their parts of 8, so only sums may round.  On 16 sites a sum is one
accumulator: 3 steps with the products of the leading parts, whose partial sums 1/3, 2/3 and 3/3
of the result lose at most 2^-23 of themselves each, and 21 steps below 2^-6 of it: 2.9e-7."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("imaginary", [False, True])
def test_sums_of_one_sign(imaginary):
    from paper_0901_3163_gb300 import dlz
    dims = (2, 2, 2, 2)
    v = np.complex64(1.0 + 2.0**-7 - 2.0**-23)
    x = np.full((1, 16, 4, 3), v, dtype=np.complex64)
    g = np.complex64(1j) * x if imaginary else x
    op = dlz.create_operator(dims, torch.from_numpy(synth.unit_links(dims)).cuda(), 0.1)
    net = dlz.net_create(op, (1, 1), [np.ones((9, 1, 1, 4, 4), dtype=np.complex64)])
    dlz.net_forward(net, torch.from_numpy(x).cuda())
    dlz.net_backward(net, torch.from_numpy(g).cuda())
    want = 48.0 * float(v.real)**2 * (1j if imaginary else 1.0)
    assert np.abs(dlz.net_get(net, 1)[0].astype(np.complex128) - want).max() <= 2.9e-7 * abs(want)
