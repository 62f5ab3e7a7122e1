"""The tensor-core form of the network's layers at the sizes where it can go wrong: site counts
around its tiles of 42, one and several vectors, channel counts that pad its chunks (odd, more
than one chunk of 6) and its columns, layers on both sides of the rule that chooses it.  Forward,
input gradient and weight gradients against the FP64 oracle with the bfloat16 weights in use.
Tolerance: 24-bit arithmetic over sums of at most 9 * 16 * 8 terms and three layers: 4e-6 of the
largest element (measured relative errors stay below 1e-6)."""
import numpy as np
import pytest
import torch

import synth
from oracle import ptc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nvec,widths", [((2, 3, 7, 1), 1, (1, 4, 1)), ((1, 2, 3, 7), 3, (1, 16, 16, 1)),
                                              ((3, 5, 2, 7), 2, (1, 5, 7, 1)), ((4, 4, 2, 8), 2, (1, 8, 13, 3, 1)),
                                              ((4, 6, 5, 8), 2, (1, 12, 16, 1))])
def test_network_against_oracle(dims, nvec, widths):
    from paper_0901_3163_gb300 import dlz
    rng = np.random.default_rng(3)
    U = synth.su3_links(dims, 6)
    Ws = [((rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(72.0 * s[2])).astype(np.complex64)
          for s in dlz.net_weight_shapes(widths)]
    V = synth.volume(dims)
    x = (rng.standard_normal((nvec, V, 4, 3)) + 1j * rng.standard_normal((nvec, V, 4, 3))).astype(np.complex64)
    g = (rng.standard_normal((nvec, V, 4, 3)) + 1j * rng.standard_normal((nvec, V, 4, 3))).astype(np.complex64)
    op = dlz.create_operator(dims, torch.from_numpy(U).cuda(), 0.2)
    net = dlz.net_create(op, widths, Ws)
    f = dlz.net_forward(net, torch.from_numpy(x).cuda()).cpu().numpy()
    gin = dlz.net_backward(net, torch.from_numpy(g).cuda(), want_input_grad=True).cpu().numpy()
    gw = dlz.net_get(net, 1)
    Wb = [w.astype(np.complex128) for w in dlz.net_get(net, 2)]
    want_w = [np.zeros(w.shape, dtype=np.complex128) for w in Wb]
    for i in range(nvec):
        want, acts = ptc.forward(Wb, U, x[i].astype(np.complex128), dims)
        wg, wi = ptc.backward(Wb, U, acts, g[i].astype(np.complex128), dims)
        assert np.abs(f[i] - want).max() <= 4e-6 * np.abs(want).max()
        assert np.abs(gin[i] - wi).max() <= 4e-6 * np.abs(wi).max()
        for a, b in zip(want_w, wg):
            a += b
    for a, b in zip(gw, want_w):
        assert np.abs(a - b).max() <= 4e-6 * np.abs(b).max()
