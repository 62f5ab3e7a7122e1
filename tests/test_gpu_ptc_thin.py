"""Layers with few channels on both sides of the rule that sends them to the tensor cores (at 4096
sites and below, with 1, 2, 3 and 4 input channels), forward, input gradient and weight gradients
against the FP64 oracle with the bfloat16 weights in use.  A vector's output does not depend on the
vectors beside it.  Tolerance: 24-bit arithmetic over sums of at most 9 * 9 * 8 terms and three
layers, and over 4096 * 3 sites and colours in the weight gradients: 4e-6 of the largest element."""
import numpy as np
import pytest
import torch

import synth
from oracle import ptc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (9, 7, 13, 5)])
@pytest.mark.parametrize("widths", [(1, 4, 1), (1, 8, 4, 1), (1, 9, 3, 1), (1, 2, 4, 1), (1, 2, 5, 1), (1, 3, 4, 1)])
def test_network_against_oracle(dims, widths):
    from paper_0901_3163_gb300 import dlz
    rng = np.random.default_rng(3)
    U = synth.su3_links(dims, 6)
    Ws = [((rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(72.0 * s[2])).astype(np.complex64)
          for s in dlz.net_weight_shapes(widths)]
    V = synth.volume(dims)
    x, g = ((rng.standard_normal((2, V, 4, 3)) + 1j * rng.standard_normal((2, V, 4, 3))).astype(np.complex64)
            for _ in range(2))
    op = dlz.create_operator(dims, torch.from_numpy(U).cuda(), 0.2)
    net = dlz.net_create(op, widths, Ws)
    xd = torch.from_numpy(x).cuda()
    alone = dlz.net_forward(net, xd[1:])
    f = dlz.net_forward(net, xd)
    assert torch.equal(f[1:], alone)
    gin = dlz.net_backward(net, torch.from_numpy(g).cuda(), want_input_grad=True).cpu().numpy()
    gw = dlz.net_get(net, 1)
    Wb = [w.astype(np.complex128) for w in dlz.net_get(net, 2)]
    want_w = [np.zeros(w.shape, dtype=np.complex128) for w in Wb]
    for i in range(2):
        want, acts = ptc.forward(Wb, U, x[i].astype(np.complex128), dims)
        wg, wi = ptc.backward(Wb, U, acts, g[i].astype(np.complex128), dims)
        assert np.abs(f[i].cpu().numpy() - want).max() <= 4e-6 * np.abs(want).max()
        assert np.abs(gin[i] - wi).max() <= 4e-6 * np.abs(wi).max()
        want_w = [p + q for p, q in zip(want_w, wg)]
    for a, b in zip(gw, want_w):
        assert np.abs(a - b).max() <= 4e-6 * np.abs(b).max()
