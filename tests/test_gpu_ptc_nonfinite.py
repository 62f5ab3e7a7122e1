"""Infinities, NaN and overflow in the network: the outputs, input gradients and weight gradients
have a finite value, an infinity of the same sign or NaN exactly where the plain complex arithmetic
of the layers has (the oracle's, whose range is wider, on inputs that are infinite to begin with),
and the finite ones its value to 4e-6 of the largest.  The gradients of a pass are added to those
of earlier ones whatever the pass holds."""
import numpy as np
import pytest
import torch

import synth
from oracle import ptc

pytestmark = pytest.mark.gpu
DIMS = (4, 3, 2, 6)
WIDTHS = (1, 5, 8, 1)


def _same(got, want):
    got, want = got.reshape(-1).view(np.float32).astype(np.float64), want.reshape(-1).view(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(np.isinf(got), inf) and np.array_equal(got[inf], want[inf])
    ok = np.isfinite(want)
    if ok.any():
        assert np.abs(got[ok] - want[ok]).max() <= 4e-6 * np.abs(want[ok]).max()


@pytest.mark.parametrize("where", ["gradient", "input", "nan"])
@pytest.mark.parametrize("in_place", [False, True])
def test_pattern_of_plain_arithmetic(where, in_place):
    from paper_0901_3163_gb300 import dlz
    rng = np.random.default_rng(4)
    U = synth.su3_links(DIMS, 6)
    Ws = [((rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(72.0 * s[2])).astype(np.complex64)
          for s in dlz.net_weight_shapes(WIDTHS)]
    V = synth.volume(DIMS)
    shape = (2, V, 4, 3)
    x = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    g = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    clean = g.copy()
    # bfloat16 values among the finite ones: their second and third parts are zero
    g[:, ::3] = np.round(g[:, ::3].view(np.float32) * 8).view(np.complex64) / 8
    if where == "gradient":
        g[1, 5, 2, 1] = complex(np.inf, 0.5)
    elif where == "input":
        x[0, 7, 1, 2] = complex(0.25, -np.inf)
    else:
        g[0, 3, 0, 0] = complex(1.0, np.nan)
    op = dlz.create_operator(DIMS, torch.from_numpy(U).cuda(), 0.2)
    net = dlz.net_create(op, WIDTHS, Ws)
    # a finite pass first: its gradients stay in the sum
    x0 = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    dlz.net_forward(net, torch.from_numpy(x0).cuda())
    dlz.net_backward(net, torch.from_numpy(clean).cuda())
    xd, gd = torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda()
    f = dlz.net_forward(net, xd).cpu().numpy()
    if in_place:
        dlz._check(dlz.lib.dlz_net_backward(net.handle, gd.data_ptr(), 2, gd.data_ptr()))
        gin = gd.cpu().numpy()
    else:
        gin = dlz.net_backward(net, gd, want_input_grad=True).cpu().numpy()
    gw = dlz.net_get(net, 1)
    Wb = [w.astype(np.complex128) for w in dlz.net_get(net, 2)]
    want_w = [np.zeros(w.shape, dtype=np.complex128) for w in Wb]
    with np.errstate(all="ignore"):
        for a, b, check in ((x0, clean, False), (x, g, True)):
            for i in range(2):
                want, acts = ptc.forward(Wb, U, a[i].astype(np.complex128), DIMS)
                wg, wi = ptc.backward(Wb, U, acts, b[i].astype(np.complex128), DIMS)
                if check:
                    _same(f[i], want)
                    _same(gin[i], wi)
                want_w = [p + q for p, q in zip(want_w, wg)]
    for a, b in zip(gw, want_w):
        _same(a, b)


def test_finite_again(m=None):
    """A pass that is finite after one that was not is computed as ever."""
    from paper_0901_3163_gb300 import dlz
    rng = np.random.default_rng(5)
    V = synth.volume(DIMS)
    x = torch.from_numpy((rng.standard_normal((1, V, 4, 3)) + 1j * rng.standard_normal((1, V, 4, 3))).astype(np.complex64)).cuda()
    op = dlz.create_operator(DIMS, torch.from_numpy(synth.su3_links(DIMS, 6)).cuda(), 0.2)
    Ws = [((rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(72.0 * s[2])).astype(np.complex64)
          for s in dlz.net_weight_shapes(WIDTHS)]
    net = dlz.net_create(op, WIDTHS, Ws)
    want = dlz.net_forward(net, x)
    dlz.net_backward(net, x)
    gw = dlz.net_get(net, 1)
    bad = x.clone()
    bad[0, 0, 0, 0] = float("inf")
    dlz.net_forward(net, bad)
    dlz.net_backward(net, bad)
    dlz.net_zero_grad(net)
    assert torch.equal(dlz.net_forward(net, x), want)
    dlz.net_backward(net, x)
    assert all(np.array_equal(a, b) for a, b in zip(dlz.net_get(net, 1), gw))
