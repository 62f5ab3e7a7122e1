"""Calls of the network that are refused, and that it is usable afterwards."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DIMS = (4, 4, 2, 4)


def _net():
    from paper_0901_3163_gb300 import dlz
    U = torch.from_numpy(synth.su3_links(DIMS, 2)).cuda()
    op = dlz.create_operator(DIMS, U, 0.2)
    rng = np.random.default_rng(1)
    Ws = [(0.1 * rng.standard_normal(s)).astype(np.complex64) for s in dlz.net_weight_shapes((1, 4, 1))]
    x = torch.from_numpy(synth.gaussian_spinors(DIMS, [1, 2]).astype(np.complex64)).cuda()
    return dlz, U, op, dlz.net_create(op, (1, 4, 1), Ws), x


def test_no_even_odd_operator():
    dlz, U, op, net, x = _net()
    want = dlz.net_forward(net, x)
    with pytest.raises(dlz.DlzError) as e:
        dlz.net_bind(net, dlz.create_operator_eo(DIMS, U, 0.2))
    assert e.value.code == dlz.ERR_BADARG
    assert torch.equal(dlz.net_forward(net, x), want)


def test_after_an_allocation_that_failed():
    dlz, U, op, net, x = _net()
    want = dlz.net_forward(net, x)
    out = torch.empty_like(x)
    # activations of 320 GB: refused when the first buffer is allocated, before any kernel
    nvec = (320 << 30) // (96 * synth.volume(DIMS))
    with pytest.raises(dlz.DlzError) as e:
        dlz._check(dlz.lib.dlz_net_forward(net.handle, x.data_ptr(), nvec, out.data_ptr()))
    assert e.value.code == dlz.ERR_OOM
    with pytest.raises(dlz.DlzError) as e:
        dlz.net_backward(net, x)                          # the forward's activations are gone
    assert e.value.code == dlz.ERR_BADARG
    assert torch.equal(dlz.net_forward(net, x), want)
