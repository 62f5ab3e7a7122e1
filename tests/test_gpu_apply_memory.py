"""dlz_apply and the work memory that an operator keeps: more right-hand sides than a kept buffer
of 64 MiB has room for go through several launches, and calls of several host threads on one
operator have a buffer each.  Both give the bits of one call per right-hand side."""
import threading

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DIMS = (8, 6, 8, 11)                     # 4224 sites: 0.81 MB per FP64 vector


def _setup():
    from paper_0901_3163_gb300 import dlz
    op = dlz.create_operator(DIMS, torch.from_numpy(synth.su3_links(DIMS, 3)).cuda(), 0.137, -1)
    torch.manual_seed(1)
    return dlz, op


# work vectors per right-hand side of D^dag D: FP64 one; FP32 that is only 8-byte aligned three;
# bfloat16 three of half the size
@pytest.mark.parametrize("form,nrhs", [("f64", 83), ("f64", 166), ("f32_odd", 56), ("bf16", 111)])
def test_several_launches(form, nrhs):
    dlz, op = _setup()
    shape = (nrhs, synth.volume(DIMS), 4, 3)
    x = torch.randn(shape, dtype=torch.complex128 if form == "f64" else torch.complex64, device="cuda")
    out = torch.empty_like(x)
    dtype = dlz.BF16 if form == "bf16" else None
    if form == "f32_odd":
        xs = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].reshape(shape)
        out = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].reshape(shape)
        x = xs.copy_(x)
    dlz.apply(op, dlz.DDAGD, x, out, dtype)
    for r in (0, 1, nrhs // 2, nrhs - 2, nrhs - 1):
        assert torch.equal(dlz.apply(op, dlz.DDAGD, x[r:r + 1], None, dtype), out[r:r + 1]), r


def test_threads():
    dlz, op = _setup()
    xs = [torch.randn((3, synth.volume(DIMS), 4, 3), dtype=torch.complex64, device="cuda") for _ in range(4)]
    want = [dlz.apply(op, dlz.DDAGD, x) for x in xs]
    outs = [[torch.empty_like(x) for _ in range(8)] for x in xs]
    torch.cuda.synchronize()

    def calls(i):
        for o in outs[i]:
            dlz.apply(op, dlz.DDAGD, xs[i], o)

    ts = [threading.Thread(target=calls, args=(i,)) for i in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for i in range(4):
        assert all(torch.equal(o, want[i]) for o in outs[i])
