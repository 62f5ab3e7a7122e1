"""The launch forms of the tensor-core products of FP32 basis vectors: coefficients that stay in
shared memory (two ring depths), that are copied per chunk (two ring depths) and the
single-stage form of the widest outputs; lengths of one float4, one element past a tile of 512
floats and a ragged end; projections of one chunk, of one segment of 64 chunks and one more.

Tolerance: as in test_gpu_tc.py, an output is within 4e-6 (combine) or 1e-5 (dots) times
sum_i |c_i| |v_i| of the FP64 product: three TF32 products of the two parts of each factor, each
part kept to 11 bits, and FP32 sums."""
import numpy as np
import pytest

from tests._lib import dlz

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nin,nout,length", [(1, 1, 4), (121, 61, 516), (150, 64, 1540), (201, 112, 516),
                                             (201, 160, 1540), (7, 256, 516), (40, 241, 4 * 999)])
def test_combine_forms(nin, nout, length):
    rng = np.random.default_rng(nin + nout)
    V = rng.standard_normal((nin, length)).astype(np.float32)
    P = rng.standard_normal((nin, nout))
    out = dlz().basis_combine(torch.from_numpy(V).cuda(), P).cpu().numpy()
    ref = P.T @ V.astype(np.float64)
    assert np.all(np.abs(out - ref) <= 4e-6 * (np.abs(P).T @ np.abs(V.astype(np.float64))))


@pytest.mark.parametrize("nin,nq,chunks", [(1, 1, 1), (128, 16, 64), (33, 8, 65), (16, 9, 152 * 64 + 3)])
def test_dots_segments(nin, nq, chunks):
    rng = np.random.default_rng(chunks)
    L = 16 * chunks

    def field(n):
        return (rng.standard_normal((n, L)) + 1j * rng.standard_normal((n, L))).astype(np.complex64)
    V, R = field(nin), field(nq)
    C = dlz().basis_dots(torch.from_numpy(V).cuda(), torch.from_numpy(R).cuda())
    V64, R64 = V.astype(np.complex128), R.astype(np.complex128)
    ref = np.conj(V64) @ R64.T
    assert np.all(np.abs(C.T - ref) <= 1e-5 * (np.abs(V64) @ np.abs(R64).T) + 1e-30)
