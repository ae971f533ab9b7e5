"""The CUDA-core sketch (FP64 data, and FP32 data whose columns are not 16-byte
aligned) at the edges of its groups and chunks: l around multiples of 16,
windows around 16, 32 and 64 columns and past one window, ragged row tiles,
several windows that add to Y, against the oracle's products, with the
repository's bars (1e-12 FP64, 1e-5 FP32); the coarse rows exactly; and
infinities and NaN in one column stay in that column of W."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1e-5), (torch.float64, 1e-12)])
@pytest.mark.parametrize("m,n,l,chunks", [
    (63, 5, 3, [5]), (65, 17, 16, [17]), (1001, 33, 17, [16, 17]), (777, 64, 32, [64]),
    (20001, 65, 33, [32, 32, 1]), (515, 97, 48, [97]), (333, 321, 49, [321]),
    (4097, 640, 64, [640])])
def test_simt_sketch_forms(dtype, tol, m, n, l, chunks):
    from paper_1905_13257_gb300 import IdSketch
    A = gaussian_matrix(m, n, seed=m + n, dtype=dtype, device="cuda")
    sk = IdSketch(m, n, 1, l, seed=7, dtype=dtype, want_Y=True, grid=(1, 1, m), ncomp=1,
                  coarse_stride=(1, 1, 3), want_coarse=True)
    j = 0
    for c in chunks:
        sk.stream_columns(A[:, j:j + c])
        j += c
    W, Y, Ac = sk.sketches()
    An = A.cpu().double().numpy()
    Wo, Yo = oracle.sketch(An, oracle.psi(l, m, 7), oracle.omega(n, l, 7))
    assert rel(W.cpu().numpy(), Wo) <= tol
    assert rel(Y.cpu().double().numpy(), Yo) <= tol
    assert torch.equal(Ac, A[::3])
    sk.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_non_finite_entries_stay_in_their_column(dtype):
    from paper_1905_13257_gb300 import IdSketch
    m, n, l = 1001, 40, 20
    A = gaussian_matrix(m, n, seed=1, dtype=dtype, device="cuda").T.contiguous().T
    A[500, 3] = float("inf")
    A[700, 9] = float("nan")
    sk = IdSketch(m, n, 1, l, seed=7, dtype=dtype, want_Y=False)
    sk.stream_columns(A)
    W = sk.sketches()[0].cpu().numpy()
    P = oracle.psi(l, m, 7)
    assert np.all(np.isinf(W[:, 3])) and np.array_equal(np.sign(W[:, 3]), np.sign(P[:, 500]))
    assert np.all(np.isnan(W[:, 9]))
    assert np.all(np.isfinite(np.delete(W, [3, 9], 1)))
    sk.close()
