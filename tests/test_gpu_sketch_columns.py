"""Windows of several buffers (the sketch's producer copies column by column)
at the edges of its boxes: ragged last row blocks of every remainder modulo 4
(the rows after the last 16 bytes), fewer than 4 rows in the last block,
windows around 32 and 128 columns, one-column buffers, several windows, with
and without Y, l up to 96, each precision form; against the oracle's products
(1e-5; precision forms: of the rounded data).  Rows and columns outside the
matrix hold NaN in the callers' buffers and must not be read into the result;
and the same columns in one buffer give bit-equal W and Y."""
import numpy as np
import pytest
import torch

import oracle
from oracle import fp8 as ofp8
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("m,widths,l,want_Y,prec", [
    (128, [1] * 9, 12, True, "exact"), (129, [31, 2], 20, True, "exact"),
    (130, [32, 32, 32, 33], 60, True, "exact"), (131, [64, 65], 64, False, "exact"),
    (1021, [16] * 8 + [3], 33, True, "exact"), (4099, [100, 300, 200], 60, True, "exact"),
    (2050, [37, 90], 96, False, "exact"), (20003, [32] * 16, 60, True, "bf16"),
    (1157, [40, 90, 1], 30, True, "fp8"), (50001, [32] * 5, 90, False, "bf16")])
def test_windows_of_several_buffers(m, widths, l, want_Y, prec):
    from paper_1905_13257_gb300 import IdSketch
    n, ld = sum(widths), (m + 3) // 4 * 4 + 4
    A = gaussian_matrix(m, n, seed=m + n, dtype=torch.float32, device="cuda")
    A = (A * torch.linspace(0.5, 2.0, n, device="cuda")).T.contiguous().T
    chunks, j = [], 0
    for i, w in enumerate(widths):
        buf = torch.full((w + 2, ld), float("nan"), device="cuda")
        buf[:w, :m] = A[:, j:j + w].T
        chunks.append(buf[:w, :m].T)
        j += w
    res = []
    for cols in (chunks, [_padded(A, ld)]):
        sk = IdSketch(m, n, 1, l, seed=11, prec=prec, want_Y=want_Y, window_cols=n)
        for c in cols:
            sk.stream_columns(c)
        W, Y, _ = sk.sketches()
        res.append((W.clone(), Y.clone() if want_Y else torch.zeros(1)))
        sk.close()
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    An = A.cpu().double().numpy()
    if prec == "bf16":
        An = A.to(torch.bfloat16).cpu().double().numpy()
    elif prec == "fp8":
        An, _ = ofp8.quantize_columns(An)
    Wo, Yo = oracle.sketch(An, oracle.psi(l, m, 11), oracle.omega(n, l, 11))
    assert rel(res[0][0].cpu().numpy(), Wo) <= 1e-5
    if want_Y:
        assert rel(res[0][1].cpu().double().numpy(), Yo) <= 1e-5


def _padded(A, ld):
    m, n = A.shape
    buf = torch.full((n, ld), float("nan"), device="cuda")
    buf[:, :m] = A.T
    return buf[:, :m].T
