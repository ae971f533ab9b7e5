"""The FP8 form's per-column scales at the edges of their row split (eighths of
the row quads, loads of eight at a time, up to three rows past the last quad):
one entry decides each column's scale, at every place where the split could
lose it.  W against the oracle's products of the dequantised matrix (1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import fp8 as ofp8
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [128, 131, 1030, 65537, 70000])
def test_one_entry_decides_the_scale(m):
    from paper_1905_13257_gb300 import IdSketch
    q = m // 4
    rows = [0, 3, m - 1, m - 2, 4 * q - 1, 4 * (q // 8), 4 * (q // 8) - 1, 4 * (7 * q // 8),
            4 * (q // 2) + 1, min(m - 1, 8 * 1024), min(m - 1, 8 * 1024 + 1), m // 3]
    n, ld = len(rows) + 1, (m + 3) // 4 * 4
    buf = torch.zeros((n, ld), dtype=torch.float32, device="cuda")
    A = buf[:, :m].T
    A.copy_(gaussian_matrix(m, n, seed=m, dtype=torch.float32, device="cuda"))
    for c, r in enumerate(rows):
        A[r, c] = -3000.0 * (c + 1)
    A[:, n - 1] = 0.0
    sk = IdSketch(m, n, 1, 12, seed=3, prec="fp8", want_Y=False)
    sk.stream_columns(A)
    W = sk.sketches()[0].cpu().numpy()
    Aq, _ = ofp8.quantize_columns(A.cpu().double().numpy())
    Wo = oracle.psi(12, m, 3) @ Aq
    for c in range(n - 1):
        assert np.linalg.norm(W[:, c] - Wo[:, c]) <= 1e-5 * np.linalg.norm(Wo[:, c]), (c, rows[c])
    assert not W[:, n - 1].any()
    sk.close()
