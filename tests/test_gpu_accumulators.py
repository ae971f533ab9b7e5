"""Sums that must not be held in fewer bits than their inputs need."""
import numpy as np
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def test_unaligned_sketch_sums_past_fp32_range():
    """W of FP32 data on the CUDA-core path accumulates in FP64: sums of 40,000
    finite entries past 3.4e38 stay finite.  Every row block's own sum stays in
    FP32's range; 64-row sums carry 24 bits, so 1e-5 as elsewhere."""
    import oracle
    from paper_1905_13257_gb300 import IdSketch
    m, n, l = 64 * 152 * 4 + 1, 3, 4
    P = oracle.psi(l, m, 7)
    A = np.empty((m, n), dtype=np.float32)
    for j in range(n):
        A[:, j] = 3e36 * np.sign(P[j])
    sk = IdSketch(m, n, 1, l, seed=7, dtype=torch.float32, want_Y=False)
    sk.stream_columns(torch.tensor(A.T.copy(), device="cuda").T)    # odd m: unaligned columns
    W = sk.sketches()[0].cpu().numpy()
    sk.close()
    Wo = P @ A.astype(np.float64)
    assert np.abs(Wo).max() > 4e40
    assert np.max(np.abs(W - Wo)) <= 1e-5 * np.abs(Wo).max()
