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


@pytest.mark.parametrize("m,n", [(64, 33), (64, 96), (127, 65)])
def test_small_fp32_error_pass_keeps_every_square(m, n):
    """FP32 data with fewer than 128 rows: every square goes into the compensated
    sums by itself.  A_hat = 1 everywhere, residuals 1 and 2^-12.5 in a pattern of
    which a chunk's plain FP32 sum loses up to 7 * 2^-25, always downwards.
    A compensated sum of positive terms is within 2^-25 (the rounding of x - c);
    numerator and denominator under the root: 2^-25 together."""
    from paper_1905_13257_gb300 import IdSketch
    A = np.full((m, n), 1.0 + 2.0 ** -12.5, dtype=np.float32)
    rows, cols = np.arange(m) % 64 < 16, np.arange(n) % 32 < 16
    A[np.ix_(rows, cols)] = 2.0
    A[:, n - 1] = 1.0                       # the skeleton column
    P = torch.ones((1, n), dtype=torch.float64)
    sk = IdSketch(m, n, 1, 1, dtype=torch.float32, want_Y=False)
    fro, _ = sk.reconstruct_error(torch.tensor(A.T.copy(), device="cuda").T,
                                  torch.tensor([n - 1]), P)
    sk.close()
    D = A - np.float32(1.0)                 # exact
    exact = np.sqrt((D * D).astype(np.float64).sum() / (A * A).astype(np.float64).sum())
    assert abs(fro - exact) <= 2.0 ** -25 * exact


@pytest.mark.parametrize("mc", [19, 31, 33, 63])
def test_coarse_products_across_lanes_in_fp64(mc):
    """FP32 A_c with an odd number of rows, one row per thread: the products are
    exact FP32 pairs, their sums FP64.  For a column almost orthogonal to the
    pivot, P's entry is a sum that cancels: within a few roundings (2^-51) of
    |a_p| |a_j| / |a_p|^2, where sums in FP32 pairs are off by 2^-48."""
    from paper_1905_13257_gb300 import IdSketch
    n = 40
    rng = np.random.default_rng(mc)
    p = rng.standard_normal(mc)
    A = rng.standard_normal((mc, n))
    A -= np.outer(p, p @ A) / (p @ p)
    A /= np.linalg.norm(A, axis=0)
    A[:, 7] = 3.0 * p / np.linalg.norm(p)
    A = A.astype(np.float32)
    sk = IdSketch(mc, n, 1, 1, dtype=torch.float32, want_Y=False, grid=(1, 1, mc), ncomp=1,
                  coarse_stride=(1, 1, 1), want_coarse=True)
    sk.stream_columns(torch.tensor(A.T.copy(), device="cuda").T)
    J, P, kout = sk.coarse_factor()
    sk.close()
    assert kout == 1 and int(J[0]) == 7
    L = A.astype(np.longdouble)
    exact = (L[:, 7] @ L) / (L[:, 7] @ L[:, 7])
    bound = np.linalg.norm(A, axis=0) / np.linalg.norm(A[:, 7]) * 2.0 ** -51
    off = np.abs(P[0].cpu().numpy() - exact.astype(np.float64)) / bound
    off[7] = 0.0
    assert off.max() <= 1.0
