"""The cooperative coarse QR over its forms: FP32 with whole row quads, FP32
with an odd number of coarse rows, FP64; one CTA to one per SM; a CTA's rows
one to 512; more columns of V than shared memory holds (77,824 x 70 at k = 64);
a rank that ends the steps early; norms that must be recomputed (columns that
lose more than 20 bits).  Against the oracle's column ID of the same A_c with
the repository's bar for P_c, 1e-8."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN, assert_valid_skeleton
from synthetic import gaussian_matrix, low_rank_matrix

pytestmark = pytest.mark.gpu


def _coarse(A, k, also_factor=False):
    """The sub-sampled ID at stride 1: A_c = A."""
    from paper_1905_13257_gb300 import IdSketch
    m, n = A.shape
    sk = IdSketch(m, n, k, k, dtype=A.dtype, want_Y=False, grid=(m, 1, 1), ncomp=1,
                  coarse_stride=(1, 1, 1), want_coarse=True)
    sk.stream_columns(A)
    if also_factor:   # starts the coarse QR beside the QR of W
        sk.factor()
    J, P, kout = sk.coarse_factor()
    out = J.cpu().numpy(), P.cpu().numpy(), kout
    sk.close()
    return out


def _check(A, k, **kw):
    J, P, kout = _coarse(A, k, **kw)
    Jo, Po, ko, margin = oracle.column_id(A.cpu().double().numpy(), k)
    assert kout == ko
    assert_valid_skeleton(J, P, kout, A.shape[1])
    if margin >= MARGIN:
        assert J.tolist() == Jo.tolist()
        assert np.max(np.abs(P - Po)) <= 1e-8 * max(1.0, np.abs(Po).max())


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m,n,k", [(8, 5, 4), (129, 20, 7), (1152, 96, 8), (1537, 33, 32),
                                   (2049, 200, 20), (20001, 130, 12), (30000, 257, 5)])
def test_coarse_forms(dtype, m, n, k):
    A = gaussian_matrix(m, n, seed=m + n, dtype=dtype, device="cuda")
    A = A * torch.linspace(0.5, 2.0, n, dtype=dtype, device="cuda")   # spread the norms
    A = A.T.contiguous().T
    _check(A, k)
    _check(A, k, also_factor=True)


def test_v_past_shared_memory():
    A = gaussian_matrix(77824, 70, seed=5, dtype=torch.float32, device="cuda")
    A = A * torch.linspace(0.5, 2.0, 70, dtype=torch.float32, device="cuda")
    _check(A.T.contiguous().T, 64)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m", [1200, 20003])
def test_recomputed_norms_and_early_stop(dtype, m):
    """Columns that are nearly combinations of a few large ones: after those
    pivots their norms have lost more than 20 bits and are recomputed; and an
    exactly rank-6 matrix stops after 6 steps (FP64)."""
    n = 60
    B = low_rank_matrix(m, n, 4, seed=3, dtype=torch.float64, device="cuda")
    E = gaussian_matrix(m, n, seed=4, dtype=torch.float64, device="cuda")
    E = E * torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")
    A = (B + 2e-5 * E).to(dtype).T.contiguous().T
    _check(A, 12)
    if dtype == torch.float64:
        R = low_rank_matrix(m, n, 6, seed=7, dtype=dtype, device="cuda").T.contiguous().T
        J, P, kout = _coarse(R, 12)
        Jo, Po, ko, _ = oracle.column_id(R.cpu().numpy(), 12)
        assert kout == ko == 6 and J[6:].tolist() == [-1] * 6
