"""The cooperative coarse QR of FP64 data at 2, 3 to 6, 7, 8 and 9 to 13 rows per
lane (its instantiations by the rows of a CTA): columns with well-separated
norms, so that J is the oracle's; P within 1e-8 (the reflectors are FP32 pairs)."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(7001, 150, 6), (16500, 90, 5), (24003, 60, 5), (33000, 70, 4),
                                   (36300, 40, 4), (41000, 50, 4), (58001, 40, 3), (64000, 33, 3)])
def test_fp64_rows_per_lane(m, n, k):
    from paper_1905_13257_gb300 import IdSketch
    A = gaussian_matrix(m, n, seed=m, dtype=torch.float64, device="cuda")
    A = (A * torch.logspace(0, -1.5, n, dtype=torch.float64, device="cuda")).T.contiguous().T
    sk = IdSketch(m, n, k, k, dtype=torch.float64, want_Y=False, grid=(1, 1, m), ncomp=1,
                  coarse_stride=(1, 1, 1), want_coarse=True)
    sk.stream_columns(A)
    J, P, kout = sk.coarse_factor()
    sk.close()
    Jo, Po, ko, margin = oracle.column_id(A.cpu().numpy(), k)
    assert margin >= MARGIN and kout == ko == k and J.tolist() == Jo.tolist()
    assert np.max(np.abs(P.cpu().numpy() - Po)) <= 1e-8 * max(1.0, np.abs(Po).max())
