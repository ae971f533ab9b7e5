"""The coarse QR of grids with more rows than the cooperative launch holds (a
ring of bulk copies feeds the row passes): five runs give the same bits, and the
oracle's column ID of the same A_c (P 1e-6: FP32 data, well-separated pivots)."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,n,k", [((64, 64, 48), 70, 8), ((100, 41, 50), 33, 5)])
def test_large_coarse_grid_repeats(grid, n, k):
    from paper_1905_13257_gb300 import IdSketch
    m = int(np.prod(grid))
    A = gaussian_matrix(m, n, seed=m, dtype=torch.float32, device="cuda")
    A = (A * torch.logspace(0, -1.5, n, device="cuda")).T.contiguous().T
    sk = IdSketch(m, n, k, k, seed=2, grid=grid, ncomp=1, coarse_stride=(1, 1, 1),
                  want_coarse=True, want_Y=False)
    got = []
    for _ in range(5):
        sk.reset()
        sk.stream_columns(A)
        J, P, _ = sk.coarse_factor()
        got.append((J.cpu().numpy().copy(), P.cpu().numpy().copy()))
    for J, P in got[1:]:
        assert np.array_equal(J, got[0][0]) and np.array_equal(P, got[0][1])
    Jo, Po, ko, _ = oracle.column_id(A.cpu().double().numpy(), k)
    assert ko == k and np.array_equal(got[0][0][:k], Jo[:k])
    assert np.linalg.norm(got[0][1] - Po) / np.linalg.norm(Po) <= 1e-6
