"""The coarse rows A_c of a window against the oracle's sub-sampling (exact
copies), where a thread copies several columns and where it copies one: column
counts around the group of eight, a window of several buffers, strides of 1 to
3, a last block of few rows."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,ncomp,stride,widths", [
    ((8, 6, 10), 1, (2, 2, 2), [9]), ((64, 33, 31), 3, (1, 1, 1), [16]),
    ((64, 33, 31), 3, (1, 2, 1), [20, 9]), ((96, 80, 72), 1, (2, 1, 1), [7, 6]),
    ((128, 65, 63), 2, (3, 1, 2), [8, 1, 24])])
def test_coarse_rows(grid, ncomp, stride, widths):
    from paper_1905_13257_gb300 import IdSketch
    m, n = int(np.prod(grid)) * ncomp, sum(widths)
    A = gaussian_matrix(m, n, seed=m, dtype=torch.float32, device="cuda").T.contiguous().T
    sk = IdSketch(m, n, 1, 10, grid=grid, ncomp=ncomp, coarse_stride=stride, want_coarse=True,
                  window_cols=n)
    j = 0
    for w in widths:
        sk.stream_columns(A[:, j:j + w].T.clone().T)
        j += w
    Ac = sk.sketches()[2].cpu().numpy()
    rows = oracle.coarse_rows(grid, ncomp, stride)
    assert np.array_equal(Ac, A.cpu().numpy()[rows])
