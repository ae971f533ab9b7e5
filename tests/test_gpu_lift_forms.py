"""The lifted skeleton M A_c(:, J_c) at the edges of its x segments (128 fine
points): one segment, one past it, a last coarse point at a segment's end,
wrapping and extrapolating ends, strides up to the whole line, a single coarse
point; against the oracle's interpolation (1e-6 FP32, 1e-13 FP64) and, on the
coarse points, exactly A_c."""
import numpy as np
import pytest
import torch

import oracle.single_pass as osp
from oracle import coarse_rows
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1e-6), (torch.float64, 1e-13)])
@pytest.mark.parametrize("grid,nc,stride,k,periodic", [
    ((128, 3, 4), 1, (4, 2, 3), 5, True), ((129, 3, 2), 2, (4, 1, 2), 3, True),
    ((129, 2, 3), 1, (4, 2, 2), 9, False), ((130, 3, 3), 1, (2, 2, 2), 33, False),
    ((257, 2, 2), 1, (128, 1, 1), 2, False), ((300, 2, 2), 1, (7, 2, 1), 40, True),
    ((6, 5, 7), 3, (10, 2, 3), 7, False), ((1, 9, 150), 1, (1, 3, 4), 4, True),
    ((40, 4, 4), 1, (1, 1, 1), 64, True)])
def test_lift_forms(dtype, tol, grid, nc, stride, k, periodic):
    from paper_1905_13257_gb300 import IdSketch
    m, n = nc * grid[0] * grid[1] * grid[2], k + 3
    A = gaussian_matrix(m, n, seed=m + k, dtype=dtype, device="cuda")
    sk = IdSketch(m, n, k, k, dtype=dtype, want_Y=False, grid=grid, ncomp=nc,
                  coarse_stride=stride, want_coarse=True)
    sk.stream_columns(A)
    coords = [np.cumsum(0.5 + np.random.default_rng(d).random(g)) for d, g in enumerate(grid)]
    per = tuple(float(c[-1] - c[0] + 0.7) if periodic else 0.0 for c in coords)
    sk.set_mesh(*coords, per)
    J = torch.arange(k, dtype=torch.int32).flip(0)
    S = sk.single_pass_lift(J).cpu().double().numpy()
    rows = coarse_rows(grid, nc, stride)
    An = A.cpu().double().numpy()
    So = osp.coarse_to_fine(grid, nc, stride, coords, per) @ An[rows][:, J.numpy()]
    assert np.linalg.norm(S - So) <= tol * np.linalg.norm(So)
    assert np.max(np.abs(S - So)) <= 8 * tol * np.abs(So).max()
    assert np.array_equal(S[rows], An[rows][:, J.numpy()])
    sk.close()
