"""The lift's two forms (a fine row per thread, and lines through shared memory)
around the rule that chooses between them, on one grid each: every k's S is the
oracle's interpolation (1e-6 FP32, 1e-13 FP64) and, on the coarse points, A_c."""
import numpy as np
import pytest
import torch

import oracle.single_pass as osp
from oracle import coarse_rows
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1e-6), (torch.float64, 1e-13)])
@pytest.mark.parametrize("grid,stride,periodic", [
    ((1, 7, 9), (1, 2, 2), False), ((3, 6, 11), (2, 1, 4), True), ((8, 5, 9), (2, 2, 2), False),
    ((16, 6, 7), (4, 3, 2), True), ((24, 5, 6), (2, 2, 2), False), ((33, 4, 5), (4, 2, 3), True),
    ((130, 3, 4), (2, 2, 2), False)])
def test_both_forms_of_a_grid(dtype, tol, grid, stride, periodic):
    from paper_1905_13257_gb300 import IdSketch
    nc, n = 2, 64
    m = nc * grid[0] * grid[1] * grid[2]
    A = gaussian_matrix(m, n, seed=m, dtype=dtype, device="cuda")
    sk = IdSketch(m, n, n, n, dtype=dtype, want_Y=False, grid=grid, ncomp=nc,
                  coarse_stride=stride, want_coarse=True)
    sk.stream_columns(A)
    coords = [np.cumsum(0.5 + np.random.default_rng(d).random(g)) for d, g in enumerate(grid)]
    per = tuple(float(c[-1] - c[0] + 0.7) if periodic else 0.0 for c in coords)
    sk.set_mesh(*coords, per)
    rows = coarse_rows(grid, nc, stride)
    An = A.cpu().double().numpy()
    So = osp.coarse_to_fine(grid, nc, stride, coords, per) @ An[rows]
    for k in (1, 3, 4, 7, 8, 15, 24, 31, 40, 64):
        J = torch.arange(k, dtype=torch.int32).flip(0)
        S = sk.single_pass_lift(J).cpu().double().numpy()
        ref = So[:, J.numpy()]
        assert np.linalg.norm(S - ref) <= tol * np.linalg.norm(ref)
        assert np.array_equal(S[rows], An[rows][:, J.numpy()])
    sk.close()
