"""Repeated error passes over the same data give the same bits (every sum has a
fixed order): the epilogue hands a ring stage back only when its reads have
returned.  Column counts around the 128-column halves, ragged last row block,
more row blocks than the ring holds boxes; also the single-pass form."""
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(200003, 512, 50), (300000, 256, 8), (150001, 37, 30)])
def test_error_pass_repeats(m, n, k):
    from paper_1905_13257_gb300 import IdSketch
    ld = (m + 3) // 4 * 4
    buf = torch.zeros((n, ld), device="cuda")
    buf[:, :m] = gaussian_matrix(m, n, seed=m, dtype=torch.float32, device="cuda").T
    A = buf[:, :m].T
    sk = IdSketch(m, n, k, k, seed=3)
    sk.stream_columns(A)
    J, P, _ = sk.factor()
    got = {sk.reconstruct_error(A, J, P) for _ in range(30)}
    assert len(got) == 1


def test_single_pass_error_repeats():
    from paper_1905_13257_gb300 import IdSketch
    grid, n, k = (64, 32, 64), 300, 20
    m = 64 * 32 * 64
    A = gaussian_matrix(m, n, seed=5, dtype=torch.float32, device="cuda").T.contiguous().T
    sk = IdSketch(m, n, k, k, seed=3, grid=grid, ncomp=1, coarse_stride=(2, 2, 2),
                  want_coarse=True)
    sk.stream_columns(A)
    Jc, Pc, _ = sk.coarse_factor()
    ax = [torch.arange(g, dtype=torch.float64).numpy() for g in grid]
    sk.set_mesh(*ax, (0.0, 0.0, 0.0))
    got = {sk.single_pass_error(A, Jc, Pc) for _ in range(30)}
    assert len(got) == 1
