"""The streamed row passes of the coarse QR over many steps (u's low part, which
only the sums' low parts take, grows with them): eight runs give the same bits,
and P the least-squares fit on the returned columns (1e-10: pairs of FP32 carry
48 bits)."""
import numpy as np
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def test_streamed_passes_over_many_steps():
    from paper_1905_13257_gb300 import IdSketch
    m, n, k = 4 * 41 * 700, 90, 24
    A = gaussian_matrix(m, n, seed=9, dtype=torch.float32, device="cuda")
    A = (A * torch.logspace(0, -2, n, device="cuda")).T.contiguous().T
    sk = IdSketch(m, n, k, k, seed=2, grid=(4, 41, 700), ncomp=1, coarse_stride=(1, 1, 1),
                  want_coarse=True, want_Y=False)
    sk.stream_columns(A)
    J, P, kout = sk.coarse_factor()
    assert kout == k
    for _ in range(7):
        J1, P1, _ = sk.coarse_factor()
        assert torch.equal(J, J1) and torch.equal(P, P1)
    sk.close()
    An, j = A.cpu().double().numpy(), J.cpu().numpy()
    fit = np.linalg.lstsq(An[:, j], An, rcond=None)[0]
    assert np.max(np.abs(P.cpu().numpy() - fit)) <= 1e-10 * max(1.0, np.abs(fit).max())
