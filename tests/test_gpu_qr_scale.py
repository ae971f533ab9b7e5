"""The pivoted QR of W where the squares of its columns' norms are near the ends
of FP64's range (denormal, or within a factor of two of overflow): J and P as
the oracle has them for W scaled to order one.  64 rows of A are one row tile of
the FP64 sketch, so that W's sums have one order."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def _factor(A, k, l, to_one):
    """J, P of A's sketch and the oracle's for the same W times `to_one`."""
    from paper_1905_13257_gb300 import IdSketch
    n = A.shape[1]
    sk = IdSketch(64, n, k, l, seed=3, dtype=torch.float64, want_Y=False)
    sk.stream_columns(A.T.contiguous().T)
    W = sk.sketches()[0].cpu().numpy() * to_one
    J, P, kout = sk.factor()
    sk.close()
    Jo, Po, ko, margin = oracle.column_id(W, k)
    assert kout == ko == k and margin >= MARGIN
    assert J.cpu().tolist() == Jo.tolist()
    # a denormal squared norm keeps 40 bits or more
    assert np.max(np.abs(P.cpu().numpy() - Po)) <= 1e-9 * max(1.0, np.abs(Po).max())


@pytest.mark.parametrize("n,k,l", [(100, 12, 30), (300, 12, 40), (600, 8, 60), (60, 20, 64)])
@pytest.mark.parametrize("exponent", [-521, -518, -500, 480])
def test_scaled_columns(n, k, l, exponent):
    A = gaussian_matrix(64, n, seed=n, dtype=torch.float64, device="cuda")
    A = A * torch.logspace(0, -1, n, base=2, dtype=torch.float64, device="cuda")
    _factor(A * 2.0 ** exponent, k, l, 2.0 ** -exponent)


@pytest.mark.parametrize("l", [2, 3, 5])
def test_norm_next_to_overflow(l):
    """One column with a squared norm of 0.97 times 2^1024, the others small."""
    from paper_1905_13257_gb300 import IdSketch
    n = 7
    A = gaussian_matrix(64, n, seed=l, dtype=torch.float64, device="cuda")
    A[:, 1:] *= 2.0 ** -20
    sk = IdSketch(64, n, 2, l, seed=3, dtype=torch.float64, want_Y=False)
    sk.stream_columns(A.T.contiguous().T)
    w0 = float(torch.linalg.norm(sk.sketches()[0][:, 0]))
    sk.close()
    _factor(A * (0.97 ** 0.5 / w0) * 2.0 ** 512, 2, l, 2.0 ** -512)
