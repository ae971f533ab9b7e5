"""The restricted ID of more columns than a cluster's registers hold (n > 1024):
the QR of the candidates (the cluster form up to 1024 of them, one CTA past
that), its reflectors applied to all columns.  Data seeds with a pivot margin:
J is the oracle's, and P both the oracle's and the least-squares fit of W on
W(:, J) (1e-9, as the other forms)."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN, assert_valid_skeleton
from oracle import learned as L
from synthetic import gaussian_matrix, low_rank_matrix

pytestmark = pytest.mark.gpu


def _sketch(n, k, l, cand, m=700):
    """A handle whose W has a margin among the candidates, and W."""
    from paper_1905_13257_gb300 import IdSketch
    for seed in range(60):
        A = gaussian_matrix(m, n, seed=1000 * n + seed, dtype=torch.float64, device="cuda")
        A = A * torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")
        sk = IdSketch(m, n, k, l, seed=3, dtype=torch.float64, want_Y=False)
        sk.stream_columns(A.T.contiguous().T)
        W = sk.sketches()[0].cpu().numpy().copy()
        if oracle.column_id(W[:, cand], k)[3] >= MARGIN:
            return sk, W
        sk.close()
    raise AssertionError("no seed with a pivot margin")


def _check_fit(W, J, P, kout):
    assert_valid_skeleton(J, P, kout, W.shape[1])
    j = np.asarray(J)[:kout]
    fit = np.linalg.lstsq(W[:, j], W, rcond=None)[0]
    assert np.max(np.abs(P[:kout] - fit)) <= 1e-9 * max(1.0, np.abs(fit).max())


@pytest.mark.parametrize("n,ncand,k,l", [(1025, 1, 1, 1), (1025, 30, 7, 17), (1030, 64, 20, 64),
                                         (2000, 100, 50, 60), (3001, 513, 16, 33),
                                         (1500, 1024, 12, 31), (1400, 1025, 9, 20),
                                         (4096, 4096, 5, 15), (20000, 40, 30, 48)])
def test_restricted_to_columns(n, ncand, k, l):
    cand = np.random.default_rng(n + ncand).permutation(n)[:ncand]   # not in column order
    sk, W = _sketch(n, k, l, cand)
    J, P, kout = sk.factor_restricted(cand)
    sk.close()
    J, P = J.cpu().numpy(), P.cpu().numpy()
    Jo, Po, ko = L.restricted_id(W, cand, k)
    assert kout == ko == k and J.tolist() == list(Jo)
    assert np.max(np.abs(P - Po)) <= 1e-9 * max(1.0, np.abs(Po).max())
    _check_fit(W, J, P, kout)


@pytest.mark.parametrize("ncand", [50, 1100])
def test_rank_deficient_candidates_and_ties(ncand):
    """Candidates of rank 3, the first and the last equal: 3 pivots, -1 past them,
    zero rows of P; the earlier of the equal candidates may be a pivot, the later
    not.  64 rows are one row tile of the FP64 sketch: equal columns of A give
    bit-equal columns of W."""
    from paper_1905_13257_gb300 import IdSketch
    n, k, l = 1300, 10, 20
    A = gaussian_matrix(64, n, seed=5, dtype=torch.float64, device="cuda").T.contiguous().T
    cand = np.random.default_rng(ncand).permutation(n)[:ncand]
    A[:, cand.tolist()] = low_rank_matrix(64, ncand, 3, seed=2, dtype=torch.float64, device="cuda")
    A[:, int(cand[0])] *= 10.0
    A[:, int(cand[-1])] = A[:, int(cand[0])]
    sk = IdSketch(64, n, k, l, seed=3, dtype=torch.float64, want_Y=False)
    sk.stream_columns(A)
    W = sk.sketches()[0].cpu().numpy().copy()
    J, P, kout = sk.factor_restricted(cand)
    sk.close()
    J, P = J.cpu().numpy(), P.cpu().numpy()
    assert kout == 3 and J[0] == cand[0] and cand[-1] not in J and J[3:].tolist() == [-1] * 7
    assert not P[3:].any()
    _check_fit(W, J, P, kout)
