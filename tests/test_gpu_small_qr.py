"""The pivoted QR of the small sketch and the solve for P at the edges of its
forms: columns per lane group (n = 128, 256, 512, 1024 on 8 CTAs), one column
past each, n below the cluster's CTAs, l not a multiple of the lane groups,
k = l, against the oracle's column ID of the same W; and the form restricted
to candidates in an order of the caller's own."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN, assert_valid_skeleton
from oracle import learned as L
from synthetic import gaussian_matrix, low_rank_matrix

pytestmark = pytest.mark.gpu


def _handle(n, k, l, seed=3, m=700):
    from paper_1905_13257_gb300 import IdSketch
    A = gaussian_matrix(m, n, seed=n + l, dtype=torch.float64, device="cuda")
    A = A * torch.linspace(0.5, 2.0, n, dtype=torch.float64, device="cuda")   # spread the norms
    sk = IdSketch(m, n, k, l, seed=seed, dtype=torch.float64, want_Y=False)
    sk.stream_columns(A.T.contiguous().T)
    return sk, sk.sketches()[0].cpu().numpy().copy()


def _check(J, P, kout, Jo, Po, ko, margin, n):
    assert kout == ko
    J, P = J.cpu().numpy(), P.cpu().numpy()
    assert_valid_skeleton(J, P, kout, n)
    if margin >= MARGIN:
        assert J.tolist() == Jo.tolist()
        assert np.max(np.abs(P - Po)) <= 1e-9 * max(1.0, np.abs(Po).max())


@pytest.mark.parametrize("n,k,l", [(5, 5, 9), (96, 8, 16), (128, 20, 33), (129, 20, 31),
                                   (256, 30, 64), (257, 64, 64), (512, 50, 60), (513, 17, 17),
                                   (1000, 50, 60), (1024, 3, 4), (1025, 20, 30)])
def test_small_qr_forms(n, k, l):
    sk, W = _handle(n, k, l)
    _check(*sk.factor(), *oracle.column_id(W, k), n)
    sk.close()


@pytest.mark.parametrize("n,k,l", [(70, 65, 65), (128, 80, 90), (129, 86, 96), (256, 70, 81),
                                   (257, 66, 96), (512, 80, 90), (513, 30, 70)])
def test_wide_qr_forms(n, k, l):
    """65 to 96 rows (FP32 data without Y): the cluster up to 512 columns, one
    CTA past them."""
    from paper_1905_13257_gb300 import IdSketch
    A = gaussian_matrix(1024, n, seed=n + l, dtype=torch.float32, device="cuda")
    A = A * torch.linspace(0.5, 2.0, n, dtype=torch.float32, device="cuda")
    sk = IdSketch(1024, n, k, l, seed=3, dtype=torch.float32, want_Y=False)
    sk.stream_columns(A.T.contiguous().T)
    W = sk.sketches()[0].cpu().numpy().copy()
    _check(*sk.factor(), *oracle.column_id(W, k), n)
    sk.close()


@pytest.mark.parametrize("spec", [
    # long QRs: run after the work list, a cluster each
    [(64, 10, 20), (128, 64, 64), (129, 20, 30), (300, 40, 50), (512, 50, 60), (200, 70, 80),
     (512, 86, 96), (8, 8, 8)],
    # short QRs: each in the CTA that completes its matrix
    [(64, 3, 13), (200, 5, 15), (512, 4, 80), (8, 8, 8)]])
def test_batch_qr_forms(spec):
    """The batch's QRs over their forms in one run: each problem's J and P
    equal those of one handle (whose W differs in FP32 summation order only,
    so P within 1e-4 of its scale, J at the oracle's margin)."""
    from paper_1905_13257_gb300 import IdBatch, IdSketch
    probs = []
    for n, k, l in spec:
        A = gaussian_matrix(2048, n, seed=n + l, dtype=torch.float32, device="cuda")
        A = A * torch.linspace(0.5, 2.0, n, dtype=torch.float32, device="cuda")
        probs.append(dict(A=A.T.contiguous().T, k=k, l=l, seed=n))
    bt = IdBatch(probs)
    bt.run()
    out = bt.wait()
    for p, (J, P, kout) in zip(probs, out):
        n = p["A"].shape[1]
        sk = IdSketch(2048, n, p["k"], p["l"], seed=p["seed"], want_Y=False)
        sk.stream_columns(p["A"])
        J1, P1, k1 = sk.factor()
        margin = oracle.column_id(sk.sketches()[0].cpu().numpy(), p["k"])[3]
        assert kout == k1 == p["k"]
        assert_valid_skeleton(J.cpu().numpy(), P.cpu().numpy(), kout, n)
        if margin >= MARGIN:
            assert torch.equal(J, J1)
            assert (P - P1).abs().max().item() <= 1e-4 * max(1.0, P1.abs().max().item())
        sk.close()
    bt.close()


@pytest.mark.parametrize("n,ncand,k,l", [(40, 12, 6, 16), (300, 90, 25, 40), (512, 100, 50, 60),
                                         (1100, 64, 20, 30)])
def test_restricted_qr_forms(n, ncand, k, l):
    sk, W = _handle(n, k, l)
    cand = np.random.default_rng(n).permutation(n)[:ncand]     # not in column order
    J, P, kout = sk.factor_restricted(cand)
    Jo, Po, ko = L.restricted_id(W, cand, k)
    margin = oracle.column_id(W[:, cand], k)[3]
    _check(J, P, kout, np.asarray(Jo), Po, ko, margin, n)
    sk.close()


def test_equal_columns_tie_to_the_first():
    """Duplicated columns have bit-equal norms: the lower index (or, among
    candidates, the earlier candidate) is the pivot.  64 rows are one row tile
    of the FP64 sketch, so that equal columns of A give bit-equal columns of W
    (several tiles add to W in no fixed order)."""
    from paper_1905_13257_gb300 import IdSketch
    B = low_rank_matrix(64, 6, 6, seed=2, dtype=torch.float64, device="cuda")
    A = torch.cat([B, B, B], 1)
    sk = IdSketch(64, 18, 6, 12, dtype=torch.float64, want_Y=False)
    sk.stream_columns(A.T.contiguous().T)
    W = sk.sketches()[0]
    assert torch.equal(W[:, :6], W[:, 6:12]) and torch.equal(W[:, :6], W[:, 12:])
    J, P, k = sk.factor()
    assert k == 6 and sorted(J.tolist()) == list(range(6))
    cand = list(range(12, 18)) + list(range(6))
    J, P, k = sk.factor_restricted(cand)
    assert k == 6 and sorted(J.tolist()) == list(range(12, 18))
    sk.close()
