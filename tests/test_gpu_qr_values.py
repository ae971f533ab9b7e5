"""J and P of the pivoted QRs at the edges of their forms, on data chosen for its
pivot margin (seeds are tried until the oracle's margin is met), so that J and P
are always compared: J equals the oracle's, and P both the oracle's and the
least-squares fit on the returned columns."""
import numpy as np
import pytest
import torch

import oracle
from margins import MARGIN, assert_valid_skeleton
from oracle import learned as L
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu

SEEDS = range(200)


def _data(m, n, seed, dtype):
    A = gaussian_matrix(m, n, seed=7919 * n + seed, dtype=dtype, device="cuda")
    return (A * torch.linspace(0.5, 2.0, n, dtype=dtype, device="cuda")).T.contiguous().T


def _fit_error(B, J, P, kout):
    """Largest distance of P from the least-squares fit of B on its columns J, as
    a share of the fit's scale."""
    assert_valid_skeleton(J, P, kout, B.shape[1])
    fit = np.linalg.lstsq(B[:, J[:kout]], B, rcond=None)[0]
    return np.max(np.abs(P[:kout] - fit)) / max(1.0, np.abs(fit).max())


def _compare(B, J, P, kout, ref, tol):
    Jo, Po, ko = ref[:3]
    J, P = J.cpu().numpy(), P.cpu().numpy()
    assert kout == ko and J.tolist() == np.asarray(Jo).tolist()
    assert np.max(np.abs(P - Po)) <= tol * max(1.0, np.abs(Po).max())
    assert _fit_error(B, J, P, kout) <= tol


def _handle(n, k, l, dtype, m, cols=None):
    """A handle whose W has a margin (among `cols` where given), W, the oracle's
    column ID of W(:, cols), and the data."""
    from paper_1905_13257_gb300 import IdSketch
    for seed in SEEDS:
        sk = IdSketch(m, n, k, l, seed=3, dtype=dtype, want_Y=False)
        A = _data(m, n, seed, dtype)
        sk.stream_columns(A)
        W = sk.sketches()[0].cpu().numpy().copy()
        ref = oracle.column_id(W if cols is None else W[:, cols], k)
        if ref[3] >= MARGIN:
            return sk, W, ref, A
        sk.close()
    raise AssertionError("no seed with a pivot margin")


@pytest.mark.parametrize("n,k,l", [(5, 5, 9), (128, 20, 33), (129, 20, 31), (256, 30, 64),
                                   (257, 64, 64), (512, 50, 60), (513, 17, 17), (1000, 50, 60),
                                   (1024, 3, 4), (1025, 20, 30)])
def test_small_qr_values(n, k, l):
    sk, W, ref, _ = _handle(n, k, l, torch.float64, 700)
    _compare(W, *sk.factor(), ref, 1e-9)
    sk.close()


@pytest.mark.parametrize("n,k,l", [(70, 65, 65), (129, 86, 96), (256, 70, 81), (257, 66, 96),
                                   (512, 80, 90), (512, 86, 96), (513, 30, 70)])
def test_wide_qr_values(n, k, l):
    sk, W, ref, _ = _handle(n, k, l, torch.float32, 1024)
    _compare(W, *sk.factor(), ref, 1e-9)
    sk.close()


@pytest.mark.parametrize("n,ncand,k,l", [(40, 12, 6, 16), (300, 90, 25, 40), (512, 100, 50, 60),
                                         (513, 64, 20, 33), (1024, 200, 40, 64)])
def test_restricted_qr_values(n, ncand, k, l):
    cand = np.random.default_rng(n).permutation(n)[:ncand]     # not in column order
    sk, W, _, _ = _handle(n, k, l, torch.float64, 700, cand)
    _compare(W, *sk.factor_restricted(cand), L.restricted_id(W, cand, k), 1e-9)
    sk.close()


@pytest.mark.parametrize("spec", [
    [(64, 10, 20), (128, 64, 64), (129, 20, 30), (300, 40, 50), (512, 50, 60), (200, 70, 80),
     (512, 86, 96), (8, 8, 8)],           # run after the work list, a cluster each
    [(100, 20, 30)] * 150])               # each in the CTA that completes its matrix
def test_batch_qr_values(spec):
    """Each problem's J equals that of the oracle for one handle's W (which differs
    from the batch's in FP32 summation order only); P within 1e-4 of its scale."""
    from paper_1905_13257_gb300 import IdBatch
    probs, refs, known = [], [], {}
    for n, k, l in spec:
        if (n, k, l) not in known:
            sk, W, ref, A = _handle(n, k, l, torch.float32, 2048)
            sk.close()
            known[(n, k, l)] = (dict(A=A, k=k, l=l, seed=3), W, ref)
        p, W, ref = known[(n, k, l)]
        probs.append(p)
        refs.append((W, ref))
    bt = IdBatch(probs)
    bt.run()
    for (W, ref), out in list(zip(refs, bt.wait()))[:20]:
        _compare(W, *out, ref, 1e-4)
    bt.close()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m,n,k", [(8, 5, 4), (129, 20, 7), (1537, 33, 32), (2049, 200, 20),
                                   (20001, 130, 12), (30000, 257, 5)])
@pytest.mark.parametrize("also_factor", [False, True])
def test_coarse_qr_values(dtype, m, n, k, also_factor):
    from paper_1905_13257_gb300 import IdSketch
    for seed in SEEDS:
        A = _data(m, n, seed, dtype)
        B = A.cpu().double().numpy()
        ref = oracle.column_id(B, k)
        if ref[3] >= MARGIN:
            break
    else:
        raise AssertionError("no seed with a pivot margin")
    sk = IdSketch(m, n, k, k, dtype=dtype, want_Y=False, grid=(1, 1, m), ncomp=1,
                  coarse_stride=(1, 1, 1), want_coarse=True)
    sk.stream_columns(A)
    if also_factor:
        sk.factor()          # starts the coarse QR on the side stream
    _compare(B, *sk.coarse_factor(), ref, 1e-8)
    sk.close()
