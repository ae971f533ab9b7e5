"""The CUDA-core error pass (FP64 data, and FP32 data with fewer than 128 rows)
at the edges of its row groups and column chunks, against the oracle:
FP64 within 1e-10 relative; FP32 within 1e-4 relative plus 2e-6 (the
repository's bars)."""
import numpy as np
import pytest
import torch

import oracle
from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (15, 33, 3), (16, 32, 2), (17, 31, 5), (64, 65, 7),
                                   (127, 16, 16), (2433, 47, 20), (19457, 100, 64),
                                   (40000, 33, 9)])
def test_recon_forms(dtype, m, n, k):
    from paper_1905_13257_gb300 import IdSketch
    if dtype == torch.float32 and m >= 128:
        m = 100 + m % 28
    A = gaussian_matrix(m, n, seed=m + n, dtype=dtype, device="cuda")
    if m * n > 1:   # (the oracle divides by ||A||: not a zero matrix)
        A[m // 2, n // 2] = 0.0
    rng = np.random.default_rng(m)
    J = rng.choice(n, k, replace=False)
    P = 0.2 * rng.standard_normal((k, n))
    P[:, J] = np.eye(k)
    sk = IdSketch(m, n, k, k, dtype=dtype, want_Y=False)
    fro, mx = sk.reconstruct_error(A, torch.tensor(J), torch.tensor(P))
    fo, mo = oracle.recon_error(A.cpu().double().numpy(), J, P)
    rt, at = (1e-10, 1e-12) if dtype == torch.float64 else (1e-4, 2e-6)
    assert abs(fro - fo) <= rt * fo + at
    assert abs(mx - mo) <= rt * mo + at
    sk.close()
