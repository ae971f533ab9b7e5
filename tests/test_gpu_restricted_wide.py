"""The restricted ID of a handle with 64 < l <= 96 is refused as unsupported,
before any work: the handle stays usable and no CUDA error is recorded."""
import pytest
import torch

from synthetic import gaussian_matrix

pytestmark = pytest.mark.gpu


def test_wide_handle_refuses_candidates_and_goes_on():
    from paper_1905_13257_gb300 import IdError, IdSketch
    from paper_1905_13257_gb300 import _binding as B
    A = gaussian_matrix(1024, 200, seed=1, dtype=torch.float32, device="cuda")
    sk = IdSketch(1024, 200, 70, 80, seed=3, dtype=torch.float32, want_Y=False)
    sk.stream_columns(A)
    with pytest.raises(IdError) as e:
        sk.factor_restricted(list(range(150)))
    assert e.value.status == B.ID_ERR_UNSUPPORTED
    J, P, kout = sk.factor()
    assert kout == 70 and bool(torch.isfinite(P).all())
    sk.close()
