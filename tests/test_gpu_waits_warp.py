"""A warp's bounded wait gives all lanes one answer, also when the phase has
completed for some of them: no lane goes on alone into a full-mask vote."""
import pytest

pytestmark = pytest.mark.gpu

ID_OK, ID_ERR_TIMEOUT = 0, 6


@pytest.mark.parametrize("mode,expected", [(4, ID_ERR_TIMEOUT), (5, ID_OK)])
def test_warp_wait_gives_up_as_one(mode, expected):
    from paper_1905_13257_gb300 import check_wait
    assert check_wait(mode) == expected
