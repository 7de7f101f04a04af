"""The bounded wait of a warp has one outcome: the code after it shuffles and
stores as a warp, so lanes must not leave it one by one, and a wait that ran
out in any lane must be reported."""
import pytest

from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("short", [0, 1, 1 << 31, 1 << 13, 0xfffffffe, 0xffffffff])
def test_a_warp_goes_on_together_or_reports_the_timeout(short):
    rc, on = B.selftest_warp_wait(short)
    assert (rc, on) == ((B.MLSW_OK, 0xffffffff) if short == 0 else (B.MLSW_ERR_TIMEOUT, 0))
    assert B.selftest_warp_wait(0)[0] == B.MLSW_OK  # the context stays usable
