"""The sweep's bounded wait is answered by the warp as one: if a single lane gives up, all of its lanes take the
timeout (the code behind it is warp-wide), and the device context stays usable."""
import pytest

pytestmark = pytest.mark.gpu


def test_one_lane_giving_up_is_a_timeout_of_the_warp():
    import __graft_entry__ as g
    g.build()
    from paper_1608_04601_gb300 import pic, _native as NV
    assert pic.debug_wait(2, 4096) == -4          # PIC_ERR_TIMEOUT
    assert pic.debug_wait(True, 4096) == NV.PIC_OK
    assert pic.debug_wait(False, 64) == -4
