"""After a bounded wait that gave up, a kernel drains what is still in flight before it frees its buffers: the drain
must wait for the phase that did not complete, not return at once on the one before."""
import pytest

from gpu_util import hyb_module, need_gpu

pytestmark = pytest.mark.gpu


def test_drain_waits_for_the_phase_that_gave_up():
    need_gpu()
    hyb = hyb_module()
    assert hyb.hyb_wait_selftest(1, 0.05) == hyb.HYB_ETIMEOUT, hyb.hyb_last_error()
