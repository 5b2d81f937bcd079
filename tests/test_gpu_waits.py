"""The bounded wait that the TMA and tcgen05 kernels share, by whole warps: what it answers, and which flags it raises."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cluster_form", [False, True])
def test_a_wait_runs_out_once_and_the_cta_drains(cluster_form):
    import paper_2505_01068_b200 as g
    assert g.last_device_status() == (0, 0)
    answers, flags = g.wait_answers(cluster_form)
    assert answers[:, 0].eq(1).all()   # a phase that is over, also after the CTA has given up
    assert answers[:, 1].eq(0).all()   # one that never will be: in all lanes of both warps
    assert flags == [g.DEVFLAG_TIMEOUT, 0]   # the second warp left because the first had run out, not by running out itself
    assert g.last_device_status() == (0, 0)
    g.expire_wait_selftest()           # the same kernel on the library's own status word
    code, raised = g.last_device_status()
    assert (code, raised) == (5, g.DEVFLAG_TIMEOUT)
    assert g.last_device_status() == (0, 0)
