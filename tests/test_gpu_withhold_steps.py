"""sff_debug_knn_withhold counts visits of 128 candidates, each visited twice: a step
of either pass makes the waits on it run out, a step past the last has no effect."""
import pytest

import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,visits", [(64, 40, 1), (136, 88, 2), (256, 80, 3)])
def test_steps_of_both_passes_and_past_the_last(w, h, visits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    m = sff.QuadMatcher(w, h)
    dev = [torch.as_tensor(im).cuda() for im in scenegen.random_images(w, h, seed=3, n=4)]
    sff.device_status(reset=True)
    try:
        for step, status in ((0, sff.ERR_TIMEOUT), (visits, sff.ERR_TIMEOUT), (2 * visits - 1, sff.ERR_TIMEOUT),
                             (2 * visits, sff.OK), (2 * visits + 1, sff.OK)):
            sff.debug_knn_withhold(step, wait_limit_us=20000)
            m.run(*dev, seed=5)
            assert sff.device_status(reset=True) == status, step
            assert sff.device_drain_timeouts() == 0, step
    finally:
        sff.debug_knn_withhold(-1, 0)
    m.run(*dev, seed=5)
    assert sff.device_status(reset=True) == sff.OK
    sff.device_timeouts(reset=True)
