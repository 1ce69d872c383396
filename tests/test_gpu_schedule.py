"""Which launches the library's own schedule takes, read from the per-kernel record:
a fused scale is one launch of all its iterations."""
import pytest

import scenegen

pytestmark = pytest.mark.gpu


def _fused_scales(w, h, tuning=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_10096_gb300 as sff
    sff.build()
    m = sff.QuadMatcher(w, h, tuning=tuning)
    dev = [torch.as_tensor(im).cuda() for im in scenegen.random_images(w, h, seed=w, n=4)]
    sff.profile_enable(True)
    try:
        m.run(*dev, seed=1)
        torch.cuda.synchronize()
        prof = sff.profile_collect(with_units=True)
    finally:
        sff.profile_enable(False)
    times = {int(k.rpartition("/s")[2]): v for k, v in prof.items() if k.startswith("k_iteration/s")}
    assert sorted(times) == [0, 1, 2, 3] and all(t[2] == m.params.iterations for t in times.values())
    return {s for s, t in times.items() if t[0] == 1}


@pytest.mark.parametrize("w,h,fused", [
    (256, 80, {1, 2, 3}),   # 67 points a SM at scale 1
    (360, 120, {2, 3}),     # 142 at scale 1: more tiles than SMs
    (432, 136, set()),      # 773 a SM at scale 0: a stage that runs beside others
    (900, 300, set()),
])
def test_fused_scales_leave_room_for_other_streams(w, h, fused):
    assert _fused_scales(w, h) == fused


@pytest.mark.parametrize("field,value,fused", [
    ("overlap", 0, {1, 2, 3}), ("features_form", 1, {1, 2, 3}), ("features_form", 2, {1, 2, 3}),
    # fields of the iterations: their setting as given
    ("group_mb", 64, set()), ("pair_fields", 1, set()), ("alternate_order", 1, set()), ("pdl", 1, set()),
])
def test_only_iteration_fields_end_the_derived_schedule(field, value, fused):
    import paper_1710_10096_gb300 as sff
    sff.build()
    t = sff.default_tuning()
    setattr(t, field, value)
    assert _fused_scales(256, 80, t) == fused


def test_a_coarse_entry_makes_the_default_values_explicit():
    import paper_1710_10096_gb300 as sff
    sff.build()
    assert _fused_scales(256, 80, sff.make_tuning(1, 32, 16, 0, [(1, 0, 32, 16)])) == set()
