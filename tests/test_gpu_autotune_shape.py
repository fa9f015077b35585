"""haru_autotune keeps the launch shape that it timed: the planner's schedule
(units_target 0) runs only without an explicit CTA count, so a context with
one must not keep the first and the second together."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_schedule_is_kept_without_a_cta_count():
    import numpy as np

    import paper_2211_07340_gb300 as haru
    haru.build_library()
    ref = synth.random_signal(60000, seed=3)
    off = np.array([0, 250], np.uint32)  # one query: the schedule cuts it finer than any queue shape, and wins
    ev = synth.random_signal(int(off[-1]), seed=4)
    with haru.Context(ctas_per_sm=1) as ctx:
        ctx.ref_load(ref)
        before = ctx.sdtw_batch(haru.HARU_FP32, ev, off)
        chosen = ctx.autotune(haru.HARU_FP32, ev, off)
        assert chosen["units_target"] == 0
        assert ctx.config.ctas_per_sm == 0
        after = ctx.sdtw_batch(haru.HARU_FP32, ev, off)
        np.testing.assert_array_equal(before[0], after[0])
        np.testing.assert_array_equal(before[1], after[1])
