"""Loading or building a reference leaves the words of the batches alone: the
counters of the batch before it (which a batch still queued on a caller's
stream would be using) and its status."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def test_reference_keeps_batch_words(haru):
    ref = synth.random_signal(9001, seed=3)
    off = np.arange(0, 41 * 100, 100, dtype=np.uint32)
    ev = synth.random_signal(int(off[-1]), seed=4)
    rng = np.random.default_rng(5)
    with haru.Context(units_target=500) as ctx:
        ctx.ref_load(ref)
        assert ctx.last_status() == haru.HARU_OK and not any(ctx.last_stats().values())  # no batch yet
        ctx.sdtw_batch(haru.HARU_INT16, ev, off)
        stats = ctx.last_stats()
        assert stats["groups"] > 0
        ctx.ref_load(ref)
        assert ctx.last_stats() == stats
        ctx.ref_build(rng.integers(0, 4, 5000, dtype=np.uint8), rng.normal(90, 12, 4 ** 6).astype(np.float32), 6)
        assert ctx.last_stats() == stats
        with pytest.raises(haru.HaruError):
            ctx.ref_load(np.full(10, 1.0, np.float32))  # zero spread: the load's status, not the batch's
        assert ctx.last_status() == haru.HARU_OK
        assert ctx.last_stats() == stats
