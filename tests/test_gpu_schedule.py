"""The planner's static schedule (the default) against unsplit sweeps from the
queue (units_target=1): batches from one query to several bundles per CTA, so
that units are cut at borders between CTAs, run as many short segments, and
leave ragged last bundles. Every result is the plain DP's: equal bit for bit."""
import numpy as np
import pytest

from gpu_util import compare_int16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def batch(nq, lo, hi, seed, n):
    rng = np.random.default_rng(seed)
    lengths = rng.integers(lo, min(hi, n) + 1, nq)
    off = np.zeros(nq + 1, np.uint32)
    off[1:] = np.cumsum(lengths)
    return rng.normal(90.0, 12.0, n).astype(np.float32), rng.normal(90.0, 12.0, int(off[-1])).astype(np.float32), off


# one query, a ragged bundle, a bundle and one more, several heights, over 12 x 152 items, a reference shorter than a
# strip, and one reference column per query event
@pytest.mark.parametrize("nq,lo,hi,n", [(1, 250, 250, 60000), (1, 512, 512, 512), (1, 2, 2, 2), (5, 2, 40, 9000),
                                        (13, 250, 250, 30011), (26, 100, 300, 30011), (300, 2, 512, 9001),
                                        (2500, 2, 512, 5003), (4000, 200, 260, 3001)])
@pytest.mark.parametrize("stack", [-1, 1])
def test_schedule_matches_unsplit(haru, nq, lo, hi, n, stack):
    ref, ev, off = batch(nq, lo, hi, nq * 7 + n, n)
    with haru.Context(stack_short=stack) as auto, haru.Context(stack_short=stack, units_target=1) as plain:
        for ctx in (auto, plain):
            ctx.ref_load(ref)
        for prec in (haru.HARU_INT16, haru.HARU_FP32, haru.HARU_INT16_ACC32):
            a, b = (ctx.sdtw_batch(prec, ev, off) for ctx in (auto, plain))
            np.testing.assert_array_equal(a[0], b[0])
            np.testing.assert_array_equal(a[1], b[1])
            if prec == haru.HARU_INT16 and nq <= 26 and stack < 0:
                compare_int16(a[0], a[1], ref, ev, off)


# Tracing starts from checkpoints (references of 2,048 columns and more) against carrying them through the sweep: just
# below and above the line; queries end anywhere, whole checkpoints back included.
@pytest.mark.parametrize("n", [2047, 2048, 2049, 30011])
@pytest.mark.parametrize("units,stack", [(0, -1), (0, 1), (1, 1), (2000, -1)])
def test_start_columns_match_oracle(haru, n, units, stack):
    import oracle
    nq = 24
    ref, ev, off = batch(nq, 1, 512, n, n)
    ref, ev = (ref - 90) / 4 + 15, (ev - 90) / 4 + 15  # codes around 960, none at the clamp
    ev[off[3]:off[4]] = ref[:off[4] - off[3]]          # from the first column on
    ev[off[5]:off[6]] = ref[n - (off[6] - off[5]):]    # to the last
    with haru.Context(stack_short=stack, units_target=units) as ctx:
        ctx.ref_load(ref, normalize=False)
        for prec, oprec in ((haru.HARU_FP32, oracle.PREC_F32), (haru.HARU_INT16_ACC32, oracle.PREC_I32)):
            cost, col, start = ctx.sdtw_batch_span(prec, ev, off, raw=False)
            o = oracle.batch(oprec, ref, ev, off, normalize_ref=False, normalize_q=False, start=True)
            np.testing.assert_array_equal(cost, o.cost)
            np.testing.assert_array_equal(col, o.col)
            np.testing.assert_array_equal(start, o.start)
