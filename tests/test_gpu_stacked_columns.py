"""Both stacks of a stacked strip start at column 0: the lower stack (lanes
16-31) opens no alignment in front of the reference. The reference stays far
from 0 and the queries begin with zeros, so a zero word in front of column 0
would win at once. Every form and the start columns equal the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import compare_fp32, compare_int16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def batch(n):
    """Four queries (one full int16 item) at the edges of every stacked strip height, that fit the reference."""
    rng = np.random.default_rng(n)
    ref = np.tile([5.0, 6.0, 7.0, 5.5], n // 4 + 1)[:n] + rng.integers(0, 3, n) / 8
    lengths = [m for k in range(17) for m in (16 * k + 1, 16 * k + 8, 16 * k + 15, 16 * k + 16) if m <= min(n, 256)]
    parts = []
    for i, m in enumerate(lengths):
        q = np.resize(ref, m) + rng.integers(-2, 3, m) / 8
        q[:1 + m * (i % 4) // 5] = 0.0
        parts.append(q)
    off = np.zeros(len(parts) + 1, np.uint32)
    off[1:] = np.cumsum(lengths)
    return ref.astype(np.float32), np.concatenate(parts).astype(np.float32), off


# shorter than a strip, below and above the line of traced start columns
@pytest.mark.parametrize("n", [40, 300, 2500])
@pytest.mark.parametrize("units", [0, 1])
def test_lower_stack_starts_at_column_zero(haru, n, units):
    ref, ev, off = batch(n)
    with haru.Context(stack_short=1, units_target=units) as ctx:
        ctx.ref_load(ref, normalize=False)
        c16, j16 = ctx.sdtw_batch(haru.HARU_INT16, ev, off, raw=False)
        c32, j32 = ctx.sdtw_batch(haru.HARU_FP32, ev, off, raw=False)
        cw, jw = ctx.sdtw_batch(haru.HARU_INT16_ACC32, ev, off, raw=False)
        spans = [ctx.sdtw_batch_span(p, ev, off, raw=False) for p in (haru.HARU_FP32, haru.HARU_INT16_ACC32)]
    compare_int16(c16, j16, ref, ev, off, normalize_ref=False, normalize_q=False)
    compare_fp32(c32, j32, ref, ev, off, normalize_ref=False, normalize_q=False)
    compare_int16(cw, jw, ref, ev, off, normalize_ref=False, normalize_q=False, prec=oracle.PREC_I32)
    for (c, j, s), prec in zip(spans, (oracle.PREC_F32, oracle.PREC_I32)):
        o = oracle.batch(prec, ref, ev, off, normalize_ref=False, normalize_q=False, start=True)
        np.testing.assert_array_equal(c, o.cost)
        np.testing.assert_array_equal(j, o.col)
        np.testing.assert_array_equal(s, o.start)
