"""int16 form at the edges of its two cells: codes whose magnitudes add up to
at most 2047 run on fp16 half codes, larger ones on two's complement codes;
a batch may hold both. Integer arithmetic: every result equals the oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import compare_int16

pytestmark = pytest.mark.gpu
SCALE = 7


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def codes(rng, n, most):
    c = rng.integers(-most, most + 1, n)
    c[:2] = (most, -most)
    return (c / float(1 << SCALE)).astype(np.float32)


# (largest |reference code|, largest |query code| of the ordinary queries, of the odd ones)
@pytest.mark.parametrize("rmax,qmax,odd", [(1023, 1024, 1024), (1023, 1024, 1025), (1, 2046, 2047), (2047, 0, 1),
                                           (2047, 2047, 2047), (300, 300, 2047)])
@pytest.mark.parametrize("stack,units", [(-1, 0), (1, 1)])
def test_code_ranges(haru, rmax, qmax, odd, stack, units):
    rng = np.random.default_rng(rmax * 4099 + qmax + odd)
    ref = codes(rng, 5003, rmax)
    lengths = np.concatenate([rng.integers(2, 513, 60), [2, 15, 16, 17, 31, 32, 33, 255, 256, 257, 511, 512] * 2])
    parts = [codes(rng, m, odd if i % 17 == 3 else qmax) for i, m in enumerate(lengths)]
    off = np.zeros(len(parts) + 1, np.uint32)
    off[1:] = np.cumsum(lengths)
    ev = np.concatenate(parts)
    with haru.Context(stack_short=stack, units_target=units) as ctx:
        ctx.ref_load(ref, normalize=False, scale_log2=SCALE)
        cost, col = ctx.sdtw_batch(haru.HARU_INT16, ev, off, raw=False)
    compare_int16(cost, col, ref, ev, off, scale_log2=SCALE, normalize_ref=False, normalize_q=False)
