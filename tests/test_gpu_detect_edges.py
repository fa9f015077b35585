"""Event detection at the edges of its paths: every window length (register sums
up to 8 samples, sliding sums above), samples whose range does and does not
fit the 32-bit sums, reads around a tile's and a vector load's length. Events
and counts equal the oracle's exactly."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def reads(rng, spread, flat):
    lengths = list(range(0, 20)) + [63, 64, 65, 1005, 1006, 1007, 1023, 1024, 1025, 2048, 4001, 16384]
    parts = []
    for i, n in enumerate(lengths):
        level = rng.normal(0.0, spread, n // 7 + 2).repeat(7)[:n]
        x = np.clip(500 + level + rng.normal(0.0, spread / 8, n), -32768, 32767)
        if flat and n > 40:
            x[n // 3: n // 2] = x[n // 3]   # flat stretch: equal statistics
            x[n // 2: n // 2 + 9] = -x[n // 3]
        if i % 5 == 4 and n > 3:
            x[n // 2] = 32767 if i % 2 else -32768  # a spike past the 32-bit range
        parts.append(np.rint(x).astype(np.int16))
    off = np.zeros(len(parts) + 1, np.uint32)
    off[1:] = np.cumsum(lengths)
    return np.concatenate(parts), off


@pytest.mark.parametrize("w1,w2", [(2, 2), (3, 6), (4, 5), (7, 8), (8, 9), (3, 16), (16, 16)])
@pytest.mark.parametrize("spread,flat", [(70.0, False), (3000.0, True), (20000.0, False)])
def test_events_match_oracle(haru, w1, w2, spread, flat):
    smp, off = reads(np.random.default_rng(w1 * 100 + w2 + int(spread)), spread, flat)
    with haru.Context() as ctx:
        p = ctx.event_params(window_short=w1, window_long=w2, trim_events=3, max_events=500)
        ev, eoff = ctx.detect_events(smp, off, p)
    oev, ooff = oracle.signal_events(smp, off, w1=w1, w2=w2, tau1_centi=p.threshold_short_centi,
                                     tau2_centi=p.threshold_long_centi, trim=3, max_events=500)
    np.testing.assert_array_equal(eoff, ooff)
    np.testing.assert_array_equal(ev, oev)
