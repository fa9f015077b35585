"""Mean, sigma and z-scores of raw queries equal the sequential double-precision
rule (FP32 results bit for bit), on events whose sums do and do not round, in
batches of each split of queries over the statistics blocks."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def query(rng, kind, m):
    x = rng.normal(90.0, 12.0, m)
    if kind == 1:
        x = x * 10.0 ** rng.uniform(-12, 12, m)          # partial sums round
    elif kind == 2:
        x = np.rint(x * 8)                                # whole numbers
    elif kind == 3:
        x = np.where(rng.random(m) < 0.5, 0.0, -x)        # zeros, negative
    elif kind == 4:
        x = np.full(m, 90.0) + (np.arange(m) == m // 2)   # one step in a flat query
    elif kind == 5:
        x = x * 1e-40                                     # subnormal
    elif kind == 6:
        x = x * 1e15 + rng.normal(0, 1, m) * 1e-15        # near the 53-bit line from above
    elif kind == 7:
        x = np.rint(x) * 2.0 ** 20 + rng.integers(0, 2, m) * 2.0 ** -20
    return x.astype(np.float32)


@pytest.mark.parametrize("nq", [1, 20, 1300, 5000])
def test_raw_queries_match_oracle(haru, nq):
    rng = np.random.default_rng(nq)
    ref = rng.normal(90.0, 12.0, 700).astype(np.float32)
    lengths = rng.integers(2, 513 if nq <= 20 else 65, nq)
    lengths[: min(nq, 6)] = [512, 2, 33, 64, 65, 511][: min(nq, 6)]
    parts = [query(rng, i % 8, m) for i, m in enumerate(lengths)]
    flat = [p for p in parts if np.ptp(p) == 0]  # short ones of whole numbers or zeros: no spread, no z-score
    spread = [p for p in parts if np.ptp(p) > 0]

    def csr(queries):
        off = np.zeros(len(queries) + 1, np.uint32)
        off[1:] = np.cumsum([q.shape[0] for q in queries])
        return np.concatenate(queries), off

    ev, off = csr(spread)
    with haru.Context(stack_short=-1) as ctx:
        ctx.ref_load(ref)
        if flat:  # one of them makes the batch invalid
            with pytest.raises(haru.HaruError) as e:
                ctx.sdtw_batch(haru.HARU_FP32, *csr(parts))
            assert e.value.code == haru.HARU_EINVAL
        cost, col = ctx.sdtw_batch(haru.HARU_FP32, ev, off)
    o = oracle.batch(oracle.PREC_F32, ref, ev, off)
    np.testing.assert_array_equal(cost, o.cost.astype(np.float32))
    np.testing.assert_array_equal(col, o.col)
