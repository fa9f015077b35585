"""int16 batches in which some queries hold codes too large for the half-code
cell: their bundles run the other cell, in the same sweep as the rest. Integer arithmetic: every result equals the oracle's."""
import numpy as np
import pytest

from gpu_util import compare_int16

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


def batch(nq, lo, hi, n, large, seed):
    """z-values in CSR form; query q of `large` holds one code of 2047 (scale 2^6), beside a reference up to 1023."""
    rng = np.random.default_rng(seed)
    ref = np.clip(rng.normal(0.0, 1.0, n), -15.0, 15.0).astype(np.float32)
    lengths = rng.integers(lo, hi + 1, nq)
    off = np.zeros(nq + 1, np.uint32)
    off[1:] = np.cumsum(lengths)
    ev = rng.normal(0.0, 1.0, int(off[-1])).astype(np.float32)
    ev[off[:-1][large]] = 2047 / 64
    return ref, ev, off


# about two bundles to a CTA, so that nearly every border between CTAs cuts a bundle holding both kinds; one strip
# height and several; bundles of twelve, a ragged one, a single query
@pytest.mark.parametrize("nq,lo,hi", [(7000, 40, 40), (1500, 2, 512), (25, 200, 260), (1, 30, 30)])
@pytest.mark.parametrize("stack,units", [(-1, 0), (1, 0), (1, 3000)])
def test_both_cells_in_one_bundle(haru, nq, lo, hi, stack, units):
    ref, ev, off = batch(nq, lo, hi, 1201, np.arange(nq) % 3 == 0, nq)
    with haru.Context(stack_short=stack, units_target=units) as ctx:
        ctx.ref_load(ref, normalize=False)
        cost, col = ctx.sdtw_batch(haru.HARU_INT16, ev, off, raw=False)
    compare_int16(cost, col, ref, ev, off, normalize_ref=False, normalize_q=False)


def test_large_codes_do_not_idle_the_rest(haru):
    """One query in twenty with a large code: at most the large cell's own extra work on every bundle (10 register
    operands a cell pair instead of 8), within 1.5x; a second sweep over the same schedule took 2.1x."""
    times, s = [], torch.cuda.Stream()
    for every in (0, 20):
        nq = 8192
        large = np.arange(nq) % every == 0 if every else np.zeros(nq, bool)
        ref, ev, off = batch(nq, 100, 500, 59796, large, 1)
        e, o = torch.from_numpy(ev).cuda(), torch.from_numpy(off.astype(np.int32)).cuda()
        cost = torch.empty(nq, device="cuda")
        col = torch.empty(nq, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        with haru.Context() as ctx:
            ctx.ref_load(ref, normalize=False)
            best = float("inf")
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(s)
                ctx.sdtw_batch_device(haru.HARU_INT16, e, o, cost, col, stream=s.cuda_stream, raw=False,
                                      asynchronous=True)
                b.record(s)
                s.synchronize()
                best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] <= 1.5 * times[0], times
