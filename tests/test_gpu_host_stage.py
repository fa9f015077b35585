"""Host calls give the results of the on-device calls at the edges of the pinned
staging: inputs just inside, at and beyond its size, results inside and beyond."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

STAGE = 1 << 20  # bytes


@pytest.fixture(scope="module")
def haru():
    import paper_2211_07340_gb300 as h
    h.build_library()
    return h


# queries of 3 events: 16 bytes a query + 4 come in, 12 (20 with starts) a query + 8 go out
@pytest.mark.parametrize("span", [False, True])
@pytest.mark.parametrize("nq", [1, STAGE // 16 - 1, STAGE // 16, (STAGE - 8) // 20, (STAGE - 8) // 20 + 1,
                                (STAGE - 8) // 12, (STAGE - 8) // 12 + 1])
def test_host_call_equals_device_call(haru, nq, span):
    rng = np.random.default_rng(nq)
    ev = rng.normal(90.0, 12.0, 3 * nq).astype(np.float32)
    off = (3 * np.arange(nq + 1)).astype(np.uint32)
    d_ev, d_off = torch.from_numpy(ev).cuda(), torch.from_numpy(off.view(np.int32)).cuda()
    cost = torch.empty(nq, device="cuda")
    col, start = (torch.empty(nq, dtype=torch.int64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    with haru.Context() as ctx:
        ctx.ref_load(rng.normal(90.0, 12.0, 60).astype(np.float32))
        if span:
            got = ctx.sdtw_batch_span(haru.HARU_FP32, ev, off)
            ctx.sdtw_batch_span_device(haru.HARU_FP32, d_ev, d_off, cost, col, start)
        else:
            got = ctx.sdtw_batch(haru.HARU_FP32, ev, off)
            ctx.sdtw_batch_device(haru.HARU_FP32, d_ev, d_off, cost, col)
    want = (cost, col, start)[: len(got)]
    for g, w in zip(got, want):
        np.testing.assert_array_equal(g, w.cpu().numpy())
