// Launch dispatch of the sweep and fix-up kernels. The kernels are defined
// in sdtw_kernels.cuh and instantiated one kernel precision per translation
// unit (sdtw_p<P>.cu: scheduled sweep; queue_p<P>.cu: the queue's sweep;
// fixup_p<P>.cu: fix-up; trace_p<P>.cu: trace), so they compile in parallel.

#include <cuda_runtime.h>

#include <mutex>
#include <vector>

#include "haru_internal.h"

namespace haru {

#define HARU_SDTW_SCHEDULED(P)                                             \
  cudaError_t sdtw_sweep_##P(const SdtwArgs &a, int grid, cudaStream_t s); \
  cudaError_t sdtw_sweep_load_##P();
#define HARU_SDTW_QUEUED(P)                                                \
  cudaError_t sdtw_queue_##P(const SdtwArgs &a, int grid, cudaStream_t s); \
  int sdtw_occupancy_##P(int tile_cols, int warps);                        \
  cudaError_t sdtw_queue_load_##P();
#define HARU_SDTW_FIXED_UP(P)                                                   \
  cudaError_t sdtw_fixup_##P(const SdtwArgs &a, int fix_items, cudaStream_t s); \
  cudaError_t sdtw_fixup_load_##P();
HARU_SDTW_SCHEDULED(0) HARU_SDTW_QUEUED(0) HARU_SDTW_FIXED_UP(0)
HARU_SDTW_SCHEDULED(1) HARU_SDTW_QUEUED(1) HARU_SDTW_FIXED_UP(1)
HARU_SDTW_SCHEDULED(2) HARU_SDTW_QUEUED(2) HARU_SDTW_FIXED_UP(2)
HARU_SDTW_QUEUED(3) HARU_SDTW_FIXED_UP(3)
HARU_SDTW_QUEUED(4) HARU_SDTW_FIXED_UP(4)
HARU_SDTW_SCHEDULED(5) HARU_SDTW_QUEUED(5)
cudaError_t sdtw_trace_3(const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s);
cudaError_t sdtw_trace_4(const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s);

size_t sdtw_smem_bytes(int precision, int tile_cols, int warps, bool solo) {
  // Shared header, per-warp tracking rings, two tile slots per stream (each
  // with the kRefFront columns before its tile)
  return kSharedHeader + static_cast<size_t>(warps) * ring_words(precision) * 4 +
         (solo ? warps : 1) * 2 * static_cast<size_t>(tile_cols + kRefFront) * 4;
}

namespace {
int occupancy_query(int precision, int tile_cols, int warps) {
  switch (precision) {
    case HARU_INT16: return sdtw_occupancy_1(tile_cols, warps);
    case HARU_INT16_ACC32: return sdtw_occupancy_2(tile_cols, warps);
    case kPrecF32Span: return sdtw_occupancy_3(tile_cols, warps);
    case kPrecWideSpan: return sdtw_occupancy_4(tile_cols, warps);
    default: return sdtw_occupancy_0(tile_cols, warps);
  }
}
}  // namespace

// Resident CTAs per SM of a launch shape of the queue's sweep, asked of the
// runtime once per (device, precision, shape): every batch launch needs it.
int sdtw_max_ctas_per_sm(int precision, int tile_cols, int warps) {
  struct Entry {
    int dev, precision, tile_cols, warps, ctas;
  };
  static std::mutex mu;
  static std::vector<Entry> memo;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return occupancy_query(precision, tile_cols, warps);
  std::lock_guard<std::mutex> lk(mu);
  for (const Entry &x : memo)
    if (x.dev == dev && x.precision == precision && x.tile_cols == tile_cols && x.warps == warps) return x.ctas;
  const int n = occupancy_query(precision, tile_cols, warps);
  if (n > 0) memo.push_back(Entry{dev, precision, tile_cols, warps, n});
  return n;
}

// Load the sweep and fix-up kernels of a precision into the context now
// rather than at their first launch (lazy module loading), so a latency-bound
// caller does not pay the load inside its first request.
cudaError_t load_sdtw(int precision) {
  cudaError_t e;
#define HARU_SDTW_LOAD(P)                                     \
  if ((e = sdtw_sweep_load_##P()) != cudaSuccess) return e;   \
  if ((e = sdtw_queue_load_##P()) != cudaSuccess) return e;   \
  return sdtw_fixup_load_##P();
  switch (precision) {
    case HARU_INT16:
      if ((e = sdtw_sweep_load_5()) != cudaSuccess) return e;
      if ((e = sdtw_queue_load_5()) != cudaSuccess) return e;
      HARU_SDTW_LOAD(1)
    case HARU_INT16_ACC32: HARU_SDTW_LOAD(2)
    case kPrecF32Span:
      if ((e = sdtw_queue_load_3()) != cudaSuccess) return e;
      return sdtw_fixup_load_3();
    case kPrecWideSpan:
      if ((e = sdtw_queue_load_4()) != cudaSuccess) return e;
      return sdtw_fixup_load_4();
    default: HARU_SDTW_LOAD(0)
  }
#undef HARU_SDTW_LOAD
}

// The sweep kernel of the precision (scheduled, or from the queue), then its
// segment fix-up kernel (which also writes the outputs), stream-ordered;
// ev_fix (if given) is recorded between the two. An int16 batch that may
// hold large codes runs the sweep with both int16 cells.
cudaError_t launch_sdtw(int precision, const SdtwArgs &a, int grid, int fix_items, cudaStream_t s,
                        cudaEvent_t ev_fix) {
  cudaError_t e;
#define HARU_SDTW_FIX(P)                                                          \
  {                                                                               \
    if (e != cudaSuccess) return e;                                               \
    if (ev_fix && (e = record_event(ev_fix, s)) != cudaSuccess) return e;         \
    return sdtw_fixup_##P(a, fix_items, s);                                       \
  }
#define HARU_SDTW_BOTH(P)                                                         \
  {                                                                               \
    e = a.solo ? sdtw_sweep_##P(a, grid, s) : sdtw_queue_##P(a, grid, s);         \
    HARU_SDTW_FIX(P)                                                              \
  }
  switch (precision) {
    case HARU_INT16:
      if (!a.large_possible) HARU_SDTW_BOTH(1)
      e = a.solo ? sdtw_sweep_5(a, grid, s) : sdtw_queue_5(a, grid, s);
      HARU_SDTW_FIX(1)
    case HARU_INT16_ACC32: HARU_SDTW_BOTH(2)
    case kPrecF32Span:
      e = sdtw_queue_3(a, grid, s);
      HARU_SDTW_FIX(3)
    case kPrecWideSpan:
      e = sdtw_queue_4(a, grid, s);
      HARU_SDTW_FIX(4)
    default: HARU_SDTW_BOTH(0)
  }
#undef HARU_SDTW_BOTH
#undef HARU_SDTW_FIX
}

cudaError_t launch_trace(int precision, const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s) {
  return precision == kPrecF32Span ? sdtw_trace_3(a, max_items, stacked, s) : sdtw_trace_4(a, max_items, stacked, s);
}

}  // namespace haru
