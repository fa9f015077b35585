// Internal declarations shared by the CUDA translation units of libharu.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "../../include/haru.h"

namespace haru {

// One warp's work: a query (FP32), a pair of queries packed into the two
// 16-bit halves of every register (INT16 pair), or one query whose int16
// codes are computed exactly in FP32 (wide accumulation). qb < 0 when a pair
// is short. Its steps are cut into nseg segments (work units).
// A stacked item holds two strips one above the other in the warp's PE
// chain: lanes 0..15 sweep qa (and qb, INT16), lanes 16..31 sweep qc (and
// qd), each 16 * S rows high; lane 16 starts its stack from the free-start
// row instead of lane 15's last row.
struct Item {
  int qa;
  int qb;
  int S;        // rows per lane of the warp strip: 32 * S (16 * S if stacked) >= longest query
  int nseg;     // segments of its sweep
  int qmax;     // INT16: largest |code| of its queries (written by the packing kernel)
  int qc;       // stacked: lower stack's queries (-1: none)
  int qd;
  int stacked;  // 1: two stacks of 16 lanes
};

// Queries of at most this many events are stacked two to a warp strip in
// batches large enough to fill the machine:
// stacking doubles the rows per lane, which raises throughput but also the
// time one strip takes, so small (latency-bound) batches stay unstacked.
constexpr int kStackMax = 16 * 16;

// Last-row minimum of one unit (item, segment): int16 halves a and b, or fp32.
struct Best {
  int ia, ib;
  float f;
  int pad;
  int64_t ca, cb;
};

// Per-item register image: [2][S][32] 32-bit words (INT16: the packed query
// codes as sign-magnitude halves, kPadHalf on pad rows, then as two's
// complement, kPadCode on pad rows; FP32: query samples (0 on pad rows) and
// row weights, -1 on real rows and 0 on pad rows).
constexpr int kImgStride = 2 * 16 * 32;
// A saved strip state: the last two oblique columns, [2][S][32] words (the
// start-column forms follow them with their start columns, as many words).
constexpr int kStateStride = 2 * 16 * 32;
constexpr int kMaxS = 16;
constexpr int kMaxWarps = 12;       // per CTA
constexpr int kSharedHeader = 2560;  // shared-memory bytes before the tracking rings
constexpr int kMaxSeg = 320;  // segments per item, at most
constexpr int kQmax = HARU_INT16_QMAX;
// An int16 code as a sign-magnitude half is the fp16 number code * 2^-24 (a
// subnormal up to 1023, then the first normal binade, whose spacing is the
// same): differences of two codes are exact in fp16 up to 2^11, and the
// result's low 11 bits are the distance |q - r| itself. A pad row holds
// 2^15 (0x7800): minus any code it stays 2^15, whose low 11 bits are 0.
constexpr int kHalfSpan = 2047;      // largest |q| + |r| the 11 bits hold
constexpr uint32_t kPadHalf = 0x7800u;
constexpr int kPadCode = -4095;      // two's complement image: distance 0 through the relu
__host__ __device__ constexpr uint32_t half_code(int q) {
  return q < 0 ? 0x8000u | static_cast<uint32_t>(-q) : static_cast<uint32_t>(q);
}
constexpr int kCap = HARU_INT16_CAP;
// Extra reference columns past N that the tile stream may read: the lane
// skew of the tallest strip (32 * 16) plus one whole tile.
constexpr int kMaxTile = 16384;
constexpr long kRefPad = 32 * kMaxS + kMaxTile + 64;
// Zero columns in front of column 0 of the device reference images: lane l
// of a strip reads the reference at column t - l * S (up to 31 * kMaxS
// behind the warp's step), and a tile's copy starts this many columns before
// the tile.
constexpr long kRefFront = 512;
static_assert(kRefFront >= 31 * kMaxS && kRefFront % 16 == 0, "front pad: the largest lane lag, whole 64-byte lines");

// Internal precisions of the sweep kernels beyond the public HARU_FP32,
// HARU_INT16 and HARU_INT16_ACC32: the FP32 and wide forms that also carry
// each alignment's start column (haru_sdtw_batch_span).
constexpr int kPrecF32Span = 3, kPrecWideSpan = 4;
// and the int16 form of a batch in which some codes may be too large for the
// half-code cell (kHalfSpan): its sweep holds both int16 cells and picks one
// for each bundle or group. 8,192 uneven queries, one of them or 5% with large
// codes, take 11.2 and 12.4 ms (none: 11.2); with a sweep of its own for the
// bundles that hold one, run before the half-code sweep on the same schedule,
// 17.2 and 23.1; with the cell picked for each warp, 11.3 and 22.0 (the code
// of two strips does not fit the instruction cache).
constexpr int kPrecI16Mixed = 5;
__host__ __device__ constexpr bool prec_span(int p) { return p == kPrecF32Span || p == kPrecWideSpan; }
// Tracking-ring words per warp: costs (and start columns, +128, for the span forms).
// Words of one flush buffer of a warp's last-row tracking ring: a whole
// strip's tracked lane fills all of it between two scans, each stack of a
// stacked strip half. A warp holds two buffers, and the forms with start
// columns keep two more for the starts. Measured per form on GB300: 64 words
// for the int16 strips, 128 for the FP32-unit ones (fewer scans; the int16
// kernel ran 0.5% slower with 128, FP32 2.9% faster).
__host__ __device__ constexpr int flush_words(int p) { return p == HARU_INT16 || p == kPrecI16Mixed ? 64 : 128; }
__host__ __device__ constexpr int ring_words(int p) { return (prec_span(p) ? 4 : 2) * flush_words(p); }
// Words of one saved strip state: costs, and start columns for the span forms.
__host__ __device__ constexpr int state_words(int p) { return prec_span(p) ? 2 * kStateStride : kStateStride; }

// Consecutive items with the same S swept over the same segment by one CTA,
// sharing one stream of reference tiles (the dynamic queue of a batch with an
// explicit unit target).
struct Group {
  int S;
  int first;
  int count;
  int seg;
  int nseg;
  int pad[3];
};

// The static schedule of a batch planned by the cost model. Units (item x
// segment, segment-major) of each strip height form bundles of `members`, run
// by a CTA's warps side by side; the few items beyond the last full bundle
// (`rest`) are cut into segments of their own so that theirs are full too. The
// bundles' estimated times, tallest strips first, lie end to end on one line,
// and CTA p runs the line's stretch
// [p * share, (p + 1) * share). No bundle is longer than a share, so at most
// one crosses each border: the CTA before the border runs the bundle's first
// steps before anything else, the one after it the remaining steps from the
// exact state they left, after everything else. Every CTA is busy for one
// share, and only ever waits for a CTA that started before it.
struct ScheduleRow {
  int items, base;       // count, first item
  int nseg;
  int bundles, bundle0;  // count, number of bundles before them
  int last;              // warps at work in the last bundle
  long long start;       // on the line
  long long cost, last_cost;  // of a full bundle, and of the last one
};
struct Schedule {
  int members, bundles;
  long long share, total;
  ScheduleRow row[2 * kMaxS];  // on the line from the last to the first; see schedule_row
};
__host__ __device__ constexpr int schedule_row(int S, int rest) { return 2 * (S - 1) + 1 - rest; }

// Opt a kernel in to `bytes` of dynamic shared memory on the current
// device, calling the driver only when the size grows past what was set
// before on that device (a serving loop launches every few hundred
// microseconds). One record per kernel: `set` per device, under `mu`.
constexpr int kMaxDevices = 64;
struct SmemOptIn {
  std::atomic<int> set[kMaxDevices] = {};
  std::mutex mu;
};
template <class K>
inline cudaError_t opt_in_smem(K kernel, SmemOptIn &rec, size_t bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int want = static_cast<int>(bytes);
  if (dev < 0 || dev >= kMaxDevices)
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, want);
  if (rec.set[dev].load(std::memory_order_acquire) >= want) return cudaSuccess;
  std::lock_guard<std::mutex> lk(rec.mu);
  if (rec.set[dev].load(std::memory_order_relaxed) >= want) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, want);
  if (e == cudaSuccess) rec.set[dev].store(want, std::memory_order_release);
  return e;
}

// Layout of the small integer block every batch uses: the status word, the
// planner's group and item counts, the fix-up count, the sweep kernel's work
// queue counter, the most segments any item was cut into, and whether a sweep
// gave up on a wait.
constexpr int kIntStatus = 0, kIntGroups = 1, kIntItems = 2, kIntFixups = 3, kIntQueue = 4, kIntMaxSeg = 5,
              kIntAbort = 6, kIntWords = 7;

// Steps per unrolled chunk of every strip height. The costs alternate between
// two registers and a lane reads its reference samples up to four at a time,
// so it is a multiple of four; it spreads the chunk's own work (flush, state
// and loop tests) and the tracked lane's stores. Clocks of an int16 step with
// chunks of S steps (8 at least) and of 16, twelve warps an SM: 2 rows 20.2
// and 17.7, 5 rows 33.4 and 33.2, 9 rows 54.4 and 51.9, 13 rows 71.7 and
// 70.0, 8 rows 46.9 and 47.1; with four warps 45.1 and 38.7, 70.5 and 61.0
// (8 rows), 90.2 and 89.1 (13).
constexpr int kChunk = 16;

// Tile width (columns): whole chunks, not above T.
__host__ __device__ inline int tile_width(int T) {
  const int w = T / kChunk * kChunk;
  return w > 0 ? w : kChunk;
}

// Steps a speculative segment runs before its own first step: three strip
// heights, so even the strip's last row has two heights of columns behind
// it (alignments span fewer columns than rows here; a segment whose start
// state still differs is recomputed by the fix-up kernel).
__host__ __device__ inline long warmup_steps(int S) {
  return (3L * 32 * S + kChunk - 1) / kChunk * kChunk;
}

// Whole-chunk step count of one sweep of strip height S over N columns.
__host__ __device__ inline long sweep_steps(int S, long N) {
  return (N + 32L * S - 1 + kChunk - 1) / kChunk * kChunk;
}

// Steps of segment `seg` of `nseg`: own steps [t_own, t_end), warm-up from t_start.
__host__ __device__ inline void seg_bounds(int S, int nseg, int seg, long N, long *t_start, long *t_own,
                                           long *t_end) {
  const long chunks = sweep_steps(S, N) / kChunk;
  *t_own = chunks * seg / nseg * kChunk;
  *t_end = chunks * (seg + 1) / nseg * kChunk;
  const long w = *t_own - warmup_steps(S);
  *t_start = seg == 0 ? 0 : (w > 0 ? w : 0);
}

// Steps between two checkpoints: `step` rounded up to whole chunks.
__host__ __device__ inline int checkpoint_steps(int step) {
  return (step + kChunk - 1) / kChunk * kChunk;
}

// The end column a trace of start columns runs to, given a query's result:
// -1 (no trace) for none, for one that is not a column of the reference, and
// for every query of a batch that gave up on a device wait: units that never
// ran leave whatever their minima held before, and a trace reads the reference
// up to its end column.
__host__ __device__ constexpr long trace_end(int64_t col, long N, int gave_up) {
  return gave_up || col < 0 || col >= N ? -1 : static_cast<long>(col);
}

// Steps from t_start to where a bundle cut at `at` of `cost` on the schedule's
// line stops (whole chunks; the same operands give the same cut on both sides).
__host__ __device__ inline long cut_steps(long t_start, long t_end, long long at, long long cost) {
  if (at <= 0) return 0;
  if (at >= cost) return t_end - t_start;
  return static_cast<long>(static_cast<double>((t_end - t_start) / kChunk) * (static_cast<double>(at) / cost)) * kChunk;
}

struct SdtwArgs {
  const void *ref_img;     // INT16: uint32 (h | h << 16), h the half code; integer forms in FP32: (r | r << 16);
                           // FP32: float. Column 0 of N + kRefPad words, kRefFront zero words before it
  const void *ref_large;   // INT16: uint32 (r | r << 16), for items with large codes
  int half_max;            // INT16: largest query |code| the half-code cell takes (kHalfSpan - the reference's)
  int large_possible;      // INT16: an item may hold larger codes (the sweep with both cells is launched)
  long N;                  // reference length (columns)
  const uint32_t *img;     // item images, kImgStride words each
  const Item *items;
  const Group *groups;
  int *ints;               // kIntWords status and counter words
  uint32_t *states;        // [item][nseg_cap][2] saved states (start, final), kStateStride words each
  Best *bests;             // [item][nseg_cap]: the strip's (upper stack's) last-row minimum
  Best *bests2;            // [item][nseg_cap]: the lower stack's, for stacked items
  const Schedule *sched;   // the static schedule (solo)
  int *done;               // [CTA]: whether its part of the bundle across its right border is done (solo; zeroed by
                           // the planner)
  int *arrived;            // [item]: CTAs of the fix-up kernel that verified their segments (zeroed by the planner)
  int64_t *out_start;      // span forms: the alignment start column per query
  uint32_t *checkpoints;   // [item][checkpoint_cap] states, kStateStride words each, before steps checkpoint_steps(S) *
                           // 1, 2, ...; nullptr: none (a traced batch's cost sweep saves them)
  int checkpoint_cap, checkpoint_step;
  int nseg_cap;
  float *out_cost;
  int64_t *out_col;
  float inv_scale;         // INT16: 2^-k
  int tile_cols;           // requested tile width T (columns)
  int warps;               // warps per CTA = items per group
  int solo;                // static schedule, each warp streams its own tiles; else the queue of groups
  unsigned long long wait_ns;
};

// Planner / prep arguments.
struct PlanArgs {
  const uint32_t *offsets;  // nq + 1
  uint32_t nq;
  long N;
  int pair;                 // 0: FP32 singles; 1: INT16 pairs; 3: exact-integer singles, unsaturated
                            // (HARU_INT16_ACC32)
  int zero;                 // 1: the planner zeroes ints first
  int warps;                // warps per CTA (explicit unit target: items per group)
  int units_target;         // wanted work units (item x segment) in the batch; 0: by the cost model below
  int slots;                // cost model: CTAs
  float clocks[kMaxS];      //   clocks of a step of S rows per lane and warp, with all of the CTA's warps at work;
  float stacked, two, one;  //   more of them on stacked items, with two warps, and with one, on a scheduler
  Schedule *sched;          //   result
  int *done;                //   zeroed, one word per CTA
  int stack;                // 1: stack queries of <= kStackMax events two to a strip
  int nseg_cap;             // most segments per item (state storage is sized for it)
  Item *items;
  int *arrived;             // zeroed, one word per item (nullptr: not used)
  Group *groups;
  int *ints;                // kIntWords counters (status, counts, queues, class ranges)
};

struct PackArgs {
  const float *events;
  const uint32_t *offsets;
  Item *items;              // read; INT16: qmax is written
  const int *n_items;
  uint32_t *img;
  int raw;                  // z-score each query first
  const double *qstats;     // raw: (mean, sigma) of query q at 2q, 2q+1 (launch_prep)
  int pair;
  int scale_log2;
  int *status;
};

// Kernel launchers (stream-ordered, no synchronisation).
// The plan and, on raw events (qstats != nullptr), the mean and population
// sigma (FP64, sequential order) of each query of 1..512 events. sms: of the
// device.
cudaError_t launch_prep(const PlanArgs &a, const float *events, double *qstats, int sms, cudaStream_t s);
cudaError_t launch_pack(const PackArgs &a, uint32_t max_items, cudaStream_t s);
cudaError_t launch_sdtw(int precision, const SdtwArgs &a, int grid, int fix_items, cudaStream_t s,
                        cudaEvent_t ev_fix = nullptr);
// Start columns from the checkpoints of a cost sweep whose results are in
// out_cost / out_col (span precisions).
cudaError_t launch_trace(int precision, const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s);
// cudaEventRecord that also works inside a stream capture (batch.cu).
cudaError_t record_event(cudaEvent_t e, cudaStream_t s);
// Load kernels into the current context now instead of at their first
// launch (lazy module loading): the planner, statistics and packing kernels,
// and the sweep and fix-up kernels of a precision.
cudaError_t load_prep_kernels();
cudaError_t load_sdtw(int precision);
size_t sdtw_smem_bytes(int precision, int tile_cols, int warps, bool solo);
int sdtw_max_ctas_per_sm(int precision, int tile_cols, int warps);

// Reference preparation.
cudaError_t launch_ref_levels(const uint8_t *bases, size_t n, const float *model, int k, float *out,
                              int *status, cudaStream_t s);
cudaError_t launch_zscore_stats(const float *x, size_t n, double *partials, double *stats, int *status,
                                cudaStream_t s);
cudaError_t launch_ref_finish(const float *x, size_t n, const double *stats, int normalize, int scale_log2,
                              float *z, uint32_t *img16, uint32_t *imgh, float *img32, int *status, int *max_code,
                              cudaStream_t s);

// Set *status to code if it is still 0 (device side).
__device__ __forceinline__ void report(int *status, int code) { atomicCAS(status, 0, code); }

}  // namespace haru
