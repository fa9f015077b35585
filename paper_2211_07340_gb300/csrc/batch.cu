// The batch engine: workspace sizing and the stream-ordered sequence of
// kernels of one batch (planner, pack, sweep, segment fix-up).

#include <cuda_runtime.h>

#include <algorithm>

#include "engine.h"

namespace haru {

cudaError_t record_event(cudaEvent_t e, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t r = cudaStreamIsCapturing(s, &cs);
  if (r != cudaSuccess) return r;
  if (cs == cudaStreamCaptureStatusActive) return cudaEventRecordWithFlags(e, s, cudaEventRecordExternal);
  return cudaEventRecord(e, s);
}

void ws_free(Workspace &ws) {
  void *p[] = {ws.ints, ws.items, ws.arrived, ws.groups, ws.sched, ws.done, ws.img, ws.states, ws.bests, ws.qstats, ws.checkpoints};
  for (void *q : p)
    if (q) cudaFree(q);
  ws = Workspace();
}

// Checkpoints per item: up to 128 (a trace runs half the distance between two
// of them on average beside two strip heights), fewer in batches whose
// states would pass 512 MB, at least 8; at least 256 steps apart. From
// kFewCheckpoints items on 4 do: 8 take an item to 52 KB, a batch of 5.4 M
// queries to the whole memory, 4 to 36 (1.1 M x 100..120 events on 20,000
// columns: 473 ms with 8, 590 with 4).
constexpr size_t kFewCheckpoints = 1u << 22;
int checkpoint_cap(size_t max_items, long N) {
  const size_t fit = (static_cast<size_t>(512) << 20) / (max_items * kStateStride * sizeof(uint32_t));
  const size_t least = max_items < kFewCheckpoints ? 8 : 4;
  const long most = std::min<long>(std::min<size_t>(std::max(fit, least), 128), (N + 32 * kMaxS) / 256);
  return static_cast<int>(std::max<long>(most, 1));
}

namespace {

// Tile of a warp's own stream: two slots of (kSoloTile + kRefFront) words and
// the tracking ring leave room for twelve warps in an SM's shared memory.
constexpr int kSoloTile = 1536;

// Clocks of one step of a strip of 1 .. 16 rows per lane, per warp of its
// scheduler: with all twelve of the CTA at work (three a scheduler), and how
// many more on stacked items, with two warps and with one. Measured on GB300,
// one strip height at a time, 152 CTAs (60,000 columns); alone on a scheduler
// a warp takes 16 (int16) and 9 clocks more there, but CTAs of few warps also
// tend to be those that change strip heights and fetch instructions anew, and
// with those figures small uneven batches were cut too finely (ten batches of
// 141 x 41..424 FP32 events on 29,166 columns: 329 us on average, 272 us with
// these; 32 x 250 FP32 133 and 141 us).
struct StepClocks {
  float full[kMaxS], stacked, two, one;
};
const StepClocks kStepI16 = {{18.2f, 18.1f, 22.2f, 25.7f, 33.7f, 35.6f, 43.4f, 45.2f, 50.6f, 56.1f, 62.2f, 65.2f,
                              70.1f, 75.9f, 81.1f, 84.6f}, 0.8f, 5.0f, 23.0f};
const StepClocks kStepF32 = {{16.8f, 15.3f, 18.2f, 20.8f, 26.2f, 30.5f, 36.6f, 38.6f, 45.1f, 48.1f, 53.8f, 56.6f,
                              61.5f, 65.1f, 70.2f, 74.7f}, 0.4f, 4.0f, 13.5f};
const StepClocks &step_clocks(int precision) {
  return precision == HARU_INT16 ? kStepI16 : kStepF32;
}

// Work units that an explicit launch shape is cut into, and the count a batch
// has to reach for its short queries to be stacked.
long stack_units(int precision, const LaunchCfg &lc) {
  return lc.units_target > 0 ? lc.units_target : 4L * lc.sms * kernel_warps(precision, lc);
}

// Buffer sizes one batch of nq queries needs.
struct WsNeeds {
  size_t max_items, units, groups, ctas, qstats, states, checkpoints;
  int nseg_cap;
};

// Start-column batches on references of at least kTraceColumns run the cost
// form and trace the starts back from checkpoints; on shorter ones, of few
// query lengths, the starts are carried along. At 2,000
// columns tracing took 163 us for one query, 479 for 100 and 2,090 for 8,000
// uneven ones, carrying 227, 615 and 1,920; at 1,000 columns 161, 494 and
// 1,754 against 165, 409 and 1,229.
constexpr long kTraceColumns = 2048;
bool traced(int precision, const LaunchCfg &lc) { return prec_span(precision) && lc.N >= kTraceColumns; }
int cost_form(int precision) {
  return precision == kPrecF32Span ? HARU_FP32 : (precision == kPrecWideSpan ? HARU_INT16_ACC32 : precision);
}

constexpr size_t kTwoSegments = 16;

int checkpoint_step(int cap, long N) { return static_cast<int>((N + 32 * kMaxS + cap) / cap); }

WsNeeds ws_needs(int precision, uint32_t nq, const LaunchCfg &lc) {
  WsNeeds w;
  const bool trace = traced(precision, lc);
  if (trace) precision = cost_form(precision);
  const BatchShape sh = batch_shape(precision, nq, lc);
  const int mode = plan_mode(precision);
  w.max_items = items_bound(mode, nq);
  // Fewest items the batch can make (stacked: four int16 or two other
  // queries per item); the segment cap is sized for that case.
  const size_t per_item = (mode == 1 ? 2 : 1) * (sh.stack ? 2 : 1);
  const size_t items_min = (static_cast<size_t>(nq) + per_item - 1) / per_item;
  if (!sh.solo) {
    // (twice the wanted segments: the planner doubles those of the queue's tail)
    const size_t units = static_cast<size_t>(stack_units(precision, lc));
    w.nseg_cap = static_cast<int>(std::min<size_t>(64, 2 * ((units + items_min - 1) / items_min)));
  } else {
    // The cost model spreads a batch over at most about two units per resident
    // warp. From kTwoSegments items per resident warp on, a third segment buys
    // no balance (60,000 x 100..500 FP32 events on 6,000 columns: 15.2 ms with
    // two and with three) and its states cost 8 KB of an item's 28.
    const size_t resident = static_cast<size_t>(lc.sms) * sh.per_sm * sh.warps;
    w.nseg_cap = static_cast<int>(std::min<size_t>(kMaxSeg, 2 + (2 * resident + items_min - 1) / items_min));
    if (items_min >= kTwoSegments * resident) w.nseg_cap = 2;
  }
  w.units = w.max_items * static_cast<size_t>(w.nseg_cap);
  w.ctas = static_cast<size_t>(lc.sms) * sh.per_sm;
  w.groups = sh.solo ? 1 : (w.max_items + kMaxS) * static_cast<size_t>(w.nseg_cap);
  w.qstats = 2 * static_cast<size_t>(nq);
  w.states = w.units * 2 * state_words(precision);
  w.checkpoints = trace ? w.max_items * static_cast<size_t>(checkpoint_cap(w.max_items, lc.N)) * kStateStride : 0;
  return w;
}

cudaError_t ws_alloc(Workspace &ws, const WsNeeds &w) {
  cudaError_t e = cudaSuccess;
  size_t c = ws.ints ? static_cast<size_t>(kIntWords) : 0;
  if ((e = grow(&ws.ints, &c, kIntWords)) != cudaSuccess) return e;
  size_t cs = ws.sched ? 1 : 0;
  if ((e = grow(&ws.sched, &cs, 1)) != cudaSuccess) return e;
  if (ws.cap_items < w.max_items) {
    cudaFree(ws.items);
    cudaFree(ws.arrived);
    cudaFree(ws.img);
    ws.items = nullptr;
    ws.arrived = nullptr;
    ws.img = nullptr;
    ws.cap_items = 0;
    size_t c0 = 0, c1 = 0, c2 = 0;
    if ((e = grow(&ws.items, &c0, w.max_items)) != cudaSuccess) return e;
    if ((e = grow(&ws.arrived, &c1, w.max_items)) != cudaSuccess) return e;
    if ((e = grow(&ws.img, &c2, w.max_items * kImgStride)) != cudaSuccess) return e;
    ws.cap_items = w.max_items;
  }
  if ((e = grow(&ws.groups, &ws.cap_groups, w.groups)) != cudaSuccess) return e;
  if ((e = grow(&ws.done, &ws.cap_done, w.ctas)) != cudaSuccess) return e;
  if ((e = grow(&ws.bests, &ws.cap_bests, 2 * w.units)) != cudaSuccess) return e;
  if ((e = grow(&ws.qstats, &ws.cap_qstats, w.qstats)) != cudaSuccess) return e;
  if (w.checkpoints && (e = grow(&ws.checkpoints, &ws.cap_checkpoints, w.checkpoints)) != cudaSuccess) return e;
  return grow(&ws.states, &ws.cap_states, w.states);
}

}  // namespace

// One CTA per SM with as many warps as the kernel's registers allow, each
// with its own tiles, on the planner's static schedule, which has a CTA's
// warps run one strip height at a time: the instruction cache holds about
// one (three four-warp CTAs of different heights took twice as long on 1,500
// uneven reads), and units of any segments spread evenly over the schedulers
// (CTAs of one warp left some with three and others with none). An explicit
// unit target or CTA count, and the start-column forms (two strip heights of
// whose code do not fit the cache together: 512 uneven queries took 5.4 ms,
// 4.1 from the queue), run the configured shape: groups from a queue, each
// sharing one stream of configured tiles. So do references of fewer than
// kScheduleColumns: a sweep as short as a strip is high leaves nothing to cut,
// and the schedule's own cost shows (20 x 30..200 FP32 z-values on 300
// columns: 58 us scheduled, 39 from the queue; on 600 columns 8..3,000
// queries of one length still gain 5% from the schedule, uneven ones lose 3%).
constexpr long kScheduleColumns = 512;
BatchShape batch_shape(int precision, uint32_t nq, const LaunchCfg &lc) {
  BatchShape sh;
  const long seg_room = std::min<long>(64, lc.N / 8192);
  const long units = stack_units(precision, lc);
  // Auto stacking: when the batch alone fills the unit count, or when its
  // stacked items (up to four queries each) cut into reference segments
  // (at most 64, each counted as 8,192 steps: about four warm-ups of a 16-row strip)
  // still do; small batches on short references stay unstacked for latency.
  const bool fills = static_cast<long>(nq) >= units || static_cast<long>(nq) * seg_room >= 4 * units;
  sh.stack = lc.stack_short > 0 || (lc.stack_short == 0 && fills);
  sh.warps = kernel_warps(precision, lc);
  sh.tile = lc.tile;
  sh.solo = false;
  sh.per_sm = lc.ctas_per_sm > 0 ? lc.ctas_per_sm : 0;
  if (sh.per_sm == 0) sh.per_sm = sdtw_max_ctas_per_sm(precision, sh.tile, sh.warps);
  if (lc.units_target == 0 && lc.ctas_per_sm == 0 && !prec_span(precision) && lc.N >= kScheduleColumns) {
    sh.solo = true;
    sh.warps = kMaxWarps;
    sh.tile = kSoloTile;
    sh.per_sm = 1;
  }
  if (sh.per_sm < 1) sh.per_sm = 1;
  return sh;
}

cudaError_t ws_reserve(Workspace &ws, int precision, uint32_t nq, const LaunchCfg &lc) {
  const WsNeeds w = ws_needs(precision, nq, lc);
  cudaError_t e = ws_alloc(ws, w);
  if (e != cudaSuccess) return e;
  ws.max_items = w.max_items;
  ws.nseg_cap = w.nseg_cap;
  return cudaSuccess;
}

cudaError_t ws_reserve_upto(Workspace &ws, int precision, uint32_t max_nq, const LaunchCfg &lc) {
  WsNeeds most{};
  for (uint32_t n = 1; n <= max_nq; ++n) {  // sizing arithmetic only; one allocation per buffer
    const WsNeeds w = ws_needs(precision, n, lc);
    most.max_items = std::max(most.max_items, w.max_items);
    most.units = std::max(most.units, w.units);
    most.groups = std::max(most.groups, w.groups);
    most.ctas = std::max(most.ctas, w.ctas);
    most.qstats = std::max(most.qstats, w.qstats);
    most.states = std::max(most.states, w.states);
    most.checkpoints = std::max(most.checkpoints, w.checkpoints);
  }
  return ws_alloc(ws, most);
}

cudaError_t ws_enqueue(Workspace &ws, int precision, const RefView &ref, const float *d_events,
                       const uint32_t *d_offsets, uint32_t nq, int raw, float *d_cost, int64_t *d_col,
                       const LaunchCfg &lc, cudaStream_t s, cudaEvent_t ev_prep, cudaEvent_t ev_sweep,
                       int64_t *d_start, bool zero_counters, cudaEvent_t ev_fix) {
  cudaError_t e;
  const int asked = precision;
  const bool trace = traced(precision, lc);
  if (trace) precision = cost_form(precision);
  if (ev_prep && (e = record_event(ev_prep, s)) != cudaSuccess) return e;
  PlanArgs pa;
  pa.offsets = d_offsets;
  pa.nq = nq;
  pa.N = ref.N;
  pa.pair = plan_mode(precision);
  const BatchShape sh = batch_shape(precision, nq, lc);
  pa.warps = sh.warps;
  pa.units_target = sh.solo ? 0 : static_cast<int>(stack_units(precision, lc));
  const int slots = lc.sms * sh.per_sm;
  pa.slots = slots;
  const StepClocks &sc = step_clocks(precision);
  for (int S = 1; S <= kMaxS; ++S) pa.clocks[S - 1] = sc.full[S - 1];
  pa.stacked = sc.stacked;
  pa.two = sc.two;
  pa.one = sc.one;
  pa.sched = ws.sched;
  pa.done = ws.done;
  pa.stack = sh.stack ? 1 : 0;
  pa.nseg_cap = ws.nseg_cap;
  pa.items = ws.items;
  pa.arrived = ws.arrived;
  pa.groups = ws.groups;
  pa.ints = ws.ints;
  // (a caller that ran kernels reporting into the status word first has zeroed the counters itself)
  pa.zero = zero_counters;
  if ((e = launch_prep(pa, d_events, raw ? ws.qstats : nullptr, lc.sms, s)) != cudaSuccess) return e;

  PackArgs ka;
  ka.events = d_events;
  ka.offsets = d_offsets;
  ka.items = ws.items;
  ka.n_items = ws.ints + kIntItems;
  ka.img = ws.img;
  ka.raw = raw;
  ka.qstats = ws.qstats;
  ka.pair = pa.pair;
  ka.scale_log2 = ref.scale_log2;
  ka.status = ws.ints + kIntStatus;
  if ((e = launch_pack(ka, static_cast<uint32_t>(ws.max_items), s)) != cudaSuccess) return e;

  SdtwArgs sa;
  const bool fp_ref = precision == HARU_FP32 || precision == kPrecF32Span;
  sa.ref_img = fp_ref ? static_cast<const void *>(ref.img32)
                      : static_cast<const void *>(precision == HARU_INT16 ? ref.imgh : ref.img16);
  sa.ref_large = ref.img16;
  sa.half_max = kHalfSpan - ref.max_code;
  sa.large_possible = precision == HARU_INT16 && large_codes_possible(ref, raw);
  sa.N = ref.N;
  sa.img = ws.img;
  sa.items = ws.items;
  sa.groups = ws.groups;
  sa.ints = ws.ints;
  sa.states = ws.states;
  sa.bests = ws.bests;
  sa.bests2 = ws.bests + ws.max_items * static_cast<size_t>(ws.nseg_cap);
  sa.sched = ws.sched;
  sa.done = ws.done;
  sa.arrived = ws.arrived;
  sa.out_start = d_start;
  sa.checkpoints = trace ? ws.checkpoints : nullptr;
  sa.checkpoint_cap = trace ? checkpoint_cap(ws.max_items, ref.N) : 0;
  sa.checkpoint_step = trace ? checkpoint_step(sa.checkpoint_cap, ref.N) : 0;
  sa.nseg_cap = ws.nseg_cap;
  sa.out_cost = d_cost;
  sa.out_col = d_col;
  sa.inv_scale = 1.0f / static_cast<float>(1 << ref.scale_log2);
  sa.tile_cols = sh.tile;
  sa.warps = sh.warps;
  sa.solo = sh.solo;
  sa.wait_ns = lc.wait_ns;
  if (ev_sweep && (e = record_event(ev_sweep, s)) != cudaSuccess) return e;
  // One persistent sweep kernel over the whole group list (tallest strips
  // first), then the fix-up kernel, which verifies segments and writes every
  // query's result.
  const size_t groups_max = ((ws.max_items + sh.warps - 1) / sh.warps + kMaxS) * static_cast<size_t>(ws.nseg_cap);
  const int grid = sh.solo ? slots : static_cast<int>(std::min<size_t>(slots, groups_max));
  if ((e = launch_sdtw(precision, sa, grid, static_cast<int>(ws.max_items), s, ev_fix)) != cudaSuccess || !trace) return e;
  return launch_trace(asked, sa, static_cast<int>(ws.max_items), sh.stack, s);
}

}  // namespace haru
