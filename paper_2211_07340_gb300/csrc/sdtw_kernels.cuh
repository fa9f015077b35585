// The sDTW wavefront kernels (Eq. 1, Section 2.3; the pipelined oblique column
// of Section 4.3 / Fig. 5, mapped onto warps).
//
// Layout of one warp's work. A query of M events is padded at the top to
// 32 * S rows (S = floor(M / 32) + 1, at most 16, so that a strip lower than
// 16 rows per lane has at least one pad row); lane l holds rows l*S .. l*S + S - 1 in
// registers (a stacked strip is two such strips of 16 * S rows, in lanes 0..15
// and 16..31, each with its own lane 0). Row i processes reference column t - i at step t, so every row
// is one processing element of the paper's PE chain and the whole strip is
// one oblique column: the S cells of a lane in one step are independent
// (instruction-level parallelism S), a cell reads
//   up   = row i-1 at step t-1,  diag = row i-1 at step t-2,  left = row i at step t-1,
// and each step one value (the bottom row's cost) crosses from lane l-1 to
// lane l by __shfl_up_sync; lane 0 takes the free-start row gamma(0, .) = 0.
// Each lane reads its row 0's reference sample, column t - l*S, from the
// shared tile itself, and the sample moves down the lane's rows by register
// renaming (the oblique column's reference stream, Fig. 5). A sweep is
// N + 32*S - 1 steps, the paper's N + M - 1 (Section 4.3) for the padded
// height. Pad rows sit above the query and hold exactly 0, the free-start
// boundary row, so the last query row is always lane 31's last register.
// A pad row's minimum includes its own 0, so whatever lane 0 receives from
// above is absorbed there, and only full-height strips (16 rows per lane,
// no pad row) have lane 0 replace that value by the zero.
//
// INT16 form: two queries share a warp, one per 16-bit half: |q - r| by an
// fp16x2 subtraction of half codes and a mask, __vimin3_u16x2, and an add, or
// __viaddmin_u16x2 on the rows that saturate at CAP (codes too large for
// halves: __vsub2 and __viaddmax_s16x2_relu); pad rows hold 0. FP32 form: one
// query per warp, 3-input min.f32, gamma = |d| + min3 with d = fma(r, w, q):
// w = -1 on real rows, 0 on pad rows (and q = 0 there).
//
// Segments. The steps of one query are cut into segments that run as
// independent work units. Segment s > 0 starts V steps early from a fresh
// state (as if the reference began there) and records its state (the last
// two oblique columns) when it reaches its own first step B_s; segment s-1
// records its exact state at the same step. The fix-up kernel compares the
// two: equal states give identical computations from B_s on (the DP is a
// deterministic function of that state and the reference), so the segment's
// results stand; otherwise it recomputes the segment from the exact state.
// The result is always the plain DP's.
//
// Schedule. Units are spread over the CTAs by estimated time (Schedule): a
// unit cut at a border between two CTAs saves its exact state there and goes
// on from it on the other one, so balance costs no further warm-up.
//
// The reference streams through shared memory, one stream per warp (a CTA's
// warps run any units of one strip height), or, in the queue, one per CTA
// (same S, same segment). Tiles of T_S columns, each with the kRefFront
// columns before it (the lanes lag the warp's step by up to 31 * S columns),
// are fetched by cp.async.bulk (TMA) into a two-slot ring guarded by mbarriers. The warp that releases a slot last issues the
// copy of the tile two ahead.
//
// The last-row minimum and its first column (Algorithm 1's final scan,
// Algorithm 2's per-column compare) are tracked through a small per-warp
// shared ring: lane 31 (and lane 15 of a stacked strip) stores its bottom-row
// cost of every step, and each time a flush buffer is full every lane scans
// its two (int16) or four entries; a warp reduction keeps the smallest cost,
// then the smallest column.
//
// Every wait is bounded by a global-timer deadline; on expiry the kernel
// records HARU_ETIMEDOUT, waits (bounded) for its own copies in flight and
// returns.

#pragma once

#include <cuda_runtime.h>

#include "haru_internal.h"

namespace haru {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for phase `parity` of `bar` to complete, giving up at `deadline`.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, unsigned parity, unsigned long long deadline) {
  while (!mbar_try_wait(bar, parity)) {
    if (now_ns() > deadline) return false;
  }
  return true;
}
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ float fmin3f(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// This lane's place in its stack: it holds rows place * S .. place * S + S - 1
// of the stack and lags the warp's step by place * S columns. Both stacks of a
// stacked strip start at column 0 on step 0.
__device__ __forceinline__ int stack_place(int lane, bool stk) { return stk ? lane & 15 : lane; }

// x == m ? a : b as a compare and a select (never a branch).
__device__ __forceinline__ int sel_eq(float x, float m, int a, int b) {
  int d;
  asm("{\n\t.reg .pred p;\n\tsetp.eq.f32 p, %1, %2;\n\tselp.b32 %0, %3, %4, p;\n\t}"
      : "=r"(d) : "f"(x), "f"(m), "r"(a), "r"(b));
  return d;
}

// d = a * b + c on the integer multiply-add unit (keeps lane-0 fix-ups off
// the half-rate pipe that the DPX min/max instructions use).
__device__ __forceinline__ uint32_t imad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// This lane's reference sample of step u of a chunk, read A at a time. The
// lane's window starts at column t0 - place * S, a multiple of A (4 when the
// strip height S is a multiple of 4, 2 when it is even, else 1; the chunk's
// first step t0 is a multiple of kChunk, which A divides), so every vector load
// is aligned.
template <int S>
struct LaneWindow {
  static constexpr int A = S % 4 == 0 ? 4 : (S % 2 == 0 ? 2 : 1);
  uint4 v4;
  uint2 v2;
  __device__ __forceinline__ uint32_t get(const uint32_t *ref, int u) {
    if constexpr (A == 4) {
      if (u % 4 == 0) v4 = reinterpret_cast<const uint4 *>(ref)[u / 4];
      const int c = u % 4;
      return c == 0 ? v4.x : (c == 1 ? v4.y : (c == 2 ? v4.z : v4.w));
    } else if constexpr (A == 2) {
      if (u % 2 == 0) v2 = reinterpret_cast<const uint2 *>(ref)[u / 2];
      return (u % 2 == 0) ? v2.x : v2.y;
    } else {
      return ref[u];
    }
  }
};

// The tracked lane's last-row value of step u goes to ring[e0 + u]. Values
// are held for four steps and written by one vector store: e0 is a multiple
// of kChunk and the ring is 16-byte aligned, so every store is aligned. The
// FP32 strips use it; the int16 strip stores every two steps, which measured
// faster there (the held values must be moved into consecutive registers).
struct RingStore {
  uint32_t v[4];
  __device__ __forceinline__ void put(uint32_t *ring, int e0, int u, bool tracked, uint32_t x) {
    v[u % 4] = x;
    if (u % 4 == 3 && tracked) *reinterpret_cast<uint4 *>(ring + e0 + u - 3) = make_uint4(v[0], v[1], v[2], v[3]);
  }
};

// ---------------------------------------------------------------- INT16 --
constexpr uint32_t kCap2 = (static_cast<uint32_t>(kCap) << 16) | static_cast<uint32_t>(kCap);

// Sparse saturation. Costs are held as unsigned 16-bit halves and only rows
// k = S-1, S-1-RUN, ... of each lane take min(CAP, .); the rows between
// add without a cap: a plain 32-bit add of the two packed words, which is the
// per-half add exactly because no half's sum reaches 2^16 (see below), and
// keeps those rows off the half-rate pipe. Every cell lies between min(CAP,
// exact) and the exact cost, and a min3 is at most its `up` input, so the
// j-th uncapped row after a capped one holds at most CAP + j * D for
// distances of at most D. Row S-1 is capped, so runs never cross lanes:
// every value and every sum before a cap stays below 2^16, and each capped
// row -- the query's last row among them -- equals min(CAP, exact), the
// value of the all-saturating recurrence.
//   half codes:  D = kHalfSpan, RUN = 16: only row S-1 is capped
//                (28673 + 16 * 2047 = 61425);
//   large codes: D = 4094, RUN = 9 (28673 + 9 * 4094 = 65519).
constexpr int kCapRunHalf = kMaxS, kCapRunLarge = 9;
static_assert(kCap + kCapRunHalf * kHalfSpan < 65536 && kCap + kCapRunLarge * 2 * kQmax < 65536, "no carry");

// q - r per half, on half codes (exact: see kHalfSpan).
__device__ __forceinline__ uint32_t half_diff(uint32_t q, uint32_t r) {
  uint32_t d;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(q), "r"(r));
  return d;
}

// State shared by the int16 strips: the last two oblique columns, the
// reference samples moving down the lane's rows, and the two oblique columns
// of the row above the lane.
template <int S>
struct StateI16 {
  uint32_t G[2][S], Rr[kChunk];
  uint32_t gprev;

  // As if the reference began at the current step: every row, pad rows
  // included, holds CAP (infinity), and the row above a stack's top row held
  // the free-start 0 one step back (gprev). The top row then turns 0 at
  // step 0 (min(up, 0, CAP) + 0; a pad row's distance is 0), each pad row
  // below turns 0 exactly at its own first column, and a real row stays at
  // or above CAP until its first column: infinity under min(CAP, .). No
  // cell is masked; every value is the plain DP's modulo min(CAP, .), which
  // is all the tracked (capped) last row and the segment check look at.
  __device__ __forceinline__ void fresh(long, int place) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[0][k] = kCap2;
      G[1][k] = kCap2;
    }
#pragma unroll
    for (int k = 0; k < kChunk; ++k) Rr[k] = 0u;
    gprev = place ? kCap2 : 0u;
  }
  // Exact state before step t: G[1] = step t-1, G[0] = step t-2, and the
  // reference samples the cells used at step t-1 (from the global image).
  __device__ __forceinline__ void restore(const uint32_t *st, const uint32_t *gref, long t, int lane, int place) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[1][k] = __ldcg(st + k * 32 + lane);
      G[0][k] = __ldcg(st + (S + k) * 32 + lane);
      Rr[(1 + k) % kChunk] = gref[t - 1 - static_cast<long>(place) * S - k];
    }
    const uint32_t g = __shfl_up_sync(kFull, G[0][S - 1], 1);
    gprev = place ? g : 0u;
  }
  __device__ __forceinline__ void save(uint32_t *st, int lane) const {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      st[k * 32 + lane] = G[1][k];
      st[(S + k) * 32 + lane] = G[0][k];
    }
  }

  // One chunk of kChunk steps; dist(k, r) is row k's distance to the sample r.
  // A step's distances, minima and sums are three passes over the rows, and
  // neighbouring rows name the value they share (G[a][k - 1]: `up` of row k,
  // `left` of row k - 1) in the same operand place: the cell is bound by
  // register operand reads (about 1.7 a clock and scheduler over all mixes
  // measured), and this order lets a minimum reuse one of its operands.
  template <int RUN, class Dist>
  __device__ __forceinline__ void steps(const uint32_t *ref, uint32_t *ring, int e0, uint32_t ng, bool tracked,
                                        const Dist &dist) {
    LaneWindow<S> win;
#pragma unroll
    for (int u = 0; u < kChunk; ++u) {
      const int p = (kChunk - u) % kChunk;
      const int a = (u + 1) & 1;
      const int b = u & 1;
      uint32_t gup = __shfl_up_sync(kFull, G[a][S - 1], 1);
      // A stack's first lane needs the free-start row, 0, above it. Strips
      // of fewer than kMaxS rows per lane are planned with a pad row on top
      // of every stack, which stays 0 whatever comes from above (its own
      // previous value, 0, is in the minimum), so only full-height strips
      // put the zero in.
      if constexpr (S == kMaxS) gup = imad(gup, ng, 0u);
      Rr[p] = win.get(ref, u);  // row 0's reference: column t - place * S
      uint32_t d[S], m[S];
#pragma unroll
      for (int k = S - 1; k >= 0; --k) d[k] = dist(k, Rr[(p + k) % kChunk]);
#pragma unroll
      for (int k = S - 1; k >= 0; --k) {
        const uint32_t up = k ? G[a][k - 1] : gup;
        const uint32_t dg = k ? G[b][k - 1] : gprev;
        m[k] = (k & 1) ? __vimin3_u16x2(up, dg, G[a][k]) : __vimin3_u16x2(G[a][k], dg, up);
      }
#pragma unroll
      for (int k = S - 1; k >= 0; --k)
        G[b][k] = (S - 1 - k) % RUN == 0 ? __viaddmin_u16x2(d[k], m[k], kCap2) : m[k] + d[k];
      gprev = gup;
      // The last row's values of steps u - 1 and u sit in G[0] and G[1]: one
      // 8-byte store every two steps (the ring is 16-byte aligned).
      if ((u & 1) && tracked)
        *reinterpret_cast<uint2 *>(ring + e0 + u - 1) = make_uint2(G[0][S - 1], G[1][S - 1]);
    }
  }
};

// The int16 strip on half codes: the distance is one fp16x2 subtraction and
// a mask, 8 register operands a cell pair with the minimum and the sum,
// where the integer form below reads 10 and holds a second query array.
template <int S>
struct StripI16 : StateI16<S> {
  uint32_t Q[S];
  __device__ __forceinline__ void load(const uint32_t *img, int lane) {
#pragma unroll
    for (int k = 0; k < S; ++k) Q[k] = img[k * 32 + lane];
  }
  __device__ __forceinline__ void chunk(const uint32_t *ref, int, uint32_t *ring, int e0, uint32_t ng, bool tracked,
                                        int) {
    this->template steps<kCapRunHalf>(ref, ring, e0, ng, tracked, [this](int k, uint32_t r) {
      return half_diff(Q[k], r) & 0x07ff07ffu;  // the low 11 bits: |q - r|; pad rows (2^15 - r = 2^15): 0
    });
  }
};

// The int16 strip on two's complement codes of any size (|q|, |r| <= 2047).
// Pad rows carry the code -4095 in both Q and NQ: |q - r| is taken as
// relu(max(r + NQ, Q - r)) = relu(negative) = 0, so a pad row stays 0 (the
// free-start row), and real rows get max(r - q, q - r).
template <int S>
struct StripI16Large : StateI16<S> {
  uint32_t Q[S], NQ[S];
  __device__ __forceinline__ void load(const uint32_t *img, int lane) {
    constexpr uint32_t kPad2 = (static_cast<uint32_t>(kPadCode) & 0xffffu) * 0x10001u;
#pragma unroll
    for (int k = 0; k < S; ++k) {
      Q[k] = img[(S + k) * 32 + lane];
      const uint32_t pad = __vcmpeq2(Q[k], kPad2);
      NQ[k] = (__vneg2(Q[k]) & ~pad) | (kPad2 & pad);
    }
  }
  __device__ __forceinline__ void chunk(const uint32_t *ref, int, uint32_t *ring, int e0, uint32_t ng, bool tracked,
                                        int) {
    this->template steps<kCapRunLarge>(ref, ring, e0, ng, tracked, [this](int k, uint32_t r) {
      return __viaddmax_s16x2_relu(r, NQ[k], __vsub2(Q[k], r));  // |q - r| per half
    });
  }
};

// A tracker holds its best value's column as a 32-bit offset from a base that
// moves with the tiles, and in full when the base moves: references may have
// more than 2^31 columns, and a 64-bit column costs the scan two selects and
// three compares an entry.
constexpr int kNoOffset = -0x7fffffff - 1;
template <int E>  // E ring entries, read at once
struct Entries;
template <>
struct Entries<2> { using T = uint2; };
template <>
struct Entries<4> { using T = uint4; };

struct TrackI16 {
  int ba = 0x7fffffff, bb = 0x7fffffff;
  int ra = kNoOffset, rb = kNoOffset;
  long ca = -1, cb = -1, base = 0;
  __device__ __forceinline__ void rebase(long to) {
    if (ra != kNoOffset) ca = base + ra;
    if (rb != kNoOffset) cb = base + rb;
    ra = rb = kNoOffset;
    base = to;
  }
  __device__ __forceinline__ void add(uint32_t v, const uint32_t *, int rel, bool in) {
    const int va = static_cast<int>(v & 0xffffu);
    const int vb = static_cast<int>(v >> 16);
    if (in && va < ba) { ba = va; ra = rel; }
    if (in && vb < bb) { bb = vb; rb = rel; }
  }
  __device__ __forceinline__ void reduce(int width) {  // over aligned groups of `width` lanes
    for (int o = width >> 1; o > 0; o >>= 1) {
      int oa = __shfl_xor_sync(kFull, ba, o), ob = __shfl_xor_sync(kFull, bb, o);
      long pa = __shfl_xor_sync(kFull, ca, o), pb = __shfl_xor_sync(kFull, cb, o);
      if (oa < ba || (oa == ba && static_cast<unsigned long>(pa) < static_cast<unsigned long>(ca))) { ba = oa; ca = pa; }
      if (ob < bb || (ob == bb && static_cast<unsigned long>(pb) < static_cast<unsigned long>(cb))) { bb = ob; cb = pb; }
    }
  }
  __device__ __forceinline__ void merge(const Best *b);
  __device__ __forceinline__ void store(Best *b) const {
    b->ia = ba; b->ib = bb; b->f = 0.0f; b->pad = 0; b->ca = ca; b->cb = cb;
  }
};

// ----------------------------------------------------------------- FP32 --
// CODES: the reference words are int16 codes (q | q << 16) and the query
// samples are int16 codes held as floats: the exact-integer form of the
// int16 arithmetic, run through the FP32 units (see FormOf below).
template <int S, bool CODES>
struct StripF32 {
  float Q[S], W[S], G[2][S], Rr[kChunk];
  float gprev;

  __device__ __forceinline__ static float ref_value(uint32_t w) {
    if constexpr (CODES)
      return __int2float_rn(static_cast<int>(static_cast<short>(w & 0xffffu)));
    else
      return __uint_as_float(w);
  }

  __device__ __forceinline__ void load(const uint32_t *img, int lane) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      Q[k] = __uint_as_float(img[k * 32 + lane]);
      W[k] = __uint_as_float(img[(S + k) * 32 + lane]);
    }
  }
  // As if the reference began at the current step, as in the int16 strip:
  // every row, pad rows included, holds kBig (+inf; sums of these stay
  // finite), and the row above a stack's top row held the free-start 0 one
  // step back. The top row turns 0 at step 0, each pad row below at its own
  // first column, and a real row stays at kBig or above until its first
  // column whatever reference samples its lane reads before the start.
  __device__ __forceinline__ void fresh(long, int place) {
    const float kBig = 1.0e30f;
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[0][k] = kBig;
      G[1][k] = kBig;
    }
#pragma unroll
    for (int k = 0; k < kChunk; ++k) Rr[k] = 0.0f;
    gprev = place ? kBig : 0.0f;
  }
  __device__ __forceinline__ void restore(const uint32_t *st, const uint32_t *gref, long t, int lane, int place) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[1][k] = __uint_as_float(__ldcg(st + k * 32 + lane));
      G[0][k] = __uint_as_float(__ldcg(st + (S + k) * 32 + lane));
      Rr[(1 + k) % kChunk] = ref_value(gref[t - 1 - static_cast<long>(place) * S - k]);
    }
    const float g = __shfl_up_sync(kFull, G[0][S - 1], 1);
    gprev = place ? g : 0.0f;
  }
  __device__ __forceinline__ void save(uint32_t *st, int lane) const {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      st[k * 32 + lane] = __float_as_uint(G[1][k]);
      st[(S + k) * 32 + lane] = __float_as_uint(G[0][k]);
    }
  }

  __device__ __forceinline__ void chunk(const uint32_t *ref, int lane, uint32_t *ring, int e0, uint32_t ng,
                                        bool tracked, int) {
    LaneWindow<S> win;
    RingStore out;
#pragma unroll
    for (int u = 0; u < kChunk; ++u) {
      const int p = (kChunk - u) % kChunk;
      const int a = (u + 1) & 1;
      const int b = u & 1;
      float gup = __shfl_up_sync(kFull, G[a][S - 1], 1);
      // The free-start row above a stack's first lane: a pad row on top of
      // the stack (weight 0, value 0) keeps it for strips of fewer than
      // kMaxS rows per lane, as in the int16 strip.
      if constexpr (S == kMaxS) gup = ng ? gup : 0.0f;
      Rr[p] = ref_value(win.get(ref, u));  // row 0's reference: column t - place * S
#pragma unroll
      for (int k = S - 1; k >= 0; --k) {
        const float r = Rr[(p + k) % kChunk];
        // q - r rounded once on real rows (weight -1), exactly 0 on pad rows
        // (weight 0, q = 0); off the critical path, so the cost update that
        // depends on the minimum is a plain add
        const float d = __fmaf_rn(r, W[k], Q[k]);
        const float up = k ? G[a][k - 1] : gup;
        const float dg = k ? G[b][k - 1] : gprev;
        // the value shared with the row above in the same operand place, as in the int16 strips
        const float m = (k & 1) ? fmin3f(up, dg, G[a][k]) : fmin3f(G[a][k], dg, up);
        G[b][k] = __fadd_rn(fabsf(d), m);
      }
      gprev = gup;
      out.put(ring, e0, u, tracked, __float_as_uint(G[b][S - 1]));
    }
  }
};

struct TrackF32 {
  float best;
  int rel_best = kNoOffset;
  long col = -1, base = 0;
  __device__ TrackF32() : best(__builtin_huge_valf()) {}
  __device__ __forceinline__ void rebase(long to) {
    if (rel_best != kNoOffset) col = base + rel_best;
    rel_best = kNoOffset;
    base = to;
  }
  __device__ __forceinline__ void add(uint32_t v, const uint32_t *, int rel, bool in) {
    const float f = __uint_as_float(v);
    if (in && f < best) { best = f; rel_best = rel; }
  }
  __device__ __forceinline__ void reduce(int width) {  // over aligned groups of `width` lanes
    for (int o = width >> 1; o > 0; o >>= 1) {
      float ob = __shfl_xor_sync(kFull, best, o);
      long oc = __shfl_xor_sync(kFull, col, o);
      if (ob < best || (ob == best && static_cast<unsigned long>(oc) < static_cast<unsigned long>(col))) {
        best = ob;
        col = oc;
      }
    }
  }
  __device__ __forceinline__ void merge(const Best *b);
  __device__ __forceinline__ void store(Best *b) const {
    b->ia = 0; b->ib = 0; b->f = best; b->pad = 0; b->ca = col; b->cb = -1;
  }
};

// ------------------------------------------------------ start columns --
// The FP32 strip that also carries each cell's alignment start column: a
// cell takes the start of its up neighbour if that is a minimum
// predecessor, else of its diagonal one if that is, else of its left one.
// Pad rows (weight 0, cost 0) take their up neighbour's start on the cost
// tie, so they pass down "my own column" from the row injected above the
// first lane of a stack (the row above row i processed column t - i at
// step t - 1); the first real row therefore starts its paths at its own
// column, like the free-start row of Eq. 1. CODES as for StripF32.
constexpr int kUnknownStart = -2147483647 - 1;
template <int S, bool CODES>
struct StripF32Span {
  float Q[S], W[S], G[2][S], Rr[kChunk];
  int P[2][S];
  float gprev;
  int pprev;

  __device__ __forceinline__ static float ref_value(uint32_t w) {
    if constexpr (CODES)
      return __int2float_rn(static_cast<int>(static_cast<short>(w & 0xffffu)));
    else
      return __uint_as_float(w);
  }
  __device__ __forceinline__ void load(const uint32_t *img, int lane) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      Q[k] = __uint_as_float(img[k * 32 + lane]);
      W[k] = __uint_as_float(img[(S + k) * 32 + lane]);
    }
  }
  // As in StripF32: every row starts at kBig and the free-start zero reaches
  // each row at its first column (a stack's top row takes the injected row
  // above it, 0 with the current column, every step), so each pad row passes
  // down its own column from then on. Before step t_start row i = place * S +
  // k of a stack held column t_start - 1 - i (t_start - 2 - i one step earlier); those
  // starts belong to values at kBig, which no finite cost takes.
  __device__ __forceinline__ void fresh(long t_start, int place) {
    const float kBig = 1.0e30f;
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[0][k] = kBig;
      G[1][k] = kBig;
      const int i = place * S + k;
      P[1][k] = static_cast<int>(t_start) - 1 - i;
      P[0][k] = static_cast<int>(t_start) - 2 - i;
    }
#pragma unroll
    for (int k = 0; k < kChunk; ++k) Rr[k] = 0.0f;
    gprev = place ? kBig : 0.0f;
    pprev = static_cast<int>(t_start) - 1 - place * S;  // the row above row 0 at step t_start - 2
  }
  // States hold G (2S rows of 32 words) then P (2S rows).
  __device__ __forceinline__ void restore(const uint32_t *st, const uint32_t *gref, long t, int lane, int place) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[1][k] = __uint_as_float(__ldcg(st + k * 32 + lane));
      G[0][k] = __uint_as_float(__ldcg(st + (S + k) * 32 + lane));
      P[1][k] = static_cast<int>(__ldcg(st + (2 * S + k) * 32 + lane));
      P[0][k] = static_cast<int>(__ldcg(st + (3 * S + k) * 32 + lane));
      Rr[(1 + k) % kChunk] = ref_value(gref[t - 1 - static_cast<long>(place) * S - k]);
    }
    const float g = __shfl_up_sync(kFull, G[0][S - 1], 1);
    const int pg = __shfl_up_sync(kFull, P[0][S - 1], 1);
    gprev = place ? g : 0.0f;
    pprev = place ? pg : static_cast<int>(t) - 1;
  }
  // A cost form's exact state before step t: every start column before it is
  // kUnknownStart; the free-start rows pass known ones down from step t on.
  __device__ __forceinline__ void restore_costs(const uint32_t *st, const uint32_t *gref, long t, int lane,
                                                int place) {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      G[1][k] = __uint_as_float(__ldcg(st + k * 32 + lane));
      G[0][k] = __uint_as_float(__ldcg(st + (S + k) * 32 + lane));
      P[1][k] = kUnknownStart;
      P[0][k] = kUnknownStart;
      Rr[(1 + k) % kChunk] = ref_value(gref[t - 1 - static_cast<long>(place) * S - k]);
    }
    const float g = __shfl_up_sync(kFull, G[0][S - 1], 1);
    gprev = place ? g : 0.0f;
    pprev = kUnknownStart;
  }
  __device__ __forceinline__ void save(uint32_t *st, int lane) const {
#pragma unroll
    for (int k = 0; k < S; ++k) {
      st[k * 32 + lane] = __float_as_uint(G[1][k]);
      st[(S + k) * 32 + lane] = __float_as_uint(G[0][k]);
      st[(2 * S + k) * 32 + lane] = static_cast<uint32_t>(P[1][k]);
      st[(3 * S + k) * 32 + lane] = static_cast<uint32_t>(P[0][k]);
    }
  }

  // t0: the absolute step of the chunk's first step. The ring's start columns
  // sit two flush buffers after the costs.
  __device__ __forceinline__ void chunk(const uint32_t *ref, int lane, uint32_t *ring, int e0, uint32_t ng,
                                        bool tracked, int t0) {
    LaneWindow<S> win;
#pragma unroll
    for (int u = 0; u < kChunk; ++u) {
      const int p = (kChunk - u) % kChunk;
      const int a = (u + 1) & 1;
      const int b = u & 1;
      float gup = __shfl_up_sync(kFull, G[a][S - 1], 1);
      int pup = __shfl_up_sync(kFull, P[a][S - 1], 1);
      gup = ng ? gup : 0.0f;             // a stack's first lane: the free-start row, 0 ...
      pup = ng ? pup : t0 + u;            // ... whose row processed column t at step t - 1
      Rr[p] = ref_value(win.get(ref, u));  // row 0's reference: column t - place * S
#pragma unroll
      for (int k = S - 1; k >= 0; --k) {
        const float r = Rr[(p + k) % kChunk];
        const float d = __fmaf_rn(r, W[k], Q[k]);  // q - r on real rows, 0 on pad rows
        const float up = k ? G[a][k - 1] : gup;
        const int pu = k ? P[a][k - 1] : pup;
        const float dg = k ? G[b][k - 1] : gprev;
        const int pd = k ? P[b][k - 1] : pprev;
        const float m = fmin3f(up, dg, G[a][k]);
        // The start of the preferred minimum predecessor: up, else diagonal, else left.
        G[b][k] = __fadd_rn(fabsf(d), m);
        P[b][k] = sel_eq(up, m, pu, sel_eq(dg, m, pd, P[a][k]));
      }
      gprev = gup;
      pprev = pup;
      if (tracked) {
        ring[e0 + u] = __float_as_uint(G[b][S - 1]);
        ring[2 * flush_words(kPrecF32Span) + e0 + u] = static_cast<uint32_t>(P[b][S - 1]);
      }
    }
  }
};

struct TrackF32Span {
  float best;
  int rel_best = kNoOffset;
  long col = -1, base = 0;
  int start = -1;
  __device__ TrackF32Span() : best(__builtin_huge_valf()) {}
  __device__ __forceinline__ void rebase(long to) {
    if (rel_best != kNoOffset) col = base + rel_best;
    rel_best = kNoOffset;
    base = to;
  }
  __device__ __forceinline__ void add(uint32_t v, const uint32_t *entry, int rel, bool in) {
    const float f = __uint_as_float(v);
    if (in && f < best) { best = f; rel_best = rel; start = static_cast<int>(entry[2 * flush_words(kPrecF32Span)]); }
  }
  __device__ __forceinline__ void reduce(int width) {  // over aligned groups of `width` lanes
    for (int o = width >> 1; o > 0; o >>= 1) {
      float ob = __shfl_xor_sync(kFull, best, o);
      long oc = __shfl_xor_sync(kFull, col, o);
      int os = __shfl_xor_sync(kFull, start, o);
      if (ob < best || (ob == best && static_cast<unsigned long>(oc) < static_cast<unsigned long>(col))) {
        best = ob;
        col = oc;
        start = os;
      }
    }
  }
  __device__ __forceinline__ void merge(const Best *b);
  __device__ __forceinline__ void store(Best *b) const {
    b->ia = 0; b->ib = 0; b->f = best; b->pad = 0; b->ca = col; b->cb = start;
  }
};

// Arithmetic forms of a strip: FP32 queries, int16 pairs (DPX), and int16
// codes computed exactly without saturation: wide accumulation (every cost
// of a query of <= 512 events is an integer below 512 * 4094 < 2^24, so FP32
// holds it exactly).
constexpr int kFormF32 = 0, kFormI16 = 1, kFormI16Large = 2, kFormExactWide = 3;
constexpr bool form_i16(int form) { return form == kFormI16 || form == kFormI16Large; }
// and the FP32 and wide forms carrying the start column
constexpr int kFormF32Span = 4, kFormWideSpan = 5;
// Rows of 32 words in a saved strip state, per strip row: two oblique
// columns of costs, and of start columns in the span forms.
template <int FORM>
constexpr int state_rows_per_s() { return (FORM == kFormF32Span || FORM == kFormWideSpan) ? 4 : 2; }

template <int FORM, int S>
struct FormOf;
template <int S>
struct FormOf<kFormI16, S> {
  using Strip = StripI16<S>;
  using Track = TrackI16;
};
template <int S>
struct FormOf<kFormI16Large, S> {
  using Strip = StripI16Large<S>;
  using Track = TrackI16;
};
template <int S>
struct FormOf<kFormF32, S> {
  using Strip = StripF32<S, false>;
  using Track = TrackF32;
};
template <int S>
struct FormOf<kFormExactWide, S> {
  using Strip = StripF32<S, true>;
  using Track = TrackF32;
};
template <int S>
struct FormOf<kFormF32Span, S> {
  using Strip = StripF32Span<S, false>;
  using Track = TrackF32Span;
};
template <int S>
struct FormOf<kFormWideSpan, S> {
  using Strip = StripF32Span<S, true>;
  using Track = TrackF32Span;
};

// ----------------------------------------------------------- tile sources --
// Shared state of one tile stream (a CTA's, or each warp's own).
struct Stream {
  uint64_t full[2];
  int cnt[2];
  int uses[2];
  int tile_base;
  int pad[3];
};
// Shared state of one CTA.
struct Shared {
  int group;
  int abort;
  int stop;
  int pad;
  Stream streams[kMaxWarps];
  Schedule sched;
};
static_assert(sizeof(Shared) <= kSharedHeader, "shared-memory header");

// Reference tiles streamed into shared memory by TMA (the sweep kernel).
// Slot of tile k: the kRefFront columns before the tile, then its
// tile_cols columns, so a lane that reads up to 31 * S columns behind the
// warp's step finds its samples in the current slot.
struct TileStream {
  Stream *sh;
  int *abort;                  // the CTA's
  char *slots;                 // two slots of tile_cols + kRefFront words
  const char *src;             // reference image (column 0; kRefFront zero words before it)
  int tile_cols;               // T_S
  int k_first;                 // first global tile of this group's steps
  int K;                       // tiles in this group's sweep
  int n_active;                // warps consuming this stream
  unsigned long long wait_ns;  // longest single wait
  int *ints;

  __device__ void issue(int k) {  // one thread
    const int gk = sh->tile_base + k;
    const int slot = gk & 1;
    const unsigned words = static_cast<unsigned>(tile_cols + kRefFront);
    const unsigned bytes = words * 4u;
    // from column (k_first + k) * tile_cols - kRefFront >= -kRefFront: the
    // image's front pad; 16-byte aligned (tile_cols and kRefFront are
    // multiples of 4 words)
    const long first = static_cast<long>(k_first + k) * tile_cols - kRefFront;
    fence_proxy_async();
    mbar_expect_tx(&sh->full[slot], bytes);
    tma_load_1d(slots + static_cast<size_t>(slot) * words * 4, src + first * 4, bytes, &sh->full[slot]);
    sh->uses[slot] += 1;
  }
  __device__ const uint32_t *acquire(int k) {  // whole warp
    const int gk = sh->tile_base + k;
    const int slot = gk & 1;
    if (!mbar_wait_bounded(&sh->full[slot], (gk >> 1) & 1, now_ns() + wait_ns)) {
      report(ints + kIntStatus, HARU_ETIMEDOUT);
      ints[kIntAbort] = 1;
      *abort = 1;
      return nullptr;
    }
    return reinterpret_cast<const uint32_t *>(slots + static_cast<size_t>(slot) * (tile_cols + kRefFront) * 4);
  }
  __device__ void release(int k) {  // lane 0 of a warp
    const int gk = sh->tile_base + k;
    const int slot = gk & 1;
    __threadfence_block();
    const int old = atomicAdd(&sh->cnt[slot], 1);
    if (old == n_active - 1) {
      sh->cnt[slot] = 0;
      __threadfence_block();
      if (k + 2 < K) issue(k + 2);
    }
  }
};

// The reference read straight from global memory (the fix-up kernel), in
// the same layout as a tile slot: the pointer of tile k is at the column
// kRefFront before the tile (inside the image's front pad for tile 0).
struct GlobalTiles {
  const uint32_t *img;
  int tile_cols;
  long k_first;
  __device__ __forceinline__ const uint32_t *acquire(int k) {
    return img + ((k_first + k) * tile_cols - kRefFront);
  }
  __device__ __forceinline__ void release(int) {}
};

// ------------------------------------------------------------ one unit --
// Runs steps [t_start, t_end) of one strip (a query or a pair) and tracks
// the last row over own steps [t_own, t_end).
// save_start / save_final: where to store the state before step t_own and
// before step t_end (nullptr: not stored). stk: a stacked item (lanes 0..15
// and 16..31 are two strips; each lane tracks its own stack's last row).
// `ring` holds ring_words() words per warp: two flush buffers of W =
// flush_words() words, each filled by the strip's tracked lane between two
// scans (or half by each stack's, the lower stack's at +W/2); forms that
// carry start columns keep them 2W further on. Each flush scans W/32
// neighbouring entries per lane, one vector load, against the range of
// columns that count: with 64-bit columns and a load, a bounds test and
// a branch per entry 8,192 uneven queries took 11.84 (int16) and 20.06 ms
// (FP32), so 11.44 and 19.64 (at the same schedule).
// Returns false on abort.
// With checkpoints (A.checkpoints, cost forms) the state before every
// checkpoint step of the own range is stored too.
template <int FORM, int S, class Src, class Track>
__device__ bool run_steps(const SdtwArgs &A, int item, typename FormOf<FORM, S>::Strip &st, Track &tr, Src &src,
                          int TS, long t_start, long t_own, long t_end, uint32_t *save_start, uint32_t *save_final,
                          uint32_t *ring, int lane, bool stk) {
  constexpr bool kCheckpoints = FORM == kFormF32 || FORM == kFormExactWide;
  const long N = A.N;
  constexpr int W = flush_words(form_i16(FORM) ? HARU_INT16 : HARU_FP32);
  // chunks between two flushes: a stack's entries fill its share of a buffer
  constexpr int kWhole = W / kChunk, kHalf = W / 2 / kChunk;
  static_assert(kHalf > 0 && kChunk % 4 == 0, "whole chunks, vector stores");
  constexpr int E = W / 32;  // entries of a lane's scan
  const int F = stk ? kHalf : kWhole;
  const int place = stack_place(lane, stk);
  const uint32_t ng = place != 0 ? 1u : 0u;  // 0 on a lane that starts a stack from the free-start row
  const bool tracked = lane == 31 || (stk && lane == 15);
  const int soff = stk && lane >= 16 ? W / 2 : 0;
  const long last_row = (stk ? 16L : 32L) * S - 1;  // of either stack
  const long k_first = t_start / TS;
  const int K = static_cast<int>((t_end + TS - 1) / TS - k_first);
  int fl = 0, buf = 0;
  const long first_col = t_own > last_row ? t_own - last_row : 0;
  for (int k = 0; k < K; ++k) {
    const uint32_t *tile = src.acquire(k);
    if (!tile) return false;
    // This tile's steps [lo, hi), walked in 32-bit offsets from lo.
    const long tk0 = (k_first + k) * TS;
    const long lo = tk0 > t_start ? tk0 : t_start;
    const long hi = tk0 + TS < t_end ? tk0 + TS : t_end;
    const int n = static_cast<int>(hi - lo);
    const int own_at = (save_start && t_own >= lo && t_own < hi) ? static_cast<int>(t_own - lo) : -1;
    const bool last_tile = t_end <= tk0 + TS;
    // columns as offsets from that of step lo: the buffer's first, the first and the end of those that count
    const long base = lo - last_row;
    tr.rebase(base);
    int fcol = -fl * kChunk;
    const long far = 1L << 30;
    const int col_lo = static_cast<int>(min(max(first_col - base, -far), far));
    const int col_hi = static_cast<int>(min(max(N - base, -far), far));
    // this lane's reference window of the chunk at o: columns from
    // lo + o - place * S, found at (column - tk0 + kRefFront) in the slot;
    // place * S <= 31 * kMaxS <= kRefFront keeps it inside the slot
    const uint32_t *tref = tile + (kRefFront + (lo - tk0) - static_cast<long>(place) * S);
    // the next step of this tile before which a state is stored
    auto next_save = [&](int from) {
      int at = own_at >= from ? own_at : n;
      if constexpr (kCheckpoints) {
        if (A.checkpoints) {
          const long D = checkpoint_steps(A.checkpoint_step);
          const long first = lo + from > t_own ? lo + from : t_own;
          const long c = (first + D - 1) / D * D - lo;
          if (c < at) at = static_cast<int>(c);
        }
      }
      return at;
    };
    int save_at = next_save(0);
    for (int o = 0; o < n; o += kChunk) {
      if (o == save_at) {
        if (o == own_at) st.save(save_start, lane);
        if constexpr (kCheckpoints) {
          if (A.checkpoints) {
            const int D = checkpoint_steps(A.checkpoint_step);
            const long c = (lo + o) / D;  // (checkpoint 0 is the fresh start)
            if (c * D == lo + o && lo + o >= t_own && c > 0 && c <= A.checkpoint_cap)
              st.save(A.checkpoints + (static_cast<size_t>(item) * A.checkpoint_cap + (c - 1)) * kStateStride, lane);
          }
        }
        save_at = next_save(o + kChunk);
      }
      uint32_t *rg = ring + buf * W + soff;
      const int tabs = static_cast<int>(lo) + o;
      st.chunk(tref + o, lane, rg, fl * kChunk, ng, tracked, tabs);
      if (++fl == F || (last_tile && o + kChunk >= n)) {
        __syncwarp();
        // entry j of the buffer: column fcol + j of this lane's stack
        const int j0 = place * E, hi_col = min(col_hi, fcol + fl * kChunk);
        const unsigned ncol = static_cast<unsigned>(max(hi_col - col_lo, 0));
        const typename Entries<E>::T v = *reinterpret_cast<const typename Entries<E>::T *>(rg + j0);
        const int rel = fcol + j0;
#pragma unroll
        for (int e = 0; e < E; ++e)
          tr.add(reinterpret_cast<const uint32_t *>(&v)[e], rg + j0 + e, rel + e,
                 static_cast<unsigned>(rel + e - col_lo) < ncol);
        fcol += fl * kChunk;
        fl = 0;
        buf ^= 1;
      }
    }
    __syncwarp();
    if (lane == 0) src.release(k);
  }
  tr.rebase(0);
  if (save_final) st.save(save_final, lane);
  return true;
}

// Merge a unit's later steps' minimum with its earlier ones': the smaller
// cost, the earlier (smaller) column on a tie.
__device__ __forceinline__ void TrackI16::merge(const Best *b) {
  const int ia = __ldcg(&b->ia), ib = __ldcg(&b->ib);
  if (ia <= ba) { ba = ia; ca = __ldcg(&b->ca); }
  if (ib <= bb) { bb = ib; cb = __ldcg(&b->cb); }
}
__device__ __forceinline__ void TrackF32::merge(const Best *b) {
  const float f = __ldcg(&b->f);
  if (f <= best) { best = f; col = __ldcg(&b->ca); }
}
__device__ __forceinline__ void TrackF32Span::merge(const Best *b) {
  const float f = __ldcg(&b->f);
  if (f <= best) { best = f; col = __ldcg(&b->ca); start = static_cast<int>(__ldcg(&b->cb)); }
}

// Steps [p_lo, p_hi) of the sweep of one unit (item, segment). From the
// segment's start they start from the fresh state, otherwise from the state
// that the steps before them saved as the unit's last one, where its final
// state goes too.
template <int FORM, int S>
__device__ void sweep_unit(const SdtwArgs &A, TileStream &ts, int nseg, int seg, long p_lo, long p_hi, int item,
                           uint32_t *ring, int lane) {
  typename FormOf<FORM, S>::Strip st;
  typename FormOf<FORM, S>::Track tr;
  st.load(A.img + static_cast<size_t>(item) * kImgStride, lane);
  long t_start, t_own, t_end;
  seg_bounds(S, nseg, seg, A.N, &t_start, &t_own, &t_end);
  const bool stk = A.items[item].stacked != 0;
  // (start-column units are never cut)
  const bool whole = FORM == kFormF32Span || FORM == kFormWideSpan || p_lo == t_start;
  const int place = stack_place(lane, stk);
  const size_t unit = static_cast<size_t>(item) * A.nseg_cap + seg;
  constexpr size_t kWords = state_rows_per_s<FORM>() * 16 * 32;
  uint32_t *ss = nullptr, *sf = nullptr;
  if (seg > 0) ss = A.states + (unit * 2 + 0) * kWords;
  if (seg + 1 < nseg || p_hi < t_end) sf = A.states + (unit * 2 + 1) * kWords;
  if (whole)
    st.fresh(t_start, place);
  else
    st.restore(A.states + (unit * 2 + 1) * kWords, reinterpret_cast<const uint32_t *>(ts.src), p_lo, lane, place);
  const bool ok = run_steps<FORM, S>(A, item, st, tr, ts, ts.tile_cols, p_lo, t_own, p_hi, ss, sf, ring, lane, stk);
  tr.reduce(stk ? 16 : 32);
  if (ok && lane == 0) {
    if (!whole) tr.merge(A.bests + unit);
    tr.store(A.bests + unit);
  }
  if (ok && stk && lane == 16) {
    if (!whole) tr.merge(A.bests2 + unit);
    tr.store(A.bests2 + unit);
  }
}

template <int PREC, int S>
__device__ __forceinline__ void sweep_any(const SdtwArgs &A, TileStream &ts, int nseg, int seg, long p_lo,
                                          long p_hi, int item, bool large, uint32_t *ring, int lane) {
  if constexpr (PREC == HARU_FP32) {
    sweep_unit<kFormF32, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  } else if constexpr (PREC == HARU_INT16_ACC32) {
    sweep_unit<kFormExactWide, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  } else if constexpr (PREC == kPrecF32Span) {
    sweep_unit<kFormF32Span, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  } else if constexpr (PREC == kPrecWideSpan) {
    sweep_unit<kFormWideSpan, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  } else if constexpr (PREC == kPrecI16Mixed) {
    if (large)
      sweep_unit<kFormI16Large, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
    else
      sweep_unit<kFormI16, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  } else {
    sweep_unit<kFormI16, S>(A, ts, nseg, seg, p_lo, p_hi, item, ring, lane);
  }
}

// Hand-over of the bundle across a border of the schedule (one thread,
// between CTA barriers): the states and minima written before finish_part are
// seen after wait_part.
__device__ __forceinline__ void finish_part(const SdtwArgs &A, int cta) {
  __threadfence();
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(A.done + cta), "r"(1) : "memory");
}
__device__ __forceinline__ bool wait_part(const SdtwArgs &A, int cta, unsigned long long limit_ns) {
  const unsigned long long deadline = now_ns() + limit_ns;
  for (;;) {
    int n;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(n) : "l"(A.done + cta) : "memory");
    if (n) break;
    if (*static_cast<volatile int *>(A.ints + kIntAbort)) return false;  // a CTA gave up: its part never finishes
    if (now_ns() > deadline) {
      report(A.ints + kIntStatus, HARU_ETIMEDOUT);
      A.ints[kIntAbort] = 1;
      return false;
    }
    __nanosleep(200);
  }
  __threadfence();
  return true;
}

// One kernel covers every strip height S = 1..16 (registers are allocated
// for the tallest).
template <int PREC, int S = 1>
__device__ __forceinline__ void dispatch_sweep(int s, const SdtwArgs &A, TileStream &ts, int nseg, int seg,
                                               long p_lo, long p_hi, int item, bool large, uint32_t *ring,
                                               int lane) {
  if constexpr (S <= kMaxS) {
    if (s == S)
      sweep_any<PREC, S>(A, ts, nseg, seg, p_lo, p_hi, item, large, ring, lane);
    else
      dispatch_sweep<PREC, S + 1>(s, A, ts, nseg, seg, p_lo, p_hi, item, large, ring, lane);
  }
}

// Up to 12 warps per CTA (3 per scheduler): the int16, FP32 and wide strips
// fit in 168 registers a thread; the start-column strips (~240) up to 8.
template <int PREC>
__host__ __device__ constexpr int cta_threads() { return prec_span(PREC) ? 256 : 384; }

// The CTA's shared state and this warp's tile slots; layout: Shared |
// per-warp tracking rings | two tile slots per stream.
__device__ __forceinline__ void init_shared(Shared *sh) {
  if (threadIdx.x < kMaxWarps) {
    Stream *t = &sh->streams[threadIdx.x];
    mbar_init(&t->full[0], 1);
    mbar_init(&t->full[1], 1);
    t->cnt[0] = t->cnt[1] = 0;
    t->uses[0] = t->uses[1] = 0;
    t->tile_base = 0;
    if (threadIdx.x == 0) sh->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}
template <int PREC>
__device__ __forceinline__ TileStream stream_of(const SdtwArgs &A, Shared *sh, int stream, int S, long p_lo, long p_hi,
                                                int n_active, bool large) {
  char *slots = reinterpret_cast<char *>(sh) + kSharedHeader + A.warps * ring_words(PREC) * 4;
  const int TS = tile_width(A.tile_cols);
  TileStream ts;
  ts.sh = &sh->streams[stream];
  ts.abort = &sh->abort;
  ts.slots = slots + static_cast<size_t>(stream) * 2 * (A.tile_cols + kRefFront) * 4;
  ts.src = reinterpret_cast<const char *>(PREC == kPrecI16Mixed && large ? A.ref_large : A.ref_img);
  ts.tile_cols = TS;
  ts.k_first = static_cast<int>(p_lo / TS);
  ts.K = static_cast<int>((p_hi + TS - 1) / TS - p_lo / TS);
  ts.n_active = n_active;
  ts.wait_ns = A.wait_ns;
  ts.ints = A.ints;
  return ts;
}
// On abort, wait (bounded) for this CTA's copies still in flight before exit.
__device__ __forceinline__ void drain_streams(const SdtwArgs &A, Shared *sh) {
  __syncthreads();
  if (threadIdx.x < kMaxWarps && sh->abort) {
    Stream *t = &sh->streams[threadIdx.x];
    const unsigned long long dl = now_ns() + A.wait_ns;
    for (int s = 0; s < 2; ++s)
      if (t->uses[s] > 0) mbar_wait_bounded(&t->full[s], (t->uses[s] - 1) & 1, dl);
  }
}

// Groups from the queue: a CTA's warps sweep one segment, sharing one tile
// stream. (A kernel apart from the scheduled sweep below: in one kernel the
// start-column strips ran 10-20% longer a step.)
template <int PREC>
__global__ void __launch_bounds__(cta_threads<PREC>(), 1) queue_kernel(SdtwArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  Shared *sh = reinterpret_cast<Shared *>(smem);
  uint32_t *rings = reinterpret_cast<uint32_t *>(smem + kSharedHeader);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  init_shared(sh);
  const int count = A.ints[kIntGroups];
  for (;;) {
    if (threadIdx.x == 0) sh->group = atomicAdd(A.ints + kIntQueue, 1);
    __syncthreads();
    const int gi = sh->group;
    if (gi >= count || sh->abort) break;
    const Group grp = A.groups[gi];
    bool large = false;  // the group holds a code too large for the half-code cell
    if constexpr (PREC == kPrecI16Mixed)
      large = __any_sync(kFull, A.items[grp.first + min(lane, grp.count - 1)].qmax > A.half_max);
    long t_start, t_own, t_end;
    seg_bounds(grp.S, grp.nseg, grp.seg, A.N, &t_start, &t_own, &t_end);
    TileStream ts = stream_of<PREC>(A, sh, 0, grp.S, t_start, t_end, grp.count, large);
    if (threadIdx.x == 0) {
      ts.issue(0);
      if (ts.K > 1) ts.issue(1);
    }
    __syncthreads();
    if (warp < grp.count)
      dispatch_sweep<PREC>(grp.S, A, ts, grp.nseg, grp.seg, t_start, t_end, grp.first + warp, large,
                           rings + warp * ring_words(PREC), lane);
    __syncthreads();
    if (threadIdx.x == 0) ts.sh->tile_base += ts.K;
  }
  drain_streams(A, sh);
}

// The bundle at place x of the schedule's line: the number of bundles that
// end at or before x; *inside: x lies within that bundle, not at its start.
__device__ __forceinline__ int bundle_at(const Schedule &c, long long x, bool *inside) {
  *inside = false;
  if (x >= c.total) return c.bundles;
  for (int k = 2 * kMaxS - 1; k >= 0; --k) {
    const ScheduleRow &r = c.row[k];
    if (r.bundles == 0) continue;
    const long long y = x - r.start;
    if (y >= (r.bundles - 1) * r.cost + r.last_cost) continue;
    const int i = min(static_cast<int>(y / r.cost), r.bundles - 1);
    *inside = y > i * r.cost;
    return r.bundle0 + i;
  }
  return c.bundles;
}
// The row of bundle b.
__device__ __forceinline__ const ScheduleRow &find_row(const Schedule &c, int b, int *S) {
  int k = 2 * kMaxS - 1;
  while (k > 0 && b >= c.row[k].bundle0 + c.row[k].bundles) --k;
  *S = k / 2 + 1;
  return c.row[k];
}

// The static schedule: this CTA's stretch of it, each warp with its own tile
// stream.
template <int PREC>
__global__ void __launch_bounds__(cta_threads<PREC>(), 1) sdtw_kernel(SdtwArgs A) {
  extern __shared__ __align__(128) unsigned char smem[];
  Shared *sh = reinterpret_cast<Shared *>(smem);
  uint32_t *rings = reinterpret_cast<uint32_t *>(smem + kSharedHeader);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // This CTA's place on the line, in the order the CTAs started, and the
  // bundles first .. first + n - 1 that its stretch touches.
  const Schedule &sched = sh->sched;
  if (threadIdx.x == 0) sh->group = atomicAdd(A.ints + kIntQueue, 1);
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(Schedule) / 4); i += blockDim.x)
    reinterpret_cast<int *>(&sh->sched)[i] = reinterpret_cast<const int *>(A.sched)[i];
  init_shared(sh);
  const int place = sh->group;
  bool left, right;  // the first / last of them crosses a border
  const int first = bundle_at(sched, place * sched.share, &left);
  const int n = bundle_at(sched, (place + 1) * sched.share, &right) - first + (right ? 1 : 0);
  for (int e = 0; e < n; ++e) {
    // the bundle across the right border first, the one across the left border last
    const int next = first + (right ? (e == 0 ? n - 1 : e - 1 + (left ? 1 : 0)) : e + (left ? 1 : 0));
    const int b = next >= first + n - (right && e > 0 ? 1 : 0) ? first : next;
    int S;
    const ScheduleRow &row = find_row(sched, b, &S);
    const int i = b - row.bundle0;
    const long long cost = i + 1 < row.bundles ? row.cost : row.last_cost;
    const long long cut_lo = place * sched.share - (row.start + i * row.cost), cut_hi = cut_lo + sched.share;
    const bool waits = left && b == first, hands = right && b == first + n - 1;
    const int members = i + 1 < row.bundles ? sched.members : row.last;
    const int u0 = i * sched.members, u = u0 + min(warp, members - 1);  // this warp's unit
    const int item = row.base + u % row.items, seg = u / row.items, nseg = row.nseg;
    bool large = false;  // the bundle holds a code too large for the half-code cell
    if constexpr (PREC == kPrecI16Mixed)
      large = __any_sync(kFull, A.items[row.base + (u0 + min(lane, members - 1)) % row.items].qmax > A.half_max);
    long t_start, t_own, t_end;
    seg_bounds(S, nseg, seg, A.N, &t_start, &t_own, &t_end);
    const long p_lo = t_start + cut_steps(t_start, t_end, cut_lo, cost);
    const long p_hi = t_start + cut_steps(t_start, t_end, cut_hi, cost);
    if (waits) {
      // the CTA placed before this one ran its part of the bundle first (a step takes well under 1 us)
      if (threadIdx.x == 0)
        sh->stop = !wait_part(A, place - 1, A.wait_ns + 1000ull * static_cast<unsigned long long>(t_end - t_start));
      __syncthreads();
      if (sh->stop) break;
    }
    // (after a wait that gave up, this CTA's streams are not used again)
    const bool runs = warp < members && p_lo < p_hi && !__any_sync(kFull, *static_cast<volatile int *>(&sh->abort));
    if (runs) {
      TileStream ts = stream_of<PREC>(A, sh, warp, S, p_lo, p_hi, 1, large);
      if (lane == 0) {
        ts.issue(0);
        if (ts.K > 1) ts.issue(1);
      }
      __syncwarp();
      dispatch_sweep<PREC>(S, A, ts, nseg, seg, p_lo, p_hi, item, large, rings + warp * ring_words(PREC), lane);
      __syncwarp();
      if (lane == 0) ts.sh->tile_base += ts.K;
    }
    if (hands) {
      __syncthreads();
      if (threadIdx.x == 0 && !sh->abort) finish_part(A, place);
    }
  }
  drain_streams(A, sh);
}

// --------------------------------------------------------------- fix-up --
// Verifies every segment boundary, recomputes segments whose speculative
// start state differs from the exact one, combines the segments' last-row
// minima (smallest cost, then smallest column) and writes the outputs.
//
// One CTA per item and kFixWarps segments: each warp compares one boundary
// (latency bound: 4S independent 128-byte loads), the item's last CTA to
// finish reads the verdicts, and its first warp does the rest. One warp per
// item that walked the boundaries in turn took 89 us where this takes 9 (51
// int16 items of up to 29 segments) and 734 us where this takes 36 (128 items of 57).
template <int FORM>
__device__ __forceinline__ void write_out(const SdtwArgs &A, const Best &b, int qa, int qb) {
  if (qa < 0) return;
  if (form_i16(FORM)) {
    A.out_cost[qa] = static_cast<float>(b.ia) * A.inv_scale;
    A.out_col[qa] = b.ca;
    if (qb >= 0) {
      A.out_cost[qb] = static_cast<float>(b.ib) * A.inv_scale;
      A.out_col[qb] = b.cb;
    }
  } else if (FORM == kFormExactWide || FORM == kFormWideSpan) {
    A.out_cost[qa] = b.f * A.inv_scale;
    A.out_col[qa] = b.ca;
  } else {
    A.out_cost[qa] = b.f;
    A.out_col[qa] = b.ca;
  }
  if (FORM == kFormF32Span || FORM == kFormWideSpan) A.out_start[qa] = b.cb;
}

// Whether segment s of an item started from the state the segment before it
// ended in (whole warp): costs, and start columns in the span forms; int16
// equal modulo min(CAP, .), which fixes every later capped value.
template <int FORM>
__device__ __forceinline__ bool boundary_exact(const SdtwArgs &A, size_t base, int s, int S, int lane) {
  constexpr int kRows = state_rows_per_s<FORM>();
  constexpr size_t kWords = kRows * 16 * 32;
  const uint32_t *exact = A.states + ((base + s - 1) * 2 + 1) * kWords + lane;
  const uint32_t *spec = A.states + ((base + s) * 2 + 0) * kWords + lane;
  unsigned diff = 0;
#pragma unroll 8
  for (int k = 0; k < kRows * S; ++k) {
    const uint32_t x = exact[k * 32], y = spec[k * 32];
    diff |= form_i16(FORM) ? __vminu2(x, kCap2) ^ __vminu2(y, kCap2) : x ^ y;
  }
  return __all_sync(kFull, diff == 0);
}

// Recompute, in order, every segment whose start state is not the exact one
// (one warp): those marked, and those after a recomputed segment that the
// new final state does not reach either.
template <int FORM, int S>
__device__ void recompute_segments(const SdtwArgs &A, int item, uint32_t *ring, int lane) {
  const Item it = A.items[item];
  const int nseg = it.nseg;
  const bool stk = it.stacked != 0;
  const uint32_t *ref = static_cast<const uint32_t *>(FORM == kFormI16Large ? A.ref_large : A.ref_img);
  const size_t base = static_cast<size_t>(item) * A.nseg_cap;
  const int TS = tile_width(A.tile_cols);
  const int place = stack_place(lane, stk);
  constexpr size_t kWords = state_rows_per_s<FORM>() * 16 * 32;
  typename FormOf<FORM, S>::Strip st;
  st.load(A.img + static_cast<size_t>(item) * kImgStride, lane);
  bool moved = false;  // the segment before was recomputed: its final state is new
  for (int s = 1; s < nseg; ++s) {
    const bool bad = moved ? !boundary_exact<FORM>(A, base, s, S, lane) : __ldcg(&A.bests[base + s].pad) != 0;
    moved = bad;
    if (!bad) continue;
    long t_start, t_own, t_end;
    seg_bounds(S, nseg, s, A.N, &t_start, &t_own, &t_end);
    st.restore(A.states + ((base + s - 1) * 2 + 1) * kWords, ref, t_own, lane, place);
    typename FormOf<FORM, S>::Track tr;
    GlobalTiles src{ref, TS, t_own / TS};
    uint32_t *sf = s + 1 < nseg ? A.states + ((base + s) * 2 + 1) * kWords : nullptr;
    run_steps<FORM, S>(A, item, st, tr, src, TS, t_own, t_own, t_end, nullptr, sf, ring, lane, stk);
    tr.reduce(stk ? 16 : 32);
    if (lane == 0) {
      tr.store(A.bests + base + s);
      atomicAdd(A.ints + kIntFixups, 1);
    }
    if (stk && lane == 16) tr.store(A.bests2 + base + s);
    __syncwarp();
  }
}

// Segment minima combine by smaller cost, then by smaller segment (its
// columns are the smaller ones).
struct Pick {
  float c = __builtin_huge_valf();
  int s = 0x7fffffff;
  int64_t col = -1, start = -1;
  __device__ __forceinline__ void take(float oc, int os, int64_t ocol, int64_t ostart) {
    if (oc < c || (oc == c && os < s)) { c = oc; s = os; col = ocol; start = ostart; }
  }
  __device__ __forceinline__ void reduce() {
    for (int o = 16; o > 0; o >>= 1) {
      const float oc = __shfl_xor_sync(kFull, c, o);
      const int os = __shfl_xor_sync(kFull, s, o);
      const int64_t ocol = __shfl_xor_sync(kFull, col, o), ostart = __shfl_xor_sync(kFull, start, o);
      take(oc, os, ocol, ostart);
    }
  }
};

// The item's result over its segments (whole warp; valid on every lane).
template <int FORM>
__device__ __forceinline__ Best combine(const Best *bests, int nseg, int lane) {
  Pick a, b;
  for (int s = lane; s < nseg; s += 32) {
    const Best o = bests[s];
    if (form_i16(FORM)) {  // costs up to CAP: exact as floats
      a.take(static_cast<float>(o.ia), s, o.ca, -1);
      b.take(static_cast<float>(o.ib), s, o.cb, -1);
    } else {
      a.take(o.f, s, o.ca, o.cb);  // cb: the start column of the span forms
    }
  }
  a.reduce();
  Best r{};
  if (form_i16(FORM)) {
    b.reduce();
    r.ia = static_cast<int>(a.c);
    r.ib = static_cast<int>(b.c);
    r.cb = b.col;
  } else {
    r.f = a.c;
    r.cb = a.start;
  }
  r.ca = a.col;
  return r;
}

template <int FORM, int S = 1>
__device__ __forceinline__ void dispatch_recompute(int s, const SdtwArgs &A, int item, uint32_t *ring, int lane) {
  if constexpr (S <= kMaxS) {
    if (s == S)
      recompute_segments<FORM, S>(A, item, ring, lane);
    else
      dispatch_recompute<FORM, S + 1>(s, A, item, ring, lane);
  }
}

// Batches cut into at most kFixSolo segments (thousands of items) give each
// warp an item of its own: a CTA per item ran 137 us on 6,571 items, this 20.
constexpr int kFixWarps = 8, kFixSolo = 8;

// part: which kFixWarps of the item's segments this CTA verifies, one to a
// warp; -1: this warp alone has the item.
template <int FORM>
__device__ void fixup_item(const SdtwArgs &A, int item, int part, uint32_t *ring, int *last) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Item it = A.items[item];
  const int nseg = it.nseg;
  const int parts = part < 0 ? 1 : (nseg + kFixWarps - 1) / kFixWarps;
  if (part >= parts) return;
  const size_t base = static_cast<size_t>(item) * A.nseg_cap;
  const int s_lo = part < 0 ? 1 : part * kFixWarps + warp;
  const int s_hi = part < 0 ? nseg : (s_lo < nseg ? s_lo + 1 : s_lo);
  for (int s = s_lo; s < s_hi; ++s) {
    if (s == 0) continue;
    const bool exact = boundary_exact<FORM>(A, base, s, it.S, lane);
    if (lane == 0) A.bests[base + s].pad = exact ? 0 : 1;
  }
  if (part >= 0) {
    __syncthreads();
    if (parts > 1) {
      if (threadIdx.x == 0) {
        __threadfence();
        *last = atomicAdd(A.arrived + item, 1) == parts - 1;
        __threadfence();
      }
      __syncthreads();
      if (!*last) return;
    }
    if (warp != 0) return;
  }
  __syncwarp();
  if (nseg > 1) {
    bool bad = false;
    for (int s = 1 + lane; s < nseg; s += 32) bad = bad || __ldcg(&A.bests[base + s].pad) != 0;
    if (__any_sync(kFull, bad)) dispatch_recompute<FORM>(it.S, A, item, ring, lane);
  }
  const Best b = combine<FORM>(A.bests + base, nseg, lane);
  if (lane == 0) write_out<FORM>(A, b, it.qa, it.qb);
  if (it.stacked) {
    const Best b2 = combine<FORM>(A.bests2 + base, nseg, lane);
    if (lane == 0) write_out<FORM>(A, b2, it.qc, it.qd);
  }
}

template <int PREC>
__global__ void __launch_bounds__(kFixWarps * 32) fixup_kernel(SdtwArgs A) {
  __shared__ __align__(16) uint32_t rings[kFixWarps * ring_words(PREC)];
  __shared__ int last;
  const int warp = threadIdx.x >> 5;
  const bool split = A.nseg_cap > kFixSolo;
  const int item = split ? blockIdx.x : blockIdx.x * kFixWarps + warp;
  const int part = split ? blockIdx.y : -1;
  uint32_t *ring = rings + warp * ring_words(PREC);
  if (item >= A.ints[kIntItems]) return;
  if constexpr (PREC == HARU_FP32) {
    fixup_item<kFormF32>(A, item, part, ring, &last);
  } else if constexpr (PREC == HARU_INT16_ACC32) {
    fixup_item<kFormExactWide>(A, item, part, ring, &last);
  } else if constexpr (PREC == kPrecF32Span) {
    fixup_item<kFormF32Span>(A, item, part, ring, &last);
  } else if constexpr (PREC == kPrecWideSpan) {
    fixup_item<kFormWideSpan>(A, item, part, ring, &last);
  } else if (A.items[item].qmax > A.half_max) {
    fixup_item<kFormI16Large>(A, item, part, ring, &last);
  } else {
    fixup_item<kFormI16>(A, item, part, ring, &last);
  }
}

// ---------------------------------------------------------------- trace --
// Start columns without carrying them through the whole reference: the cost
// sweep gives each query's cost and end column and leaves exact states
// behind (checkpoints); from the nearest one at least two strip heights
// before the end, the start-column strip runs on to the end column alone.
// Every cost there is exact, so every cell picks the predecessor the full
// sweep would; starts before the checkpoint are kUnknownStart, and the end
// cell's is unknown only if its alignment began before the checkpoint: then
// the strip runs again from an earlier one, at last from the fresh start.
// (512 uneven FP32 queries on 59,796 columns: the whole call 4.1 ms with the
// starts carried through the sweep, 1.6 ms this way.)
struct TrackAt {
  long want;  // the end column on the lanes of the query's stack, -1 on the others
  int want_rel = kNoOffset, start = kUnknownStart;
  __device__ __forceinline__ void rebase(long to) {
    const long d = want - to;
    want_rel = d > kNoOffset && d < 0x7fffffff ? static_cast<int>(d) : kNoOffset;
  }
  __device__ __forceinline__ void add(uint32_t, const uint32_t *entry, int rel, bool in) {
    if (in && rel == want_rel) start = static_cast<int>(entry[2 * flush_words(kPrecF32Span)]);
  }
};

template <int FORM, int S>
__device__ void trace_query(const SdtwArgs &A, int item, int q, bool lower, uint32_t *ring, int lane) {
  const bool stk = A.items[item].stacked != 0;
  const uint32_t *ref = static_cast<const uint32_t *>(A.ref_img);
  const int place = stack_place(lane, stk);
  const long end = trace_end(A.out_col[q], A.N, A.ints[kIntAbort]);
  int start = -1;
  if (end >= 0) {
    const int TS = tile_width(4096), D = checkpoint_steps(A.checkpoint_step);
    const int rows = stk ? 16 * S : 32 * S;
    const long t_last = end + rows - 1, t_end = (t_last + kChunk) / kChunk * kChunk;
    const long back = t_last - 2 * rows - 32;
    typename FormOf<FORM, S>::Strip st;
    st.load(A.img + static_cast<size_t>(item) * kImgStride, lane);
    long c = back > 0 ? back / D : 0, less = 1;
    if (c > A.checkpoint_cap) c = A.checkpoint_cap;
    for (;;) {
      const long t0 = c * D;
      if (c == 0)
        st.fresh(0, place);
      else
        st.restore_costs(A.checkpoints + (static_cast<size_t>(item) * A.checkpoint_cap + (c - 1)) * kStateStride, ref,
                         t0, lane, place);
      TrackAt tr;
      tr.want = !stk || (lane >= 16) == lower ? end : -1;
      GlobalTiles src{ref, TS, t0 / TS};
      run_steps<FORM, S>(A, item, st, tr, src, TS, t0, t0, t_end, nullptr, nullptr, ring, lane, stk);
      start = __reduce_max_sync(kFull, tr.start);
      if (start != kUnknownStart || c == 0) break;
      c = c > less ? c - less : 0;
      less *= 2;
    }
  }
  if (lane == 0) A.out_start[q] = start;
}

template <int FORM, int S = 1>
__device__ __forceinline__ void dispatch_trace(int s, const SdtwArgs &A, int item, int q, bool lower, uint32_t *ring,
                                               int lane) {
  if constexpr (S <= kMaxS) {
    if (s == S)
      trace_query<FORM, S>(A, item, q, lower, ring, lane);
    else
      dispatch_trace<FORM, S + 1>(s, A, item, q, lower, ring, lane);
  }
}

constexpr int kTraceWarps = 4;

// One warp per query (`parts` = 2 in batches with stacked items).
template <int PREC>
__global__ void __launch_bounds__(kTraceWarps * 32) trace_kernel(SdtwArgs A, int parts) {
  __shared__ __align__(16) uint32_t rings[kTraceWarps * ring_words(PREC)];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = blockIdx.x * kTraceWarps + warp, item = w / parts;
  const bool lower = w % parts != 0;
  if (item >= A.ints[kIntItems]) return;
  const int q = lower ? A.items[item].qc : A.items[item].qa;
  if (q < 0) return;
  constexpr int kForm = PREC == kPrecF32Span ? kFormF32Span : kFormWideSpan;
  dispatch_trace<kForm>(A.items[item].S, A, item, q, lower, rings + warp * ring_words(PREC), lane);
}

template <int PREC>
cudaError_t launch_trace_prec(const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s) {
  const int parts = stacked ? 2 : 1;
  trace_kernel<PREC><<<(max_items * parts + kTraceWarps - 1) / kTraceWarps, kTraceWarps * 32, 0, s>>>(a, parts);
  return cudaGetLastError();
}

template <int PREC, bool SOLO>
SmemOptIn &smem_record() {
  static SmemOptIn rec;
  return rec;
}
template <int PREC, bool SOLO>
constexpr auto sweep_kernel() {
  if constexpr (SOLO)
    return sdtw_kernel<PREC>;
  else
    return queue_kernel<PREC>;
}

template <int PREC, bool SOLO>
cudaError_t launch_sweep_prec(const SdtwArgs &a, int grid, cudaStream_t s) {
  const size_t sm = sdtw_smem_bytes(PREC, a.tile_cols, a.warps, SOLO);
  const auto kernel = sweep_kernel<PREC, SOLO>();
  cudaError_t e = opt_in_smem(kernel, smem_record<PREC, SOLO>(), sm);
  if (e != cudaSuccess) return e;
  kernel<<<grid, a.warps * 32, sm, s>>>(a);
  return cudaGetLastError();
}

template <int PREC>
cudaError_t launch_fixup_prec(const SdtwArgs &a, int fix_items, cudaStream_t s) {
  if (fix_items <= 0) return cudaSuccess;
  const bool split = a.nseg_cap > kFixSolo;
  const dim3 grid(split ? fix_items : (fix_items + kFixWarps - 1) / kFixWarps,
                  split ? (a.nseg_cap + kFixWarps - 1) / kFixWarps : 1);
  fixup_kernel<PREC><<<grid, kFixWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

template <int PREC>
int occupancy_prec(int tile_cols, int warps) {
  int n = 0;
  const size_t sm = sdtw_smem_bytes(PREC, tile_cols, warps, false);
  if (opt_in_smem(queue_kernel<PREC>, smem_record<PREC, false>(), sm) != cudaSuccess) return 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, queue_kernel<PREC>, warps * 32, sm);
  return n;
}

}  // namespace
}  // namespace haru

// Define the entry points of a kernel for kernel precision P (0 FP32, 1
// INT16, 2 int16 inputs with wide accumulation, 3 FP32 with start columns, 4
// wide with start columns, 5 INT16 with both cells): the scheduled
// sweep, the queue's sweep, the segment fix-up, the trace. One per
// translation unit, so the kernels compile in parallel.
#define HARU_SDTW_SWEEP_INSTANCE(P)                                                                        \
  namespace haru {                                                                                         \
  cudaError_t sdtw_sweep_##P(const SdtwArgs &a, int grid, cudaStream_t s) {                               \
    return launch_sweep_prec<P, true>(a, grid, s);                                                         \
  }                                                                                                        \
  cudaError_t sdtw_sweep_load_##P() {                                                                      \
    cudaFuncAttributes f;                                                                                  \
    return cudaFuncGetAttributes(&f, sdtw_kernel<P>);                                                      \
  }                                                                                                        \
  }
#define HARU_SDTW_QUEUE_INSTANCE(P)                                                                        \
  namespace haru {                                                                                         \
  cudaError_t sdtw_queue_##P(const SdtwArgs &a, int grid, cudaStream_t s) {                               \
    return launch_sweep_prec<P, false>(a, grid, s);                                                        \
  }                                                                                                        \
  int sdtw_occupancy_##P(int tile_cols, int warps) { return occupancy_prec<P>(tile_cols, warps); }         \
  cudaError_t sdtw_queue_load_##P() {                                                                      \
    cudaFuncAttributes f;                                                                                  \
    return cudaFuncGetAttributes(&f, queue_kernel<P>);                                                     \
  }                                                                                                        \
  }
#define HARU_SDTW_FIXUP_INSTANCE(P)                                                            \
  namespace haru {                                                                             \
  cudaError_t sdtw_fixup_##P(const SdtwArgs &a, int fix_items, cudaStream_t s) {              \
    return launch_fixup_prec<P>(a, fix_items, s);                                              \
  }                                                                                            \
  cudaError_t sdtw_fixup_load_##P() {                                                          \
    cudaFuncAttributes f;                                                                      \
    return cudaFuncGetAttributes(&f, fixup_kernel<P>);                                         \
  }                                                                                            \
  }
#define HARU_SDTW_TRACE_INSTANCE(P)                                                            \
  namespace haru {                                                                             \
  cudaError_t sdtw_trace_##P(const SdtwArgs &a, int max_items, bool stacked, cudaStream_t s) { \
    return launch_trace_prec<P>(a, max_items, stacked, s);                                     \
  }                                                                                            \
  }
