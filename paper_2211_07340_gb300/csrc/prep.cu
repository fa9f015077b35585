// Device-side preparation: reference synthesis and normalisation (Section
// 4.1), the batch planner, and per-query normalisation, quantisation and
// packing into the warp-strip register images the sweep kernels load.
//
// z-score reading (the paper does not say how mean and sigma are formed):
// population sigma; sums in double, in blocks of 4096 consecutive samples
// added in index order, block sums added in index order; every double
// operation is an explicitly rounded intrinsic so no contraction occurs;
// z = (float)((x - mean) / sigma). Quantiser: clamp(rint(z * 2^k), +-2047).

#include <cuda_runtime.h>

#include "haru_internal.h"

namespace haru {
namespace {

constexpr int kZBlock = 4096;

__device__ __forceinline__ bool finite_d(double v) { return isfinite(v); }

__device__ __forceinline__ int quantise(float z, float s) {
  int v = __float2int_rn(__fmul_rn(z, s));
  return v > kQmax ? kQmax : (v < -kQmax ? -kQmax : v);
}

// ------------------------------------------------------------ reference --
__global__ void ref_levels_kernel(const uint8_t *bases, size_t n, const float *model, int k, float *out,
                                  int *status) {
  const size_t per = n - static_cast<size_t>(k) + 1;
  for (size_t j = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; j < 2 * per;
       j += static_cast<size_t>(gridDim.x) * blockDim.x) {
    long code = 0;
    bool bad = false;
    if (j < per) {
      for (int u = 0; u < k; ++u) {
        uint8_t b = bases[j + u];
        bad |= b > 3;
        code = code * 4 + (b & 3);
      }
    } else {
      const size_t jj = j - per;  // k-mer jj of the reverse complement
      for (int u = 0; u < k; ++u) {
        uint8_t b = bases[n - 1 - (jj + u)];
        bad |= b > 3;
        code = code * 4 + (3 - (b & 3));
      }
    }
    if (bad) report(status, HARU_EINVAL);
    out[j] = model[code];
  }
}

// One thread per block of kZBlock samples: the block's sum (pass 0) or sum
// of squared deviations from stats[0] (pass 1), in index order.
__global__ void block_sums_kernel(const float *x, size_t n, const double *stats, int pass, double *partials) {
  const size_t b = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const size_t lo = b * kZBlock;
  if (lo >= n) return;
  const size_t hi = lo + kZBlock < n ? lo + kZBlock : n;
  double acc = 0.0;
  if (pass == 0) {
    for (size_t i = lo; i < hi; ++i) acc = __dadd_rn(acc, static_cast<double>(x[i]));
  } else {
    const double mean = stats[0];
    for (size_t i = lo; i < hi; ++i) {
      const double d = __dsub_rn(static_cast<double>(x[i]), mean);
      acc = __dadd_rn(acc, __dmul_rn(d, d));
    }
  }
  partials[b] = acc;
}

// Single thread: add the block sums in order; pass 0 -> mean, pass 1 -> sigma.
__global__ void finish_sums_kernel(const double *partials, size_t nblocks, size_t n, int pass, double *stats,
                                   int *status) {
  double acc = 0.0;
  for (size_t b = 0; b < nblocks; ++b) acc = __dadd_rn(acc, partials[b]);
  if (pass == 0) {
    stats[0] = __ddiv_rn(acc, static_cast<double>(n));
    if (!finite_d(stats[0])) report(status, HARU_EINVAL);
  } else {
    const double sigma = __dsqrt_rn(__ddiv_rn(acc, static_cast<double>(n)));
    stats[1] = sigma;
    if (!(sigma > 0.0) || !finite_d(sigma)) report(status, HARU_EINVAL);
  }
}

__global__ void ref_finish_kernel(const float *x, size_t n, const double *stats, int normalize, float s,
                                  float *z, uint32_t *img16, uint32_t *imgh, float *img32, int *status,
                                  int *max_code) {
  int most = 0;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    float v = x[i];
    if (normalize) {
      const double mean = stats[0], sigma = stats[1];
      v = __double2float_rn(__ddiv_rn(__dsub_rn(static_cast<double>(v), mean), sigma));
    }
    if (!isfinite(v)) report(status, HARU_EINVAL);
    const int q = quantise(v, s);
    z[i] = v;
    img16[i] = (static_cast<uint32_t>(q) & 0xffffu) | (static_cast<uint32_t>(q) << 16);
    imgh[i] = half_code(q) * 0x10001u;
    img32[i] = v;
    most = max(most, abs(q));
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) atomicMax(max_code, most);
}

// --------------------------------------------------------------- planner --
// Bucket key of query q: its strip height S (rows per lane), plus kMaxS + 1
// if it is stacked (16 lanes); 0 for an invalid length. S is the least
// height that leaves a pad row on top of the query (S = floor(M / 32) + 1,
// or floor(M / 16) + 1 stacked), at most kMaxS: the sweep relies on that
// row to hold the free-start zero in strips lower than kMaxS.
__device__ __forceinline__ int bucket_key(const uint32_t *off, uint32_t q, long N, int mode, int stack, int *status) {
  const uint32_t m = off[q + 1] - off[q];
  const long lim = N < HARU_MAX_QUERY ? N : HARU_MAX_QUERY;
  if (m < 1 || static_cast<long>(m) > lim) {
    if (status) report(status, HARU_EINVAL);
    return 0;
  }
  if (stack && m <= static_cast<uint32_t>(kStackMax))
    return min(static_cast<int>(m / 16) + 1, kMaxS) + kMaxS + 1;
  return min(static_cast<int>(m / 32) + 1, kMaxS);
}

// Items of a bucket of n queries. Modes 0 (FP32) and 3 (int16 inputs, wide
// accumulation) make one item per query (two per stacked item); mode 1
// pairs int16 queries (four per stacked item).
__device__ __forceinline__ bool singles(int mode) { return mode == 0 || mode == 3; }
__device__ __forceinline__ int stacked_items(int mode, int n) { return singles(mode) ? (n + 1) / 2 : (n + 3) / 4; }
__device__ __forceinline__ int bucket_items(int mode, int n) { return singles(mode) ? n : (n + 1) / 2; }

// Segments of each strip height and the static schedule by a cost model (the
// whole CTA).
//
// A step of a strip of S rows takes I = clocks[S - 1] for each warp on its
// scheduler when all of the CTA's warps are at work, some more with fewer. A
// segment after the first repeats warmup_steps(S). A candidate is a longest
// segment time h, which gives n = ceil(T * I / h) segments of each height,
// and m warps at work per CTA; its estimate is a CTA's share: the bundles'
// whole time over the CTAs, or the longest bundle's. Each warp estimates
// candidates with a lane per strip height and part: kTries values of h, 2^(1/4)
// apart, by three of m, then kTries between the best one's neighbours.
// Segments shorter than a quarter of their warm-up buy too little for their
// work.
constexpr int kTries = 32;

struct PlanTables {
  int cnt[2 * (kMaxS + 1)];                                   // queries per bucket key
  int ibase[kMaxS + 1], sbase[kMaxS + 1], icount[kMaxS + 1];  // items
  int nseg[2 * kMaxS], full[kMaxS + 1];  // of 2 * (16 - S) + rest; items of S before its rest
  int gbase[kMaxS + 1], gcount[kMaxS + 1];
  float est[3 * kTries];
  float h;  // the cost model's choice
  int c;
};

__device__ __forceinline__ float warp_max(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ void cost_model(const PlanArgs &a, PlanTables &t) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // lane l: strip height 16 - l / 2, its full bundles or its rest (the schedule's order)
  const int S = kMaxS - lane / 2;
  const bool rest = lane & 1;
  const int items = t.icount[S];
  const float T = static_cast<float>(sweep_steps(S, a.N)), V = static_cast<float>(warmup_steps(S));
  const float I = a.clocks[S - 1] +
                  (items > 0 ? a.stacked * (items - (t.sbase[S] - t.ibase[S])) / static_cast<float>(items) : 0.0f);
  const float most_n = floorf(fminf(fmaxf(4.0f * T / V, 1.0f), static_cast<float>(a.nseg_cap)));
  const float longest = warp_max(items > 0 ? T * I : 0.0f);
  // all of the CTA's warps at work, or four or eight fewer (a warp per scheduler at least)
  auto width = [&](int c) { return max(min(a.warps, 4), a.warps - 4 * c); };
  auto segments = [&](float h) { return static_cast<int>(fminf(ceilf(T * I / h), most_n)); };
  auto bundle = [&](int n, int warps) {  // a bundle's time
    const int x = (warps + 3) / 4;
    return (T / n + (n > 1 ? V : 0.0f)) * x * (I + (x * 4 >= a.warps ? 0.0f : (x == 1 ? a.one : a.two)));
  };
  auto time_of = [&](int units, int n, int m, float *top) {  // all bundles' time, and the longest one's
    const int full = units / m, last = units - full * m;
    *top = units > 0 ? bundle(n, full > 0 ? m : last) : 0.0f;
    return full * *top + (last > 0 ? bundle(n, last) : 0.0f);
  };
  auto try_h = [&](float h, int round, int q) {
    return round == 0 ? longest * exp2f(-0.25f * q) * 1.0001f
                      : h * exp2f(0.25f * (q - 0.5f * (kTries - 1)) / (0.5f * kTries));
  };
  float h = longest;
  for (int round = 0; round < 2; ++round) {
    for (int k = warp; k < 3 * kTries; k += nw) {
      float all = 0.0f, top = 0.0f;
      if (items > 0 && !rest) {
        const int n = segments(try_h(h, round, k % kTries));
        all = time_of(items * n, n, width(k / kTries), &top);
      }
      const float e = fmaxf(warp_max(top), warp_sum(all) / a.slots);
      if (lane == 0) t.est[k] = e;
    }
    __syncthreads();
    if (warp == 0) {  // the smallest estimate; the wider bundles and longer segments on a tie
      float e = t.est[lane];
      int at = lane;
      for (int k = lane + 32; k < 3 * kTries; k += 32)
        if (t.est[k] < e) { e = t.est[k]; at = k; }
      for (int o = 16; o > 0; o >>= 1) {
        const float oe = __shfl_xor_sync(0xffffffffu, e, o);
        const int oat = __shfl_xor_sync(0xffffffffu, at, o);
        if (oe < e || (oe == e && oat < at)) { e = oe; at = oat; }
      }
      if (lane == 0) {
        t.h = try_h(h, round, at % kTries);
        t.c = at / kTries;
      }
    }
    __syncthreads();
    h = t.h;
  }
  if (warp == 0) {
    const int m = width(t.c);
    int n = items > 0 ? segments(h) : 1;
    // Items beyond those whose n segments fill whole bundles: they take the
    // multiple of n (up to kMore) that runs them in the least time.
    constexpr int kMore = 6;
    int g = m;  // m / gcd(m, n): items that fill bundles together
    for (int f = 2; f <= 3; ++f)
      for (int k = n; g % f == 0 && k % f == 0; k /= f) g /= f;
    const int own = rest ? items % g : items - items % g;
    if (rest && own > 0) {
      const int base = n;
      float least = 0.0f, top_k;
      for (int k = 1; k <= kMore && base * k <= static_cast<int>(fmaxf(most_n, base)); ++k) {
        const float all_k = time_of(own * base * k, base * k, m, &top_k);
        if (k == 1 || all_k < least) { least = all_k; n = base * k; }
      }
    }
    const int units = own * n, bundles = (units + m - 1) / m, last = units - (bundles - 1) * m;
    const long long cost = own > 0 ? static_cast<long long>(bundle(n, m)) + 1 : 0;
    const long long last_cost = own > 0 ? static_cast<long long>(bundle(n, last)) + 1 : 0;
    const long long all = bundles > 0 ? (bundles - 1) * cost + last_cost : 0;
    long long end = all, top = bundles > 1 ? cost : last_cost;
    int bend = bundles;
    for (int o = 1; o < 32; o <<= 1) {
      const long long v = __shfl_up_sync(0xffffffffu, end, o);
      const int b = __shfl_up_sync(0xffffffffu, bend, o);
      if (lane >= o) { end += v; bend += b; }
    }
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
    t.nseg[lane] = n;
    if (!rest) t.full[S] = own;
    ScheduleRow r;
    r.items = own;
    r.base = t.ibase[S] + (rest ? items - own : 0);
    r.nseg = n;
    r.bundles = bundles;
    r.bundle0 = bend - bundles;
    r.last = last;
    r.start = end - all;
    r.cost = cost;
    r.last_cost = last_cost;
    a.sched->row[schedule_row(S, rest)] = r;
    if (lane == 31) {
      a.sched->members = m;
      a.sched->bundles = bend;
      a.sched->total = end;
      a.sched->share = max(top, (end + a.slots - 1) / a.slots);
      a.ints[kIntGroups] = bend;
    }
    const int most = __reduce_max_sync(0xffffffffu, own > 0 ? n : 0);
    if (lane == 0) a.ints[kIntMaxSeg] = most;
  }
  for (int p = threadIdx.x; p < a.slots; p += blockDim.x) a.done[p] = 0;
  __syncthreads();
}

// One CTA of 1024 threads. Buckets queries by strip height S (descending,
// the longest-processing-time-first order of the work queue), keeps the
// input order inside a bucket, pairs neighbours for the int16 form, and writes
// the static schedule or (explicit unit target) the queue of groups.
constexpr int kKeys = 2 * (kMaxS + 1);  // plain and stacked buckets of each S
struct PlanShared {
  PlanTables t;
  int wrun[32][kKeys];  // per warp and bucket: count, then next position
};
__device__ void plan_block(const PlanArgs &a, PlanShared &sm) {
  PlanTables &t = sm.t;
  auto &wrun = sm.wrun;
  int *const ibase = t.ibase, *const sbase = t.sbase, *const icount = t.icount;
  auto nseg_of = [&](int S, int item) { return t.nseg[2 * (kMaxS - S) + (item - t.ibase[S] >= t.full[S] ? 1 : 0)]; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  int *status = a.ints + kIntStatus;
  if (a.zero) {
    if (tid < kIntWords) a.ints[tid] = 0;
    __syncthreads();
  }
  // Each warp owns a contiguous range of queries, so bucket positions
  // (earlier warps first, then the order inside the warp) keep input order.
  const uint32_t per_warp = (a.nq + nw - 1) / nw;
  const uint32_t q_lo = min(a.nq, static_cast<uint32_t>(warp) * per_warp);
  const uint32_t q_hi = min(a.nq, q_lo + per_warp);
  for (int b = lane; b < kKeys; b += 32) wrun[warp][b] = 0;
  __syncwarp();
  auto key_of = [&](uint32_t q, int *st) {
    return q < q_hi ? bucket_key(a.offsets, q, a.N, a.pair, a.stack, st) : 0;
  };
  for (uint32_t q0 = q_lo, key = key_of(q_lo + lane, status); q0 < q_hi; q0 += 32) {
    const uint32_t after = key_of(q0 + 32 + lane, status);  // loaded a round ahead
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (key && lane == __ffs(peers) - 1) wrun[warp][key] += __popc(peers);
    __syncwarp();
    key = after;
  }
  __syncthreads();
  if (tid >= 1 && tid < kKeys) {
    int c = 0;
    for (int w = 0; w < nw; ++w) {
      const int v = wrun[w][tid];
      wrun[w][tid] = c;
      c += v;
    }
    t.cnt[tid] = c;
  }
  __syncthreads();
  if (warp == 0) {  // lane l: height 16 - l, its plain items, then its stacked ones
    const int S = lane < kMaxS ? kMaxS - lane : 0;
    const int plain = S ? bucket_items(a.pair, t.cnt[S]) : 0;
    const int items = S ? plain + stacked_items(a.pair, t.cnt[S + kMaxS + 1]) : 0;
    int end = items;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += v;
    }
    if (S) {
      icount[S] = items;
      ibase[S] = end - items;
      sbase[S] = end - items + plain;
    }
    if (lane == 31) {
      a.ints[kIntItems] = t.cnt[0] = end;
      a.ints[kIntQueue] = 0;
    }
    __syncwarp();
  }
  if (tid == 0) {
    const int base = t.cnt[0];
    if (a.units_target > 0) {
      // An explicit unit target: segments per item to reach it, each
      // at least four warm-ups (and 2048 steps) long.
      int want = base > 0 ? (a.units_target + base - 1) / base : 1;
      if (want < 1) want = 1;
      if (want > a.nseg_cap) want = a.nseg_cap;
      // The buckets at the end of the longest-first queue (the cheapest strips,
      // up to a fifth of the work) get twice the segments: shorter final work
      // units leave less of the machine idle while the last ones finish.
      long total = 0, acc = 0;
      for (int S = 1; S <= kMaxS; ++S) total += static_cast<long>(icount[S]) * S;
      int tail_to = 0;  // buckets S <= tail_to form the tail
      if (a.units_target > 1) {
        for (int S = 1; S <= kMaxS; ++S) {
          const long w = static_cast<long>(icount[S]) * S;
          if ((acc + w) * 5 > total) break;
          acc += w;
          tail_to = S;
        }
      }
      // Groups, tallest strips first: one longest-first queue for the sweep kernel.
      int g = 0;
      for (int S = kMaxS; S >= 1; --S) {
        const long minlen = 4 * warmup_steps(S) > 2048 ? 4 * warmup_steps(S) : 2048;
        long lim = sweep_steps(S, a.N) / minlen;
        if (lim < 1) lim = 1;
        int ws = S <= tail_to ? 2 * want : want;
        if (ws > a.nseg_cap) ws = a.nseg_cap;
        const int n = ws < lim ? ws : static_cast<int>(lim);
        t.nseg[2 * (kMaxS - S)] = n;
        t.full[S] = icount[S];
        t.gbase[S] = g;
        t.gcount[S] = n * ((icount[S] + a.warps - 1) / a.warps);
        g += t.gcount[S];
      }
      a.ints[kIntGroups] = g;
      int most = 0;
      for (int S = 1; S <= kMaxS; ++S)
        if (icount[S] > 0 && t.nseg[2 * (kMaxS - S)] > most) most = t.nseg[2 * (kMaxS - S)];
      a.ints[kIntMaxSeg] = most;
    }
  }
  __syncthreads();
  if (a.units_target == 0) {
    cost_model(a, t);
  } else {
    // Groups of each bucket, segment-major: (seg, first item), in parallel.
    for (int S = kMaxS; S >= 1; --S) {
      const int per_seg = (icount[S] + a.warps - 1) / a.warps;
      for (int j = tid; j < t.gcount[S]; j += blockDim.x) {
        const int seg = j / per_seg, f = (j % per_seg) * a.warps;
        Group gr;
        gr.S = S;
        gr.first = ibase[S] + f;
        gr.count = icount[S] - f < a.warps ? icount[S] - f : a.warps;
        gr.seg = seg;
        gr.nseg = t.nseg[2 * (kMaxS - S)];
        gr.pad[0] = gr.pad[1] = gr.pad[2] = 0;
        a.groups[t.gbase[S] + j] = gr;
      }
    }
    __syncthreads();
  }
  const int n_items = t.cnt[0];
  for (int i = tid; i < n_items; i += blockDim.x) {
    Item it;
    it.qa = -1; it.qb = -1; it.S = 0; it.nseg = 1;
    it.qmax = 0;
    it.qc = -1; it.qd = -1; it.stacked = 0;
    a.items[i] = it;
    if (a.arrived) a.arrived[i] = 0;
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  for (uint32_t q0 = q_lo, next = key_of(q_lo + lane, nullptr); q0 < q_hi; q0 += 32) {
    const uint32_t q = q0 + lane;
    const int key = static_cast<int>(next);
    next = key_of(q0 + 32 + lane, nullptr);
    const unsigned peers = __match_any_sync(0xffffffffu, key);
    if (key > kMaxS) {  // stacked: slots qa, qb | qc, qd (INT16) or qa | qc (FP32)
      const int b = key - kMaxS - 1;
      const int pos = wrun[warp][key] + __popc(peers & lt);
      const int per = singles(a.pair) ? 2 : 4;
      const int slot = singles(a.pair) ? 2 * (pos % 2) : pos % 4;
      const int item = sbase[b] + pos / per;
      Item *it = &a.items[item];
      if (slot == 0) { it->qa = static_cast<int>(q); it->S = b; it->nseg = nseg_of(b, item); it->stacked = 1; }
      else if (slot == 1) it->qb = static_cast<int>(q);
      else if (slot == 2) it->qc = static_cast<int>(q);
      else it->qd = static_cast<int>(q);
    } else if (key) {
      const int b = key;
      const int pos = wrun[warp][b] + __popc(peers & lt);  // position in bucket b
      if (a.pair == 1) {
        const int item = ibase[b] + pos / 2;
        Item *it = &a.items[item];
        if (pos % 2 == 0) { it->qa = static_cast<int>(q); it->S = b; it->nseg = nseg_of(b, item); }
        else it->qb = static_cast<int>(q);
      } else {
        Item it;
        it.qa = static_cast<int>(q); it.qb = -1; it.S = b; it.nseg = nseg_of(b, ibase[b] + pos);
        it.qmax = 0;
        it.qc = -1; it.qd = -1; it.stacked = 0;
        a.items[ibase[b] + pos] = it;
      }
    }
    __syncwarp();
    if (key && lane == __ffs(peers) - 1) wrun[warp][key] += __popc(peers);
    __syncwarp();
  }
}

// ----------------------------------------------------------------- pack --
// z = (float)((x - mean) / sigma), both roundings of the quotient kept, from
// the reciprocal r = 1 / sigma: d * r is within two units in the last place
// of the quotient in double, so the quotient's float is the product's unless
// the product lies within a few units of the midpoint between two floats (29
// bits below a float's last), is as small as a subnormal float, or is not
// finite: then the division is done. (The double-precision unit takes 16
// clocks a warp instruction on GB300; a division is about ten of them.)
__device__ __forceinline__ float z_of(float x, double mean, double sigma, double r) {
  const double d = __dsub_rn(static_cast<double>(x), mean);
  const double q = __dmul_rn(d, r);
  const unsigned hi = static_cast<unsigned>(__double2hiint(q)), lo = static_cast<unsigned>(__double2loint(q));
  const unsigned exponent = (hi >> 20) & 0x7ffu;
  const unsigned below = lo & 0x1fffffffu;  // the bits under a float's last
  const bool near_half = below - (0x10000000u - 8u) <= 16u;
  if (near_half || exponent < 1023u - 120u || exponent > 1023u + 120u) return __double2float_rn(__ddiv_rn(d, sigma));
  return __double2float_rn(q);
}

// Mean and sigma (FP64) of each query of 1..512 events: the sums are those of
// sequential additions in index order.
// Mean: if every event is a multiple of 2^low and below 2^top in magnitude
// with top + 9 - low <= 53, no partial sum of up to 512 of them rounds, in
// any order, and the sum is taken on integers across a warp; other queries
// are added up one by one.
// Sigma: the additions of the squared deviations round, so they stay one
// chain per query, 64 clocks each; a lane of the block's first warps (chain
// warps) holds the chain of one query, and the other warps compute the
// squares of the next chunk of events meanwhile (one thread per query, with
// its loads and conversions in the chain, took 52 us at 250 events and 104
// us on 8,192 queries of up to 500; this kernel, planner included, 16 and 48).
constexpr int kStatQueries = 64;  // per block at most: two chain warps
constexpr int kStatSquares = kStatQueries * 33;
struct StatShared {
  double sq[2][kStatSquares];  // [query][chunk + 1]
  long long sum[kStatQueries];
  double mean[kStatQueries];
  int low[kStatQueries];  // exponent of the integer sum's unit; kInexact: add one by one
  int length[kStatQueries];
  uint32_t base[kStatQueries];
  int longest;
};
constexpr int kInexact = 0x7fffffff;
struct StatArgs {
  const float *events;
  const uint32_t *offsets;
  uint32_t nq;
  int per_block;  // queries: 8, 32 or 64
  double *qstats;
};

__device__ __forceinline__ double as_double(float x) {  // exact; normal numbers without the conversion unit
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e == 0u || e == 255u) return static_cast<double>(x);
  return __hiloint2double(static_cast<int>((b & 0x80000000u) | ((e + 896u) << 20) | ((b >> 3) & 0xfffffu)),
                          static_cast<int>(b << 29));
}

__device__ void stat_block(const StatArgs &a, int block, StatShared &sm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const uint32_t q0 = static_cast<uint32_t>(block) * a.per_block;
  // a block of up to 32 queries takes chunks of 64 events, one of 64 queries 32
  const int chunk = a.per_block > 32 ? 32 : 64, row = chunk + 1, chain_warps = (a.per_block + 31) / 32;
  if (tid == 0) sm.longest = 0;
  __syncthreads();
  if (tid < a.per_block) {
    const uint32_t q = q0 + tid, b = q < a.nq ? a.offsets[q] : 0u, m = q < a.nq ? a.offsets[q + 1] - b : 0u;
    const int len = m <= HARU_MAX_QUERY ? static_cast<int>(m) : 0;  // other lengths are rejected by the planner
    sm.length[tid] = len;
    sm.base[tid] = b;
    atomicMax(&sm.longest, len);
  }
  __syncthreads();
  for (int k = warp; k < a.per_block; k += nw) {
    const float *x = a.events + sm.base[k];
    const int m = sm.length[k];
    constexpr int kPer = HARU_MAX_QUERY / 32;
    unsigned v[kPer];
    int low = 1 << 20, top = -(1 << 20);
    bool finite = true;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const int i = j * 32 + lane;
      v[j] = i < m ? __float_as_uint(__ldg(x + i)) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      const unsigned mag = v[j] & 0x7fffffffu, e = mag >> 23;
      if (mag == 0u) continue;
      finite = finite && e != 255u;
      const unsigned mant = (mag & 0x7fffffu) | (e ? 0x800000u : 0u);
      const int at = max(static_cast<int>(e), 1) - 150;  // of the mantissa's last bit
      low = min(low, at + __ffs(mant) - 1);
      top = max(top, at + 32 - __clz(mant));
    }
    low = __reduce_min_sync(0xffffffffu, low);
    top = __reduce_max_sync(0xffffffffu, top);
    finite = __all_sync(0xffffffffu, finite);
    const bool exact = finite && top + 9 - low <= 53;
    long long sum = 0;
    if (exact) {
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const unsigned mag = v[j] & 0x7fffffffu, e = mag >> 23;
        const unsigned mant = (mag & 0x7fffffu) | (e ? 0x800000u : 0u);
        const int up = max(static_cast<int>(e), 1) - 150 - low;
        const long long u = mag == 0u ? 0 : (up >= 0 ? static_cast<long long>(mant) << up : mant >> -up);
        sum += (v[j] >> 31) ? -u : u;
      }
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
      sm.sum[k] = sum;
      sm.low[k] = exact ? low : kInexact;
    }
  }
  __syncthreads();
  const bool chain = tid < a.per_block;  // this thread's query: tid
  double ss = 0.0, count = 1.0;
  int own = 0;
  if (chain) {
    const float *x = a.events + sm.base[tid];
    own = sm.length[tid];
    double acc = 0.0;
    if (sm.low[tid] != kInexact) {
      // (low = 1 << 20: every event is 0)
      const int low = sm.low[tid];
      if (sm.sum[tid] != 0)
        acc = __dmul_rn(__ll2double_rn(sm.sum[tid]), __hiloint2double((1023 + low) << 20, 0));
    } else {
      for (int i = 0; i < own; ++i) acc = __dadd_rn(acc, static_cast<double>(__ldg(x + i)));
    }
    count = static_cast<double>(max(own, 1));
    sm.mean[tid] = __ddiv_rn(acc, count);
  }
  __syncthreads();
  const int chunks = (sm.longest + chunk - 1) / chunk;
  auto squares = [&](int c, int from, int warps) {  // by `warps` warps, this one's number `from`
    for (int k = from; k < a.per_block; k += warps) {
      const float *x = a.events + sm.base[k];
      const int m = sm.length[k];
      const double mean = sm.mean[k];
      for (int o = lane; o < chunk; o += 32) {
        const int i = c * chunk + o;
        double p = 0.0;  // beyond the query: adding 0 changes nothing
        if (i < m) {
          const double d = __dsub_rn(as_double(__ldg(x + i)), mean);
          p = __dmul_rn(d, d);
        }
        sm.sq[c & 1][k * row + o] = p;
      }
    }
  };
  if (chunks > 0) squares(0, warp, nw);
  __syncthreads();
  for (int c = 0; c < chunks; ++c) {
    if (chain) {
      const double *sq = &sm.sq[c & 1][tid * row];
#pragma unroll 16
      for (int i = 0; i < chunk; ++i) ss = __dadd_rn(ss, sq[i]);
    } else if (warp >= chain_warps && c + 1 < chunks) {
      squares(c + 1, warp - chain_warps, nw - chain_warps);
    }
    __syncthreads();
  }
  if (chain && q0 + tid < a.nq) {
    const size_t q = q0 + tid;
    a.qstats[2 * q] = own > 0 ? sm.mean[tid] : 0.0;
    a.qstats[2 * q + 1] = own > 0 ? __dsqrt_rn(__ddiv_rn(ss, count)) : 1.0;
  }
}

// Block 0 plans the batch; the others, on raw events, form the queries'
// means and sigmas at the same time.
__global__ void __launch_bounds__(1024) prep_kernel(PlanArgs p, StatArgs st) {
  __shared__ union Shared {
    PlanShared plan;
    StatShared stat;
    __device__ Shared() {}
  } sm;
  if (blockIdx.x == 0)
    plan_block(p, sm.plan);
  else
    stat_block(st, static_cast<int>(blockIdx.x) - 1, sm.stat);
}

// One warp per item: lane l writes rows l*S .. l*S+S-1 of both halves (of
// its own stack, for stacked items).
__global__ void pack_kernel(PackArgs a) {
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (item >= *a.n_items) return;
  const Item it = a.items[item];
  const int S = it.S;
  // Stacked items: lanes 16..31 hold the lower stack (qc, qd).
  const bool low = it.stacked && lane >= 16;
  const int qs[2] = {low ? it.qc : it.qa, low ? it.qd : it.qb};
  const int H = it.stacked ? 16 * S : 32 * S;             // rows of this lane's stack
  const int lane_in = it.stacked ? (lane & 15) : lane;   // lane within the stack
  int m[2] = {0, 0};
  uint32_t base[2] = {0, 0};
  double mean[2] = {0.0, 0.0}, sigma[2] = {1.0, 1.0}, inv[2] = {1.0, 1.0};
  const bool packed = a.pair == 1;  // two int16 queries per word
  const bool codes = a.pair != 0;   // int16 codes (packed, or as floats)
  int most = 0;
  const int halves = packed ? 2 : 1;
  for (int h = 0; h < halves; ++h) {
    if (qs[h] >= 0) {
      base[h] = a.offsets[qs[h]];
      m[h] = static_cast<int>(a.offsets[qs[h] + 1] - base[h]);
    }
  }
  if (a.raw) {
    for (int h = 0; h < halves; ++h) {
      if (qs[h] >= 0) {
        mean[h] = a.qstats[2 * static_cast<size_t>(qs[h])];
        sigma[h] = a.qstats[2 * static_cast<size_t>(qs[h]) + 1];
        inv[h] = __drcp_rn(sigma[h]);
      }
    }
  }
  const float s = static_cast<float>(1 << a.scale_log2);
  uint32_t *img = a.img + static_cast<size_t>(item) * kImgStride;
  for (int k = 0; k < S; ++k) {
    const int row = lane_in * S + k;
    uint32_t w0 = 0, w1 = 0;
    for (int h = 0; h < halves; ++h) {
      const int P = H - m[h];
      const bool real = m[h] > 0 && row >= P;
      float z = 0.0f;
      if (real) {
        const float x = a.events[base[h] + (row - P)];
        z = a.raw ? z_of(x, mean[h], sigma[h], inv[h]) : x;
        // (a query without spread has sigma 0: its quotients are not finite)
        if (!isfinite(z) || fabsf(z) > 1.0e20f) report(a.status, HARU_EINVAL);
      }
      if (packed) {
        const int qv = real ? quantise(z, s) : kPadCode;
        if (real) most = max(most, abs(qv));
        w0 |= (real ? half_code(qv) : kPadHalf) << (16 * h);
        w1 |= (static_cast<uint32_t>(qv) & 0xffffu) << (16 * h);
      } else {
        // FP32: the z-value; exact form: the int16 code as a float; the row
        // weight the sweep multiplies the reference sample by: -1 on real
        // rows (fma(r, -1, q) = q - r, rounded once), 0 on pad rows (which
        // hold q = 0, so their distance is 0)
        w0 = __float_as_uint(codes ? (real ? static_cast<float>(quantise(z, s)) : 0.0f) : z);
        w1 = __float_as_uint(real ? -1.0f : 0.0f);
      }
    }
    img[k * 32 + lane] = w0;
    img[(S + k) * 32 + lane] = w1;
  }
  if (packed) {  // warp-uniform
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) a.items[item].qmax = most;
  }
}

}  // namespace

cudaError_t launch_prep(const PlanArgs &a, const float *events, double *qstats, int sms, cudaStream_t s) {
  StatArgs st{events, a.offsets, a.nq, kStatQueries, qstats};
  // As few queries to a block as leave a block to an SM: the chains share the
  // SM's double-precision unit with the squares of their block's queries.
  // Eight SMs (of 152) stay free of them, one of which runs the planner's block.
  const uint32_t blocks_at_once = static_cast<uint32_t>(sms > 16 ? sms - 8 : 8);
  for (int k : {32, 8})
    if (a.nq <= static_cast<uint32_t>(k) * blocks_at_once) st.per_block = k;
  const unsigned blocks = qstats ? (a.nq + st.per_block - 1) / st.per_block : 0;
  prep_kernel<<<1 + blocks, 1024, 0, s>>>(a, st);
  return cudaGetLastError();
}

cudaError_t load_prep_kernels() {
  cudaFuncAttributes f;
  cudaError_t e = cudaFuncGetAttributes(&f, prep_kernel);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&f, pack_kernel);
  return e;
}

cudaError_t launch_pack(const PackArgs &a, uint32_t max_items, cudaStream_t s) {
  if (max_items == 0) return cudaSuccess;
  const int warps = 8;
  pack_kernel<<<(max_items + warps - 1) / warps, warps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_ref_levels(const uint8_t *bases, size_t n, const float *model, int k, float *out, int *status,
                              cudaStream_t s) {
  const size_t total = 2 * (n - k + 1);
  const int th = 256;
  size_t blocks = (total + th - 1) / th;
  if (blocks > 65535) blocks = 65535;
  ref_levels_kernel<<<static_cast<unsigned>(blocks), th, 0, s>>>(bases, n, model, k, out, status);
  return cudaGetLastError();
}

cudaError_t launch_zscore_stats(const float *x, size_t n, double *partials, double *stats, int *status,
                                cudaStream_t s) {
  const size_t nb = (n + kZBlock - 1) / kZBlock;
  const int th = 128;
  const unsigned blocks = static_cast<unsigned>((nb + th - 1) / th);
  block_sums_kernel<<<blocks, th, 0, s>>>(x, n, stats, 0, partials);
  finish_sums_kernel<<<1, 1, 0, s>>>(partials, nb, n, 0, stats, status);
  block_sums_kernel<<<blocks, th, 0, s>>>(x, n, stats, 1, partials);
  finish_sums_kernel<<<1, 1, 0, s>>>(partials, nb, n, 1, stats, status);
  return cudaGetLastError();
}

cudaError_t launch_ref_finish(const float *x, size_t n, const double *stats, int normalize, int scale_log2,
                              float *z, uint32_t *img16, uint32_t *imgh, float *img32, int *status, int *max_code,
                              cudaStream_t s) {
  const int th = 256;
  size_t blocks = (n + th - 1) / th;
  if (blocks > 65535) blocks = 65535;
  ref_finish_kernel<<<static_cast<unsigned>(blocks), th, 0, s>>>(x, n, stats, normalize,
                                                                 static_cast<float>(1 << scale_log2), z, img16,
                                                                 imgh, img32, status, max_code);
  return cudaGetLastError();
}

}  // namespace haru
