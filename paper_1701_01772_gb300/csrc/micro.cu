// Algorithm 7 (micro-level estimation): per sampled edge e = (u, v) the
// vector x3..x17 of the paper's micro-level graphlet statistics, from
// ceil(d_w p_e) probes of N(w) for every w in the edge's neighbourhood.
//
// For e with d_u <= d_v (ties: smaller id is u), T = N(u) cap N(v),
// S_u = N(u) \ {v} \ T, S_v = N(v) \ {u} \ T. Each w of T, S_u and S_v
// reads a circular window of c_w = ceil(d_w p_e) consecutive entries of
// N(w) from the offset o_w = floor(h d_w / 2^64), h = sm(sm(seed ^ sm(key))
// ^ w), key = (min(u,v) << 32) | max(u,v), sm the SplitMix64 output
// function. A probe r counts, weighted d_w / c_w,
//   w in T:    r in T, r > w                    -> x7 (4-cliques)
//   w in S_u:  r in S_v                         -> x10 (4-cycles)
//              r in S_u, r > w                  -> x9 (tailed triangles)
//              r in T                           -> omega
//   w in S_v:  r in S_v, r > w                  -> x9
//              r in T                           -> omega
// ("r > w": each unordered pair inside a set counts once, from its smaller
// member, as the algorithm's label resets do). The remaining statistics
// follow from t, a = |S_u|, b = |S_v|, R = n - 2 - t - a - b:
//   x3 = t, x4 = a + b, x5 = R, x6 = C(n,3) - x3 - x4 - x5, x8 = C(t,2) - x7,
//   x11 = C(a,2) + C(b,2) - x9, x12 = a b - x10, x13 = t R, x14 = (a+b) R,
//   x15 = m - (t + d_u + d_v + 1) - omega, x16 = C(R,2),
//   x17 = C(n,4) - (x7 + ... + x16).
//
// GPU structure (same flattening as the 4-node pass of count.cu):
//   prep    k_prep of count.cu: orientation, edge check, duplicate check.
//   chunks  the two lists N(u), N(v) of every edge are cut into chunks of
//           32 positions (each list padded to 32); one warp per chunk
//           classifies its positions (T, S_u, S_v or none) with one
//           membership test each, counts t and the chunk's probes, and
//           turns them into tasks of kTaskProbes probes.
//   probe   warps take runs of tasks from a counter; lanes take consecutive
//           probes of a task (item descriptors in shared memory); a probe
//           costs up to two membership tests (in N(v), in N(u)).
//   final   one thread per edge writes the 15 statistics and keeps the
//           column maxima (the extremal statistics of Sec. 7).
// Weighted hits are accumulated exactly: weight d_w / c_w = q + f / 2^64
// with q = floor(d_w / c_w), f = floor((d_w mod c_w) 2^64 / c_w), per edge
// and statistic an integer part and a 128-bit fraction part, added with
// integer atomics (so the result does not depend on the order of the work)
// and converted to FP64 once. At p_e = 1 every weight is 1 and the
// statistics are exact integers.
#include <math.h>
#include <string.h>

#include "common.cuh"

namespace gs {

// count.cu: orientation (u = smaller degree), edge and duplicate checks,
// len[e] = d_u (pad = 0).
__global__ void k_prep(DevGraph g, const int32_t* __restrict__ pairs, int64_t K, int pad,
                       unsigned long long* __restrict__ dup_table, int64_t dup_mask,
                       int2* __restrict__ uv, int64_t* __restrict__ len, DevError* err);

namespace {

constexpr int kThreads = 256;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kProbeBlocksPerSm = 5;
constexpr int64_t kTaskProbes = 512;
// Tasks a probe warp takes from the counter, at most (a run sets its chunks up
// anew: 26.0 / 19.1 / 18.3 ms at 1 / 8 / 32 tasks).
constexpr int kRunTasks = 32;
constexpr int kCats = 4;   // x7, x9, x10, omega
constexpr int kCols = 15;  // x3 .. x17
constexpr int kNone = 0, kT = 1, kSu = 2, kSv = 3;

typedef unsigned __int128 u128;

__device__ __forceinline__ uint64_t splitmix(uint64_t x) {
  uint64_t z = x + 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ int64_t probes_of(int64_t d, double pe) {
  return (int64_t)ceil((double)d * pe);
}

// Per-edge set-up: chunk counts of the two lists.
__global__ void k_micro_chunks(const int64_t* __restrict__ row_ptr, const int2* __restrict__ uv,
                               int64_t K, int64_t* __restrict__ nch,
                               unsigned long long* __restrict__ t,
                               unsigned long long* __restrict__ acc) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 pr = uv[e];
    const int64_t du = __ldg(row_ptr + pr.x + 1) - __ldg(row_ptr + pr.x);
    const int64_t dv = __ldg(row_ptr + pr.y + 1) - __ldg(row_ptr + pr.y);
    nch[e] = ((du + 31) >> 5) + ((dv + 31) >> 5);
    t[e] = 0;
#pragma unroll
    for (int i = 0; i < 3 * kCats; ++i) acc[e * 3 * kCats + i] = 0;
  }
}

// Edge of every chunk. One warp per edge.
__global__ void k_micro_fill(const int64_t* __restrict__ choff, int64_t K,
                             int64_t* __restrict__ chunk_e) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < K; e += warps)
    for (int64_t c = choff[e] + lane; c < choff[e + 1]; c += 32) chunk_e[c] = e;
}

// Where chunk c of edge e lies: list owner (u side: N(u), else N(v)) and
// the first position.
struct ChunkAt {
  int32_t u, v, owner, other;
  int64_t bu, du, bv, dv, bo, dow, bx, dx;  // (bo, dow): owner list, (bx, dx): other's
  int64_t first;
  bool vside;
};

__device__ __forceinline__ ChunkAt chunk_at(const DevGraph& g, const int2* __restrict__ uv,
                                            const int64_t* __restrict__ choff, int64_t e,
                                            int64_t c) {
  ChunkAt a;
  const int2 pr = uv[e];
  a.u = pr.x;
  a.v = pr.y;
  a.bu = __ldg(g.row_ptr + a.u);
  a.du = __ldg(g.row_ptr + a.u + 1) - a.bu;
  a.bv = __ldg(g.row_ptr + a.v);
  a.dv = __ldg(g.row_ptr + a.v + 1) - a.bv;
  const int64_t lc = c - __ldg(choff + e), cu = (a.du + 31) >> 5;
  a.vside = lc >= cu;
  a.first = (a.vside ? lc - cu : lc) * 32;
  a.owner = a.vside ? a.v : a.u;
  a.other = a.vside ? a.u : a.v;
  a.bo = a.vside ? a.bv : a.bu;
  a.dow = a.vside ? a.dv : a.du;
  a.bx = a.vside ? a.bu : a.bv;
  a.dx = a.vside ? a.du : a.dv;
  return a;
}

// Class of position i of a chunk (one membership test in the other list).
__device__ __forceinline__ int classify(const DevGraph& g, const ChunkAt& a, int64_t i,
                                        int32_t* w_out) {
  if (i >= a.dow) return kNone;
  const int32_t w = __ldg(g.col + a.bo + i);
  *w_out = w;
  if (w == a.other) return kNone;
  const int32_t xs = g.col_hm != nullptr ? (int32_t)__ldg(g.col_hm + a.bo + i) : kNoSlotInfo;
  const bool both = adj_contains(g, a.other, a.bx, a.dx, w, xs);
  if (!a.vside) return both ? kT : kSu;
  return both ? kNone : kSv;  // T members are handled from the u side
}

// Classes, t and probe counts per chunk; tasks per chunk.
__global__ void __launch_bounds__(kThreads)
    k_micro_items(DevGraph g, const int2* __restrict__ uv, const int64_t* __restrict__ choff,
                  const int64_t* __restrict__ chunk_e, int64_t C, double pe,
                  unsigned long long* __restrict__ t, uint32_t* __restrict__ tmask,
                  int64_t* __restrict__ task_cnt, unsigned long long* __restrict__ stats) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  unsigned long long probes = 0;
  for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < C; c += warps) {
    const int64_t e = chunk_e[c];
    const ChunkAt a = chunk_at(g, uv, choff, e, c);
    int32_t w = 0;
    const int cls = classify(g, a, a.first + lane, &w);
    int64_t cost = 0;
    if (cls != kNone) cost = probes_of(__ldg(g.row_ptr + w + 1) - __ldg(g.row_ptr + w), pe);
    const unsigned inT = __ballot_sync(kFull, cls == kT);
    const unsigned live = __ballot_sync(kFull, cls != kNone);
    int64_t total = cost;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
    if (lane == 0) {
      tmask[2 * c] = inT;
      tmask[2 * c + 1] = live;
      task_cnt[c] = (total + kTaskProbes - 1) / kTaskProbes;
      if (inT) atomicAdd(t + e, (unsigned long long)__popc(inT));
      probes += (unsigned long long)total;
    }
  }
  if (lane == 0 && probes) atomicAdd(stats, probes);
}

// The items of the chunk a warp works on (live positions only, in order),
// field by field so that lanes that read different items hit different banks.
struct WarpItems {
  int64_t bw[32];  // start of N(w)
  int32_t dw[32], o[32], w[32];
  uint16_t who[32];  // position in the chunk
  uint8_t cls[32];
};

// Adds a 64-bit integer part and a 128-bit fraction to an edge's
// accumulator {I, F_lo, F_hi} with integer atomics (exact, order-free).
__device__ __forceinline__ void acc_add(unsigned long long* a, unsigned long long I, u128 F) {
  if (I) atomicAdd(a, I);
  const unsigned long long lo = (unsigned long long)F, hi = (unsigned long long)(F >> 64);
  if (lo) {
    const unsigned long long old = atomicAdd(a + 1, lo);
    if (old + lo < old) atomicAdd(a + 2, 1ull);
  }
  if (hi) atomicAdd(a + 2, hi);
}

__device__ __forceinline__ u128 shfl_xor_u128(u128 v, int o) {
  unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
  lo = __shfl_xor_sync(kFull, lo, o);
  hi = __shfl_xor_sync(kFull, hi, o);
  return ((u128)hi << 64) | lo;
}

// Statistic (0: x7, 1: x9, 2: x10, 3: omega, -1: none) of a probe that read x
// from N(w). v is tested first; u only where its answer matters.
__device__ __forceinline__ int probe_cat(const EndSet& su, const EndSet& sv, int32_t u, int32_t v,
                                         int cls, int32_t w, int32_t x, int32_t xs) {
  const bool above = x > w;
  if (cls == kT) return above && set_has(sv, x, xs) && set_has(su, x, xs) ? 0 : -1;
  if (x == u || x == v) return -1;
  const bool in_v = set_has(sv, x, xs);
  if (!in_v && !(cls == kSu && above)) return -1;
  const bool in_u = set_has(su, x, xs);
  if (!in_v) return in_u ? 1 : -1;                  // S_u pair
  if (in_u) return 3;                               // omega
  return cls == kSu ? 2 : above ? 1 : -1;           // 4-cycle; S_v pair
}

// Probes. A chunk's probes (its items in order) are one index space cut into
// tasks; warps take runs of tasks from a counter. From probe r on a warp walks
// either a run of 32 or more probes of one item (its descriptor is the same in
// every lane) or 32 probes of several items, found from a bit mask of the item
// starts among them. Lane i owns item i: it counts the item's hits per
// statistic (from the hit ballots, whose bits [start, end) are the item's
// probes), and the item's weight d_w / c_w multiplies the counts once per
// chunk. Issue bound before: five shuffles to find the item, two general
// membership look-ups and 4 x 192-bit predicated additions per probe. 20,000
// edges of the 100k-vertex power-law graph at p_e = 0.1 (2.1e9 probes): 29.2
// -> 18.3 ms for the whole call (20.8 / 20.2 / 19.1 / 19.3 ms at 3 / 4 / 5 / 6
// CTAs per SM and runs of 8 tasks).
__global__ void __launch_bounds__(kThreads, kProbeBlocksPerSm)
    k_micro_probe(const __grid_constant__ DevGraph g, const int2* __restrict__ uv,
                  const int64_t* __restrict__ choff, const int64_t* __restrict__ chunk_e,
                  const uint32_t* __restrict__ tmask, const int64_t* __restrict__ task_off,
                  int64_t C, double pe, uint64_t seed, unsigned long long* __restrict__ acc,
                  unsigned long long* __restrict__ counter) {
  __shared__ WarpItems items[kThreads / 32];
  const int lane = threadIdx.x & 31;
  const unsigned upto = kFull >> (31 - lane);
  WarpItems* my = items + (threadIdx.x >> 5);
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  // at least eight runs per warp, at most kRunTasks tasks each
  const int64_t share = __ldg(task_off + C) / (warps * 8);
  const int grab = share < 1 ? 1 : share < kRunTasks ? (int)share : kRunTasks;
  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(counter, (unsigned long long)grab);
    int64_t task = (int64_t)__shfl_sync(kFull, got, 0);
    int left = (int)min((int64_t)grab, __ldg(task_off + C) - task);
    if (left <= 0) break;
    int64_t c = last_le_warp(task_off, C, task);
    while (left > 0) {
      while (__ldg(task_off + c + 1) <= task) ++c;
      int here = (int)min((int64_t)left, __ldg(task_off + c + 1) - task);
      left -= here;
      const int64_t e = chunk_e[c];
      const ChunkAt a = chunk_at(g, uv, choff, e, c);
      const EndSet su = end_set(g, a.u, a.bu, a.du), sv = end_set(g, a.v, a.bv, a.dv);
      const bool slots = su.mrow != nullptr || sv.mrow != nullptr;
      const uint32_t inT = tmask[2 * c], alive = tmask[2 * c + 1];
      const int live = __popc(alive);
      __syncwarp();  // the previous chunk's items are no longer read
      if ((alive >> lane) & 1u) my->who[__popc(alive & ((1u << lane) - 1u))] = (uint16_t)lane;
      __syncwarp();
      int64_t mine = 0;
      uint64_t q = 0, f = 0;  // weight d_w / c_w = q + f / 2^64 of the lane's item
      if (lane < live) {
        const int at = my->who[lane];
        const int32_t w = __ldg(g.col + a.bo + a.first + at);
        const int64_t bw = __ldg(g.row_ptr + w);
        const uint32_t dw = (uint32_t)(__ldg(g.row_ptr + w + 1) - bw);  // < 2^31
        mine = probes_of((int64_t)dw, pe);
        const uint64_t key = ((uint64_t)(uint32_t)min(a.u, a.v) << 32) | (uint32_t)max(a.u, a.v);
        const uint64_t hh = splitmix(splitmix(seed ^ splitmix(key)) ^ (uint64_t)(uint32_t)w);
        my->bw[lane] = bw;
        my->dw[lane] = (int32_t)dw;
        my->o[lane] = (int32_t)__umul64hi(hh, (uint64_t)dw);
        my->w[lane] = w;
        my->cls[lane] = (uint8_t)(a.vside ? kSv : (((inT >> at) & 1u) ? kT : kSu));
        const uint32_t cw = (uint32_t)mine;
        q = dw / cw;
        // floor((d_w mod c_w) 2^64 / c_w), 32 bits of the quotient at a time
        const uint64_t r0 = (uint64_t)(dw % cw) << 32;
        const uint64_t r1 = (r0 % cw) << 32;
        f = ((r0 / cw) << 32) | (r1 / cw);
      }
      __syncwarp();
      int64_t start = mine;  // first probe of the item; the total past the items
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, start, s);
        if (lane >= s) start += y;
      }
      const int64_t ctotal = __shfl_sync(kFull, start, 31);
      start -= mine;
      unsigned cnt[kCats];
#pragma unroll
      for (int k = 0; k < kCats; ++k) cnt[k] = 0;
      for (; here > 0; --here, ++task) {
        const int64_t lo = (task - __ldg(task_off + c)) * kTaskProbes;
        const int32_t len = (int32_t)min(ctotal - lo, kTaskProbes);
        // item starts relative to the task's first probe, clamped to 32 bits
        // (order kept; the item holding a probe of this task starts less than
        // one item's probes before lo)
        const int32_t srel = (int32_t)max(min(start - lo, kTaskProbes), (int64_t)INT32_MIN + 1);
        const int32_t sd = __shfl_down_sync(kFull, srel, 1);
        const int32_t se = lane < 31 ? min(sd, len) : len;
        for (int32_t r = 0; r < len;) {
          const int j0 = 31 - __clz(__ballot_sync(kFull, srel <= r));
          const int32_t sj = __shfl_sync(kFull, srel, j0);
          const int32_t end = __shfl_sync(kFull, se, j0);
          if (end - r >= 32) {
            const int32_t dw = my->dw[j0], w = my->w[j0];
            const int64_t bw = my->bw[j0];
            const int cls = my->cls[j0];
            // position in the window; o < d_w and fewer than d_w probes, so
            // the sum can pass 2^31
            uint32_t p = (uint32_t)my->o[j0] + (uint32_t)(r - sj) + lane;
            unsigned c1 = 0, c2 = 0, c3 = 0;
            for (; end - r >= 32; r += 32, p += 32) {
              const uint32_t pp = p >= (uint32_t)dw ? p - (uint32_t)dw : p;
              const int32_t x = __ldg(g.col + bw + pp);
              const int32_t xs = slots ? (int32_t)__ldg(g.col_hm + bw + pp) : -1;
              const int cat = probe_cat(su, sv, a.u, a.v, cls, w, x, xs);
              c1 += cat == 0 || cat == 1;
              c2 += cat == 2;
              c3 += cat == 3;
            }
            c1 = __reduce_add_sync(kFull, c1);
            if (cls != kT) {
              c2 = __reduce_add_sync(kFull, c2);
              c3 = __reduce_add_sync(kFull, c3);
            }
            if (lane == j0) {
              cnt[0] += cls == kT ? c1 : 0u;
              cnt[1] += cls == kT ? 0u : c1;
              cnt[2] += c2;
              cnt[3] += c3;
            }
            continue;
          }
          const int32_t ds = srel - r;
          const unsigned marks = __reduce_or_sync(kFull, ds > 0 && ds < 32 ? 1u << ds : 0u);
          const int j = min(j0 + __popc(marks & upto), 31);
          const int32_t o = r + lane - __shfl_sync(kFull, srel, j);
          int cat = -1;
          if (r + lane < len) {
            const uint32_t dw = (uint32_t)my->dw[j];
            uint32_t pp = (uint32_t)my->o[j] + (uint32_t)o;
            if (pp >= dw) pp -= dw;
            const int32_t x = __ldg(g.col + my->bw[j] + pp);
            const int32_t xs = slots ? (int32_t)__ldg(g.col_hm + my->bw[j] + pp) : -1;
            cat = probe_cat(su, sv, a.u, a.v, my->cls[j], my->w[j], x, xs);
          }
          const unsigned range = bits_below(se - r) & ~bits_below(srel - r);
#pragma unroll
          for (int k = 0; k < kCats; ++k)
            cnt[k] += __popc(__ballot_sync(kFull, cat == k) & range);
          r += 32;
        }
      }
      // weighted counts to the edge
#pragma unroll
      for (int k = 0; k < kCats; ++k) {
        if (!__any_sync(kFull, cnt[k] != 0)) continue;
        unsigned long long I = (unsigned long long)cnt[k] * q;
        u128 F = (u128)cnt[k] * f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          I += __shfl_xor_sync(kFull, I, o);
          F += shfl_xor_u128(F, o);
        }
        if (lane == 0) acc_add(acc + e * 3 * kCats + 3 * k, I, F);
      }
    }
  }
}

__device__ __forceinline__ double acc_value(const unsigned long long* a) {
  // I + (F_hi 2^64 + F_lo) / 2^64
  return (double)(a[0] + a[2]) + (double)a[1] * 0x1p-64;
}

struct ColMax {
  double v;
  int64_t i;
};

__device__ __forceinline__ bool better(double v, int64_t i, const ColMax& m) {
  return v > m.v || (v == m.v && i < m.i);
}

// Rows x3..x17 and per-block column maxima (value, smallest edge index).
__global__ void __launch_bounds__(kThreads)
    k_micro_final(const int64_t* __restrict__ row_ptr, const int2* __restrict__ uv, int64_t K,
                  int64_t n, int64_t m, double cn3, double cn4,
                  const unsigned long long* __restrict__ t,
                  const unsigned long long* __restrict__ acc, double* __restrict__ x,
                  ColMax* __restrict__ part) {
  __shared__ ColMax red[kThreads / 32][kCols];
  ColMax best[kCols];
#pragma unroll
  for (int k = 0; k < kCols; ++k) best[k] = ColMax{-INFINITY, INT64_MAX};
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 pr = uv[e];
    const int64_t du = __ldg(row_ptr + pr.x + 1) - __ldg(row_ptr + pr.x);
    const int64_t dv = __ldg(row_ptr + pr.y + 1) - __ldg(row_ptr + pr.y);
    const int64_t tt = (int64_t)t[e], a = du - 1 - tt, b = dv - 1 - tt;
    const int64_t R = n - 2 - tt - a - b;
    const unsigned long long* ac = acc + e * 3 * kCats;
    const double x7 = acc_value(ac), x9 = acc_value(ac + 3), x10 = acc_value(ac + 6);
    const double om = acc_value(ac + 9);
    double r[kCols];
    r[0] = (double)tt;
    r[1] = (double)(a + b);
    r[2] = (double)R;
    r[3] = cn3;  // C(n,3) - t - (a+b) - R = C(n,3) - (n - 2), rounded on the host
    r[4] = x7;
    r[5] = (double)(tt * (tt - 1) / 2) - x7;
    r[6] = x9;
    r[7] = x10;
    r[8] = (double)(a * (a - 1) / 2 + b * (b - 1) / 2) - x9;
    r[9] = (double)(a * b) - x10;
    r[10] = (double)(tt * R);
    r[11] = (double)((a + b) * R);
    r[12] = (double)(m - (tt + du + dv + 1)) - om;
    r[13] = (double)(R * (R - 1) / 2);
    double s = 0.0;
#pragma unroll
    for (int k = 4; k <= 13; ++k) s += r[k];
    r[14] = cn4 - s;
#pragma unroll
    for (int k = 0; k < kCols; ++k) {
      x[e * kCols + k] = r[k];
      if (better(r[k], e, best[k])) best[k] = ColMax{r[k], e};
    }
  }
  if (part == nullptr) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kCols; ++k) {
    ColMax b = best[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(kFull, b.v, o);
      const long long oi = __shfl_xor_sync(kFull, (long long)b.i, o);
      if (better(ov, oi, b)) b = ColMax{ov, oi};
    }
    if (lane == 0) red[wid][k] = b;
  }
  __syncthreads();
  if (threadIdx.x < kCols) {
    ColMax b = red[0][threadIdx.x];
    for (int i = 1; i < kThreads / 32; ++i) {
      const ColMax& c = red[i][threadIdx.x];
      if (better(c.v, c.i, b)) b = c;
    }
    part[(int64_t)blockIdx.x * kCols + threadIdx.x] = b;
  }
}

__global__ void k_micro_max_final(const ColMax* __restrict__ part, int blocks,
                                  ColMax* __restrict__ out) {
  if (threadIdx.x < kCols) {
    ColMax b = part[threadIdx.x];
    for (int i = 1; i < blocks; ++i) {
      const ColMax& c = part[(int64_t)i * kCols + threadIdx.x];
      if (better(c.v, c.i, b)) b = c;
    }
    out[threadIdx.x] = b;
  }
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" gs_status gs_micro(const gs_graph* gr, gs_workspace* ws, const int32_t* d_pairs,
                              int64_t K, double p_e, uint64_t seed, double* d_x, double* h_max,
                              int64_t* h_argmax, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || K < 0 || !(p_e > 0.0 && p_e <= 1.0) ||
      (K > 0 && (d_pairs == nullptr || d_x == nullptr))) {
    set_error("gs_micro: invalid arguments (need 0 < p_e <= 1, device pairs and output)");
    return GS_EINVAL;
  }
  memset(&ws->stats, 0, sizeof(ws->stats));
  ws->stats.k = K;
  if (h_max != nullptr)
    for (int k = 0; k < kCols; ++k) h_max[k] = NAN;
  if (h_argmax != nullptr)
    for (int k = 0; k < kCols; ++k) h_argmax[k] = -1;
  if (K == 0) return GS_OK;
  const DevGraph& g = gr->dev;
  const int64_t n = g.n, m = gr->m;
  // C(n,3) - (n - 2) and C(n,4), exact in 128 bits, rounded once
  const unsigned __int128 N = (unsigned __int128)n;
  const unsigned __int128 c3 = n >= 3 ? N * (N - 1) * (N - 2) / 6 : 0;
  const unsigned __int128 c4 = n >= 4 ? N * (N - 1) / 2 * (N - 2) * (N - 3) / 12 : 0;
  const double cn3 = (double)(c3 - (unsigned __int128)(n - 2));
  const double cn4 = (double)c4;

  int64_t dup_cap = 1;
  while (dup_cap < 2 * K) dup_cap <<= 1;
  const int final_blocks = grid_for(K, kThreads, 1);
  const size_t front = Carve::bytes_for<DevError>(1) + Carve::bytes_for<unsigned long long>(8) +
                       Carve::bytes_for<int2>(K) + Carve::bytes_for<int64_t>(K + 1) * 2 +
                       Carve::bytes_for<unsigned long long>(K) +
                       Carve::bytes_for<unsigned long long>(K * 3 * kCats) +
                       Carve::bytes_for<int64_t>(scan_tmp_elems(K + 1)) +
                       Carve::bytes_for<unsigned long long>(dup_cap) +
                       Carve::bytes_for<ColMax>((int64_t)final_blocks * kCols + kCols);
  void* base0 = nullptr;
  GS_TRY(ws_reserve(ws, 0, front, stream, &base0));
  Carve c0{(char*)base0, 0};
  DevError* err = c0.take<DevError>(1);
  unsigned long long* stats = c0.take<unsigned long long>(8);
  int2* uv = c0.take<int2>(K);
  int64_t* len = c0.take<int64_t>(K + 1);
  int64_t* choff = c0.take<int64_t>(K + 1);
  unsigned long long* t = c0.take<unsigned long long>(K);
  unsigned long long* acc = c0.take<unsigned long long>(K * 3 * kCats);
  int64_t* tmp0 = c0.take<int64_t>(scan_tmp_elems(K + 1));
  unsigned long long* dup = c0.take<unsigned long long>(dup_cap);
  ColMax* part = c0.take<ColMax>((int64_t)final_blocks * kCols);
  ColMax* best = c0.take<ColMax>(kCols);

  GS_CUDA(cudaMemsetAsync(err, 0, sizeof(DevError), stream));
  GS_CUDA(cudaMemsetAsync(stats, 0, sizeof(unsigned long long) * 8, stream));
  GS_CUDA(cudaMemsetAsync(dup, 0xff, sizeof(unsigned long long) * dup_cap, stream));
  k_prep<<<grid_for(K, kThreads, 8), kThreads, 0, stream>>>(g, d_pairs, K, 0, dup, dup_cap - 1,
                                                            uv, len, err);
  k_micro_chunks<<<grid_for(K, kThreads, 8), kThreads, 0, stream>>>(g.row_ptr, uv, K, choff, t,
                                                                     acc);
  GS_TRY(exclusive_scan_i64(choff, choff, K, tmp0, stream));
  DevError herr;
  int64_t C = 0;
  GS_CUDA(cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaMemcpyAsync(&C, choff + K, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  if (herr.code != 0) {
    set_error("gs_micro: %s (pair %lld)",
              herr.code == GS_EDUPSAMPLE ? "edge sampled twice"
                                         : "sampled pair is out of range or not an edge",
              (long long)herr.index);
    return herr.code;
  }
  int64_t launches = 2 + scan_launches(K);
  if (C > 0) {
    const size_t mid = Carve::bytes_for<int64_t>(C) + Carve::bytes_for<uint32_t>(2 * C) +
                       Carve::bytes_for<int64_t>(C + 1) +
                       Carve::bytes_for<int64_t>(scan_tmp_elems(C + 1));
    void* base1 = nullptr;
    GS_TRY(ws_reserve(ws, 1, mid, stream, &base1));
    Carve c1{(char*)base1, 0};
    int64_t* chunk_e = c1.take<int64_t>(C);
    uint32_t* tmask = c1.take<uint32_t>(2 * C);
    int64_t* task_off = c1.take<int64_t>(C + 1);
    int64_t* tmp1 = c1.take<int64_t>(scan_tmp_elems(C + 1));
    k_micro_fill<<<grid_for(K * 32, kThreads, 8), kThreads, 0, stream>>>(choff, K, chunk_e);
    k_micro_items<<<grid_for(C * 32, kThreads, 8), kThreads, 0, stream>>>(
        g, uv, choff, chunk_e, C, p_e, t, tmask, task_off, stats);
    GS_TRY(exclusive_scan_i64(task_off, task_off, C, tmp1, stream));
    k_micro_probe<<<sm_count() * kProbeBlocksPerSm, kThreads, 0, stream>>>(
        g, uv, choff, chunk_e, tmask, task_off, C, p_e, seed, acc, stats + 1);
    launches += 3 + scan_launches(C);
  }
  k_micro_final<<<final_blocks, kThreads, 0, stream>>>(
      g.row_ptr, uv, K, n, m, cn3, cn4, t, acc, d_x,
      (h_max != nullptr || h_argmax != nullptr) ? part : nullptr);
  ++launches;
  GS_CUDA(cudaGetLastError());
  unsigned long long hs[8];
  GS_CUDA(cudaMemcpyAsync(hs, stats, sizeof(hs), cudaMemcpyDeviceToHost, stream));
  if (h_max != nullptr || h_argmax != nullptr) {
    k_micro_max_final<<<1, 32, 0, stream>>>(part, final_blocks, best);
    ++launches;
    GS_CUDA(cudaGetLastError());
    ColMax hb[kCols];
    GS_CUDA(cudaMemcpyAsync(hb, best, sizeof(hb), cudaMemcpyDeviceToHost, stream));
    GS_CUDA(cudaStreamSynchronize(stream));
    for (int k = 0; k < kCols; ++k) {
      if (h_max != nullptr) h_max[k] = hb[k].v;
      if (h_argmax != nullptr) h_argmax[k] = hb[k].i;
    }
  }
  GS_CUDA(cudaStreamSynchronize(stream));
  ws->stats.micro_probes = (int64_t)hs[0];
  ws->stats.launches = launches;
  ws->launches_total += launches;
  return GS_OK;
}
