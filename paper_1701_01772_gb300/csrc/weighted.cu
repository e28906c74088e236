// Fixed-size uniform edge sampling (Algorithm 1 with a sample size K,
// without replacement: the K edges of smallest sampler key), weighted edge
// sampling (Algorithm 1 with a non-uniform distribution F,
// Sec. 3.1: edges drawn by k-core numbers, degrees or any vertex property),
// the k-core numbers it is usually weighted by (the extremal problem of
// Sec. 7 samples edges of large k-core number), and the estimators with a
// per-edge inverse inclusion probability (Sec. 2.3's sigma = 1/p applied
// edge by edge: Horvitz-Thompson).
//
// Edge weight w_e = min(w[u], w[v]) for a vertex weight w (with core
// numbers: the edge's own core number). Each canonical edge i (the i-th
// pair u < v in row-major CSR order) is kept independently with
// probability pi_e = min(1, s w_e), s = fraction M / W, W = sum_e w_e, by
// the uniform sampler's key: keep iff (sm(seed ^ sm(i)) >> 11) <
// floor(pi_e 2^53). The estimate of graphlet i is
//   X_i = sum_{e in J} N_i(e) / (D_i pi_e),
//   V_i = sum_{e in J} (1 - pi_e) N_i(e)^2 / (D_i^2 pi_e^2),
// with N_i the per-edge numerators of gs_count. pi_e depends only on the
// integer w_e, so the library folds exact 128-bit sums of N_i and N_i^2 per
// weight class on the device and the host evaluates the FP64 sums over the
// classes in increasing weight.
//
// k-core numbers by parallel peeling (k_core_peel).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace gs {

namespace {

constexpr int kThreads = 256;
constexpr unsigned kFull = 0xffffffffu;
constexpr int64_t kMaxClasses = (int64_t)1 << 22;
constexpr int kSampItems = 16;
constexpr int64_t kSampTile = (int64_t)kThreads * kSampItems;

typedef unsigned __int128 u128;
typedef __int128 i128;

__device__ __forceinline__ uint64_t splitmix(uint64_t x) {
  uint64_t z = x + 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// ------------------------------------------------------------------ k-core

// The whole peeling is one cooperative kernel. At each level k the remaining
// vertices are scanned: those of current degree <= k get core number k and
// are listed for removal, the others are listed again (so later scans are
// shorter) and their least degree is kept; if none was removed, k jumps to
// it. Removing a vertex takes one from every remaining neighbour; the one
// subtraction that takes a neighbour from k + 1 to k removes that neighbour in
// the same level. The list of removals holds (vertex, part) entries of
// kPeelPart neighbours, so a hub is spread over many warps; a warp removes the
// vertices that its own subtractions expose at once, from a queue in shared
// memory, and only what does not fit the queue goes to the next round.
//
// Bound by latency: a level is a few chains of dependent subtractions. A host
// loop with a launch and a wait per level and per round, one warp per vertex,
// took 917 launches on the 100k-vertex power-law graph (a hub's 24,000
// neighbours were one warp's walk): core numbers 23.1 -> 3.7 ms. With few levels
// it is the lists' traffic: entries are listed and counted once per warp, not by
// two additions per vertex at one address, and the first level is the least
// degree (4-regular graph of 8M vertices 10.1 -> 6.7 ms; 1.5 with the host loop),
// and short entries share a warp's step (6.7 -> 1.2; R-MAT 22 9.4 -> 8.6).
constexpr int kPeelThreads = 512;
constexpr int64_t kPeelPart = 256;  // neighbours per removal entry
constexpr int kPeelQueue = 16;      // queued vertices of a warp
// Looks at the barrier counter before a block gives up on the others (each
// takes at least 100 ns, so at least 25 s; a round of removals is over in
// milliseconds, since a warp's queue does not wrap: a long path goes on in the
// next round after kPeelQueue steps).
constexpr int64_t kPeelSpins = (int64_t)1 << 28;

// Counters of one phase (a scan or a round of removals).
struct PeelPhase {
  unsigned long long entries;  // removal entries listed
  unsigned long long remaining;
  unsigned long long least;    // least remaining degree above k
  unsigned long long removed;  // vertices given a core number by the scan
};

struct PeelState {
  PeelPhase phase[4];
  unsigned long long arrived;  // barrier: blocks that came, over all barriers
  int32_t failed;              // a barrier ran out of looks
  int32_t max_core;
};

// Grid-wide barrier of a cooperative launch. False (in every thread of the
// block) when it ran out of looks or another block did.
__device__ __forceinline__ bool peel_barrier(PeelState* st, int64_t most) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned long long n = gridDim.x;
    const unsigned long long mine = atomicAdd(&st->arrived, 1ull);
    const unsigned long long all = (mine / n + 1) * n;
    volatile unsigned long long* arrived = &st->arrived;
    volatile int32_t* failed = &st->failed;
    int64_t looks = 0;
    while (*arrived < all && *failed == 0 && looks < most) ++looks;
    if (*arrived < all) *failed = 1;
    ok = *failed == 0;
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Lists the removal entries of v.
__device__ __forceinline__ void list_removal(int32_t v, int64_t d, int2* __restrict__ list,
                                             unsigned long long* __restrict__ entries) {
  const int64_t parts = (d + kPeelPart - 1) / kPeelPart;
  if (parts == 0) return;
  const unsigned long long at = atomicAdd(entries, (unsigned long long)parts);
  for (int64_t i = 0; i < parts; ++i) list[at + i] = make_int2(v, (int32_t)i);
}

__global__ void __launch_bounds__(kPeelThreads)
    k_core_peel(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t n,
                int32_t* __restrict__ deg, int32_t* __restrict__ core, int32_t* rem0,
                int32_t* rem1, int2* list0, int2* list1, PeelState* st, int64_t most) {
  __shared__ int32_t queue[kPeelThreads / 32][kPeelQueue];
  __shared__ int32_t queued[kPeelThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t threads = (int64_t)gridDim.x * blockDim.x;
  const int64_t warp = thread >> 5, warps = threads >> 5;
  // the least degree of all is the first level; slot 3 keeps it until phase 1
  unsigned long long first_k = ~0ull;
  for (int64_t v = thread; v < n; v += threads) {
    const int32_t d = (int32_t)(row_ptr[v + 1] - row_ptr[v]);
    deg[v] = d;
    core[v] = -1;
    first_k = min(first_k, (unsigned long long)d);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) first_k = min(first_k, __shfl_xor_sync(kFull, first_k, o));
  if (lane == 0 && first_k != ~0ull) atomicMin(&st->phase[3].least, first_k);
  // phase ph uses slot ph & 3; the slot of phase ph + 2 was last read before
  // the barrier that ended phase ph - 1, so it is cleared in phase ph
  int ph = 0;
  auto begin = [&]() {
    if (thread == 0) {
      PeelPhase* z = &st->phase[(ph + 2) & 3];
      z->entries = 0;
      z->remaining = 0;
      z->least = ~0ull;
      z->removed = 0;
    }
    return &st->phase[ph & 3];
  };
  if (!peel_barrier(st, most)) return;
  int64_t remaining = n;
  bool first = true;
  int32_t k = (int32_t)__ldcg(&st->phase[3].least);
  while (remaining > 0) {
    // scan
    PeelPhase* p = begin();
    unsigned long long least = ~0ull;
    unsigned out = 0;  // removed by the lane
    for (int64_t i0 = warp * 32; i0 < remaining; i0 += threads) {
      const int64_t i = i0 + lane;
      const int32_t v = i >= remaining ? -1 : first ? (int32_t)i : __ldcg(rem0 + i);
      bool stays = false;
      int parts = 0;
      if (v >= 0 && __ldcg(core + v) == -1) {
        const int32_t d = __ldcg(deg + v);
        if (d <= k) {
          __stcg(core + v, k);
          ++out;
          parts = (int)((__ldg(row_ptr + v + 1) - __ldg(row_ptr + v) + kPeelPart - 1) / kPeelPart);
        } else {
          stays = true;
          least = min(least, (unsigned long long)d);
        }
      }
      if (__any_sync(kFull, parts > 0)) {  // one place in the list for the warp's entries
        int upto = parts;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kFull, upto, o);
          if (lane >= o) upto += y;
        }
        unsigned long long to = 0;
        if (lane == 31) to = atomicAdd(&p->entries, (unsigned long long)upto);
        to = __shfl_sync(kFull, to, 31) + (upto - parts);
        for (int j = 0; j < parts; ++j) __stcg(list0 + to + j, make_int2(v, j));
      }
      const unsigned b = __ballot_sync(kFull, stays);
      unsigned long long at = 0;
      if (lane == 0 && b) at = atomicAdd(&p->remaining, (unsigned long long)__popc(b));
      at = __shfl_sync(kFull, at, 0);
      if (stays) __stcg(rem1 + at + __popc(b & ((1u << lane) - 1u)), v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) least = min(least, __shfl_xor_sync(kFull, least, o));
    if (lane == 0 && least != ~0ull) atomicMin(&p->least, least);
    out = __reduce_add_sync(kFull, out);
    if (lane == 0 && out) atomicAdd(&p->removed, (unsigned long long)out);
    if (!peel_barrier(st, most)) return;
    ++ph;
    remaining = (int64_t)__ldcg(&p->remaining);
    const unsigned long long low = __ldcg(&p->least);
    int64_t entries = (int64_t)__ldcg(&p->entries);
    const bool any = __ldcg(&p->removed) != 0;
    first = false;
    int32_t* t = rem0;
    rem0 = rem1;
    rem1 = t;
    if (!any) {  // no vertex of degree <= k left: jump
      if (low == ~0ull) break;
      k = (int32_t)low;
      continue;
    }
    if (thread == 0) st->max_core = k;
    // rounds of removals
    int2* from = list0;
    int2* to = list1;
    while (entries > 0) {
      p = begin();
      // takes one from every remaining vertex among x; every look and every
      // subtraction in flight at once (in a loop they were one chain of 24
      // latencies)
      constexpr int kEach = (int)(kPeelPart / 32);
      auto take_away = [&](const int32_t (&x)[kEach]) {
        int32_t old[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u) old[u] = x[u] >= 0 ? __ldcg(core + x[u]) : 0;
#pragma unroll
        for (int u = 0; u < kEach; ++u) old[u] = old[u] == -1 ? atomicSub(deg + x[u], 1) : -1;
#pragma unroll
        for (int u = 0; u < kEach; ++u)
          if (old[u] == k + 1) {
            __stcg(core + x[u], k);
            const int64_t d = __ldg(row_ptr + x[u] + 1) - __ldg(row_ptr + x[u]);
            const int at = d <= kPeelPart ? atomicAdd(&queued[wid], 1) : kPeelQueue;
            if (at < kPeelQueue) queue[wid][at] = x[u];
            else list_removal(x[u], d, to, &p->entries);
          }
      };
      auto part = [&](int32_t v, int32_t i) {
        const int64_t b = __ldg(row_ptr + v) + (int64_t)i * kPeelPart;
        const int64_t e = min(__ldg(row_ptr + v + 1), b + kPeelPart);
        int32_t x[kEach];
#pragma unroll
        for (int u = 0; u < kEach; ++u)
          x[u] = b + 32 * u + lane < e ? __ldg(col + b + 32 * u + lane) : -1;
        take_away(x);
      };
      // with entries for all warps, a warp takes kEach of them at once: short
      // ones fill the places of one part
      const bool many = entries >= warps * kEach;
      const int64_t step = many ? kEach : 1;
      for (int64_t i = warp * step; i < entries; i += warps * step) {
        if (lane == 0) queued[wid] = 0;
        __syncwarp();
        if (many) {
          int2 it = make_int2(-1, 0);
          int64_t b = 0;
          int32_t len = 0;
          if (lane < kEach && i + lane < entries) {
            it = __ldcg(from + i + lane);
            b = __ldg(row_ptr + it.x) + (int64_t)it.y * kPeelPart;
            len = (int32_t)min(__ldg(row_ptr + it.x + 1) - b, kPeelPart);
          }
          if (__all_sync(kFull, len <= 32)) {
            int32_t x[kEach];
#pragma unroll
            for (int u = 0; u < kEach; ++u) {
              const int64_t bu = __shfl_sync(kFull, b, u);
              x[u] = lane < __shfl_sync(kFull, len, u) ? __ldg(col + bu + lane) : -1;
            }
            take_away(x);
          } else {
            for (int u = 0; u < kEach && i + u < entries; ++u)
              part(__shfl_sync(kFull, it.x, u), __shfl_sync(kFull, it.y, u));
          }
        } else {
          const int2 it = __ldcg(from + i);
          part(it.x, it.y);
        }
        for (int head = 0;; ++head) {
          __syncwarp();
          if (head >= min(queued[wid], kPeelQueue)) break;
          part(queue[wid][head], 0);
        }
        __syncwarp();
      }
      if (!peel_barrier(st, most)) return;
      ++ph;
      entries = (int64_t)__ldcg(&p->entries);
      int2* l = from;
      from = to;
      to = l;
    }
    ++k;
  }
}

// ------------------------------------------------------------------ sampler

__device__ __forceinline__ int32_t edge_weight(const int32_t* __restrict__ vw, int32_t u,
                                               int32_t v) {
  const int32_t a = __ldg(vw + u), b = __ldg(vw + v);
  return a < b ? a : b;
}

// W = sum of edge weights, the largest vertex weight seen and whether any
// weight is negative. One warp per vertex over its upper neighbours.
__global__ void k_weight_sum(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                             const int64_t* __restrict__ up_ptr, const int32_t* __restrict__ vw,
                             int64_t n, unsigned long long* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  unsigned long long s = 0, neg = 0;
  for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += warps) {
    if (lane == 0 && __ldg(vw + u) < 0) neg = 1;
    for (int64_t p = up_ptr[u] + lane; p < row_ptr[u + 1]; p += 32) {
      const int32_t w = edge_weight(vw, (int32_t)u, col[p]);
      s += (unsigned long long)(w > 0 ? w : 0);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(kFull, s, o);
    neg |= __shfl_xor_sync(kFull, neg, o);
  }
  if (lane == 0) {
    if (s) atomicAdd(out, s);
    if (neg) atomicOr(out + 1, 1ull);
  }
}

__device__ __forceinline__ uint64_t keep_threshold(double scale, int32_t w) {
  double pi = scale * (double)w;
  if (pi > 1.0) pi = 1.0;
  return (uint64_t)floor(pi * 9007199254740992.0);
}

// keep[i] for every canonical edge. Warps take equal contiguous ranges of the
// edges (a warp per vertex left a hub's edges to one warp: 0.53 of 5.8 ms of a
// weighted estimate on the 100k-vertex power-law graph).
__global__ void __launch_bounds__(kThreads)
    k_weighted_flags(const int32_t* __restrict__ col, const int64_t* __restrict__ up_ptr,
                     const int64_t* __restrict__ edge_off, const int32_t* __restrict__ vw,
                     int64_t n, int64_t m, double scale, uint64_t seed,
                     uint8_t* __restrict__ keep) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t per = ((m + 31) / 32 + warps - 1) / warps * 32;
  const int64_t i0 = warp * per, i1 = min(m, i0 + per);
  if (i0 >= i1) return;
  int64_t u = last_le_warp(edge_off, n, i0);  // the row of the canonical edge
  for (int64_t ib = i0; ib < i1; ib += 32) {
    const int64_t i = ib + lane;
    u = last_le_lanes(edge_off, n, u, min(i, i1 - 1));
    if (i < i1) {
      const int32_t v = __ldg(col + up_ptr[u] + (i - __ldg(edge_off + u)));
      const uint64_t key = splitmix(seed ^ splitmix((uint64_t)i)) >> 11;
      keep[i] = key < keep_threshold(scale, edge_weight(vw, (int32_t)u, v)) ? 1 : 0;
    }
    u = __shfl_sync(kFull, u, 31);
  }
}

__global__ void k_flag_count(const uint8_t* __restrict__ keep, int64_t m,
                             int64_t* __restrict__ tile_cnt) {
  __shared__ int wsum[kThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kSampTile + (int64_t)threadIdx.x * kSampItems;
  int c = 0;
#pragma unroll
  for (int j = 0; j < kSampItems; ++j)
    if (base + j < m) c += keep[base + j];
  c = __reduce_add_sync(kFull, c);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t s = 0;
    for (int w = 0; w < kThreads / 32; ++w) s += wsum[w];
    tile_cnt[blockIdx.x] = s;
  }
}

// Kept edges in increasing canonical index: pairs (u, v), u < v, and w_e.
__global__ void k_flag_write(const int32_t* __restrict__ col, const int64_t* __restrict__ up_ptr,
                             const int64_t* __restrict__ edge_off, const int32_t* __restrict__ vw,
                             int64_t n, int64_t m, const uint8_t* __restrict__ keep,
                             const int64_t* __restrict__ tile_off, int32_t* __restrict__ pairs,
                             int32_t* __restrict__ pw) {
  __shared__ int wsum[kThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kSampTile + (int64_t)threadIdx.x * kSampItems;
  unsigned bits = 0;
#pragma unroll
  for (int j = 0; j < kSampItems; ++j)
    if (base + j < m && keep[base + j]) bits |= 1u << j;
  const int c = __popc(bits);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = c;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(kFull, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  int before = 0;
  for (int w = 0; w < warp; ++w) before += wsum[w];
  int64_t pos = tile_off[blockIdx.x] + before + x - c;
  while (bits) {
    const int j = __ffs(bits) - 1;
    bits &= bits - 1;
    const int64_t i = base + j;
    int64_t lo = 0, len = n;  // row owning canonical edge i
    while (len > 1) {
      const int64_t half = len >> 1;
      lo = (edge_off[lo + half] <= i) ? lo + half : lo;
      len -= half;
    }
    const int32_t v = col[up_ptr[lo] + (i - edge_off[lo])];
    pairs[2 * pos] = (int32_t)lo;
    pairs[2 * pos + 1] = v;
    if (pw != nullptr) pw[pos] = edge_weight(vw, (int32_t)lo, v);
    ++pos;
  }
}

// ------------------------------------------------------------------ fixed size

// Histogram of one radix digit of the 53-bit sampler keys, over the edges
// whose key agrees with `prefix` on the bits above `shift + bits`.
constexpr int kSelBins = 2048;

__global__ void k_key_hist(int64_t m, uint64_t seed, uint64_t prefix, int above, int shift,
                           int bits, unsigned long long* __restrict__ hist) {
  __shared__ unsigned int h[kSelBins];
  for (int b = threadIdx.x; b < kSelBins; b += blockDim.x) h[b] = 0;
  __syncthreads();
  const uint64_t dmask = ((uint64_t)1 << bits) - 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = splitmix(seed ^ splitmix((uint64_t)i)) >> 11;
    if (above >= 53 || (key >> above) == prefix) atomicAdd(h + ((key >> shift) & dmask), 1u);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < (1 << bits); b += blockDim.x)
    if (h[b]) atomicAdd(hist + b, (unsigned long long)h[b]);
}

// (key, i) of the edges whose key agrees with lo.prefix above bit lo.above, and
// with hi.prefix above hi.above (the buckets that hold two order statistics),
// into out_lo and out_hi.
struct KeyPrefix {
  uint64_t prefix;
  int32_t above;  // 53: no bucket
};
__global__ void k_key_collect(int64_t m, uint64_t seed, KeyPrefix lo, KeyPrefix hi,
                              ulonglong2* __restrict__ out_lo, ulonglong2* __restrict__ out_hi,
                              unsigned long long* __restrict__ cnt) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = splitmix(seed ^ splitmix((uint64_t)i)) >> 11;
    if (lo.above < 53 && (key >> lo.above) == lo.prefix)
      out_lo[atomicAdd(cnt, 1ull)] = make_ulonglong2(key, (unsigned long long)i);
    if (hi.above < 53 && (key >> hi.above) == hi.prefix)
      out_hi[atomicAdd(cnt + 1, 1ull)] = make_ulonglong2(key, (unsigned long long)i);
  }
}

// keep[i]: (key, i) among the k_hi smallest and not among the k_lo
// smallest; each set is {key < T} plus {key == T, i <= i_cut}.
__global__ void k_fixed_flags(int64_t m, uint64_t seed, uint64_t T_lo, int64_t cut_lo,
                              uint64_t T_hi, int64_t cut_hi, uint8_t* __restrict__ keep) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t key = splitmix(seed ^ splitmix((uint64_t)i)) >> 11;
    const bool in_hi = key < T_hi || (key == T_hi && i <= cut_hi);
    const bool in_lo = key < T_lo || (key == T_lo && i <= cut_lo);
    keep[i] = (in_hi && !in_lo) ? 1 : 0;
  }
}

// ------------------------------------------------------------------ HT fold

// Largest and smallest edge weight of a sampled list ([0] max, [1] min).
__global__ void k_pair_weight_range(const int2* __restrict__ uv, int64_t K,
                                    const int32_t* __restrict__ vw,
                                    unsigned long long* __restrict__ out) {
  unsigned long long mx = 0, mn = ~0ull;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 pr = uv[e];
    const int32_t w = edge_weight(vw, pr.x, pr.y);
    const unsigned long long ww = w < 0 ? 0ull : (unsigned long long)w;
    mx = ww > mx ? ww : mx;
    mn = ww < mn ? ww : mn;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(kFull, mx, o);
    const unsigned long long b = __shfl_xor_sync(kFull, mn, o);
    mx = a > mx ? a : mx;
    mn = b < mn ? b : mn;
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, mx);
    atomicMin(out + 1, mn);
  }
}

// Per-edge numerators (order 3, 4, 7, 8, 9, 10, 11, 12) and their squares
// added to the edge's weight class as four 32-bit limbs per 128-bit value
// (exact for fewer than 2^32 edges).
__global__ void __launch_bounds__(kThreads)
    k_fold_class(const int64_t* __restrict__ row_ptr, const int2* __restrict__ uv, int64_t K,
                 const unsigned long long* __restrict__ t, const unsigned long long* __restrict__ k2,
                 const unsigned long long* __restrict__ q, const int32_t* __restrict__ vw,
                 unsigned long long* __restrict__ limbs) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int2 pr = uv[e];
    const i128 du = __ldg(row_ptr + pr.x + 1) - __ldg(row_ptr + pr.x);
    const i128 dv = __ldg(row_ptr + pr.y + 1) - __ldg(row_ptr + pr.y);
    const i128 tt = (i128)t[e];
    const i128 kk = k2 != nullptr ? (i128)k2[e] : 0;
    const i128 qq = q != nullptr ? (i128)(long long)q[e] : 0;
    const i128 a = du - 1 - tt, b = dv - 1 - tt;
    const i128 n8 = tt * (tt - 1) / 2 - kk;
    i128 N[8];
    N[0] = tt;
    N[1] = a + b;
    N[2] = kk;
    N[3] = n8;
    N[4] = tt * (a + b) - 4 * n8;
    N[5] = qq;
    N[6] = 2 * (a * (a - 1) / 2 + b * (b - 1) / 2) - tt * (a + b) + 4 * n8;
    N[7] = a * b - qq;
    unsigned long long* dst = limbs + (int64_t)edge_weight(vw, pr.x, pr.y) * 64;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const u128 s = (u128)N[i];
      const u128 mg = (u128)(N[i] < 0 ? -N[i] : N[i]);
      const u128 sq = mg * mg;
#pragma unroll
      for (int l = 0; l < 4; ++l) {
        const unsigned long long a1 = (unsigned long long)((s >> (32 * l)) & 0xffffffffu);
        const unsigned long long a2 = (unsigned long long)((sq >> (32 * l)) & 0xffffffffu);
        if (a1) atomicAdd(dst + i * 4 + l, a1);
        if (a2) atomicAdd(dst + (8 + i) * 4 + l, a2);
      }
    }
  }
}

}  // namespace
}  // namespace gs

using namespace gs;

namespace {

u128 limb_value(const unsigned long long* l) {
  u128 s = 0;
  for (int j = 0; j < 4; ++j) s += (u128)l[j] << (32 * j);
  return s;
}

double i128_to_double(u128 v) {  // two's complement
  return (v >> 127) ? -(double)(u128)(-(i128)v) : (double)v;
}

}  // namespace

extern "C" gs_status gs_workspace_set_wait_limit(gs_workspace* ws, int64_t looks) {
  if (ws == nullptr || looks < 0) {
    set_error("gs_workspace_set_wait_limit: null workspace or negative limit");
    return GS_EINVAL;
  }
  ws->has_wait_limit = 1;
  ws->wait_limit = looks;
  return GS_OK;
}

extern "C" gs_status gs_core_numbers(const gs_graph* gr, gs_workspace* ws, int32_t* d_core,
                                     int32_t* h_max_core, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || (d_core == nullptr && gr->dev.n > 0)) {
    set_error("gs_core_numbers: invalid arguments");
    return GS_EINVAL;
  }
  const int64_t n = gr->dev.n;
  if (h_max_core) *h_max_core = 0;
  if (n == 0) return GS_OK;
  // removal entries of one list: a part per vertex and one per kPeelPart
  // neighbours beyond
  const int64_t entries = n + gr->dev.nnz / kPeelPart;
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 0,
                    Carve::bytes_for<int32_t>(n) * 3 + Carve::bytes_for<int2>(entries) * 2 +
                        Carve::bytes_for<PeelState>(1),
                    stream, &base));
  Carve c{(char*)base, 0};
  int32_t* deg = c.take<int32_t>(n);
  int32_t* rem0 = c.take<int32_t>(n);
  int32_t* rem1 = c.take<int32_t>(n);
  int2* list0 = c.take<int2>(entries);
  int2* list1 = c.take<int2>(entries);
  PeelState* st = c.take<PeelState>(1);
  PeelState init;
  memset(&init, 0, sizeof(init));
  for (PeelPhase& p : init.phase) p.least = ~0ull;
  GS_CUDA(cudaMemcpyAsync(st, &init, sizeof(init), cudaMemcpyHostToDevice, stream));
  // every block resident at once (the blocks wait on one another): at most
  // one per SM (two make the barriers dearer: 9.1 against 8.8 ms for core
  // numbers, a weighted sample and its estimates on the 100k-vertex power-law
  // graph, before removals had all loads in flight), fewer for a small graph
  int per_sm = 0;
  GS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_core_peel, kPeelThreads, 0));
  const int64_t most = (int64_t)sm_count() * std::min(per_sm, 1);
  const int64_t want = (n + gr->dev.nnz / 16 + kPeelThreads - 1) / kPeelThreads;
  const int blocks = (int)std::max<int64_t>(1, std::min(most, want));
  const int64_t* row_ptr = gr->dev.row_ptr;
  const int32_t* col = gr->dev.col;
  int64_t n_arg = n;
  int64_t limit = ws->has_wait_limit ? ws->wait_limit : kPeelSpins;
  void* args[] = {&row_ptr, &col,   &n_arg, &deg, &d_core, &rem0,
                  &rem1,    &list0, &list1, &st,  &limit};
  GS_CUDA(cudaLaunchCooperativeKernel((const void*)k_core_peel, dim3(blocks), dim3(kPeelThreads),
                                      args, 0, stream));
  ws->launches_total += 1;
  PeelState done;
  GS_CUDA(cudaMemcpyAsync(&done, st, sizeof(done), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  if (done.failed != 0) {
    set_error("gs_core_numbers: a grid-wide wait ran out");
    return GS_ETIMEOUT;
  }
  if (h_max_core) *h_max_core = done.max_core;
  return GS_OK;
}

extern "C" gs_status gs_sample_weighted(const gs_graph* gr, gs_workspace* ws,
                                        const int32_t* d_vertex_w, double fraction,
                                        uint64_t seed, int32_t* d_pairs, int32_t* d_pair_w,
                                        int64_t max_k, int64_t* k_out, double* scale_out,
                                        void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || d_vertex_w == nullptr || d_pairs == nullptr ||
      k_out == nullptr || max_k < 0 || !(fraction >= 0.0 && fraction <= 1.0)) {
    set_error("gs_sample_weighted: invalid arguments (fraction must lie in [0, 1])");
    return GS_EINVAL;
  }
  *k_out = 0;
  if (scale_out) *scale_out = 0.0;
  const int64_t n = gr->dev.n, m = gr->m;
  if (m == 0) return GS_OK;
  const int64_t tiles = (m + kSampTile - 1) / kSampTile;
  const size_t bytes = Carve::bytes_for<unsigned long long>(8) + Carve::bytes_for<uint8_t>(m) +
                       Carve::bytes_for<int64_t>(tiles + 1) * 2 +
                       Carve::bytes_for<int64_t>(scan_tmp_elems(tiles));
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 0, bytes, stream, &base));
  Carve c{(char*)base, 0};
  unsigned long long* acc = c.take<unsigned long long>(8);
  uint8_t* keep = c.take<uint8_t>(m);
  int64_t* cnt = c.take<int64_t>(tiles + 1);
  int64_t* off = c.take<int64_t>(tiles + 1);
  int64_t* tmp = c.take<int64_t>(scan_tmp_elems(tiles));
  GS_CUDA(cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 8, stream));
  k_weight_sum<<<grid_for(n * 32, kThreads, 8), kThreads, 0, stream>>>(
      gr->dev.row_ptr, gr->dev.col, gr->up_ptr, d_vertex_w, n, acc);
  unsigned long long h[2];
  GS_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  if (h[1] != 0 || h[0] == 0) {
    set_error("gs_sample_weighted: vertex weights must be >= 0 and some edge weight > 0");
    return GS_EINVAL;
  }
  const double scale = fraction * (double)m / (double)h[0];
  if (scale_out) *scale_out = scale;
  k_weighted_flags<<<grid_for(m, kThreads, 8), kThreads, 0, stream>>>(
      gr->dev.col, gr->up_ptr, gr->edge_off, d_vertex_w, n, m, scale, seed, keep);
  k_flag_count<<<(unsigned)tiles, kThreads, 0, stream>>>(keep, m, cnt);
  GS_TRY(exclusive_scan_i64(cnt, off, tiles, tmp, stream));
  int64_t kept = 0;
  GS_CUDA(cudaMemcpyAsync(&kept, off + tiles, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  *k_out = kept;
  ws->launches_total += 3 + scan_launches(tiles);
  if (kept > max_k) {
    set_error("gs_sample_weighted: %lld edges kept but the output holds %lld", (long long)kept,
              (long long)max_k);
    return GS_ECAPACITY;
  }
  if (kept > 0) {
    k_flag_write<<<(unsigned)tiles, kThreads, 0, stream>>>(gr->dev.col, gr->up_ptr, gr->edge_off,
                                                           d_vertex_w, n, m, keep, off, d_pairs,
                                                           d_pair_w);
    ws->launches_total += 1;
  }
  GS_CUDA(cudaGetLastError());
  GS_CUDA(cudaStreamSynchronize(stream));
  return GS_OK;
}

extern "C" gs_status gs_count_weighted(const gs_graph* gr, gs_workspace* ws,
                                       const int32_t* d_pairs, int64_t K,
                                       const int32_t* d_vertex_w, double scale, uint32_t mask,
                                       double z, gs_result* out, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || out == nullptr || d_vertex_w == nullptr || K < 0 ||
      (K > 0 && d_pairs == nullptr) || !(scale > 0.0) || !(z >= 0.0) || mask == 0 ||
      (mask & ~(uint32_t)GS_CONNECTED) != 0) {
    set_error("gs_count_weighted: invalid arguments (scale > 0, mask a non-empty subset of "
              "GS_CONNECTED)");
    return GS_EINVAL;
  }
  memset(out, 0, sizeof(*out));
  static const uint32_t bit[8] = {GS_G3, GS_G4, GS_G7, GS_G8, GS_G9, GS_G10, GS_G11, GS_G12};
  static const int D[8] = {3, 2, 6, 1, 2, 4, 6, 1};
  for (int i = 0; i < 8; ++i)
    if (mask & bit[i]) out->flags[i] = GS_F_COMPUTED;
  if (K == 0) return GS_OK;
  CountBufs b;
  const Tuning tu = ws->has_tuning ? ws->tuning : default_tuning();
  GS_TRY(count_run(gr, ws, d_pairs, K, mask, true, nullptr, nullptr, 0, tu, b, stream,
                   "gs_count_weighted"));
  // weight classes present
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 3, Carve::bytes_for<unsigned long long>(8), stream, &base));
  unsigned long long* range = (unsigned long long*)base;
  const unsigned long long init[2] = {0ull, ~0ull};
  GS_CUDA(cudaMemcpyAsync(range, init, sizeof(init), cudaMemcpyHostToDevice, stream));
  k_pair_weight_range<<<grid_for(K, kThreads, 4), kThreads, 0, stream>>>(b.uv, K, d_vertex_w,
                                                                          range);
  unsigned long long hr[2];
  GS_CUDA(cudaMemcpyAsync(hr, range, sizeof(hr), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  if (hr[1] == 0 || (int64_t)hr[0] >= kMaxClasses) {
    set_error("gs_count_weighted: every sampled edge needs a weight in [1, 2^22) (pi_e > 0)");
    return GS_EINVAL;
  }
  const int64_t classes = (int64_t)hr[0] + 1;
  GS_TRY(ws_reserve(ws, 3, Carve::bytes_for<unsigned long long>(classes * 64), stream, &base));
  unsigned long long* limbs = (unsigned long long*)base;
  GS_CUDA(cudaMemsetAsync(limbs, 0, sizeof(unsigned long long) * classes * 64, stream));
  const bool four = (mask & (GS_G7 | GS_G8 | GS_G9 | GS_G10 | GS_G11 | GS_G12)) != 0;
  k_fold_class<<<grid_for(K, kThreads, 4), kThreads, 0, stream>>>(
      gr->dev.row_ptr, b.uv, K, b.t, four ? b.k2 : nullptr, four ? b.q : nullptr, d_vertex_w,
      limbs);
  GS_CUDA(cudaGetLastError());
  ws->launches_total += 3;
  const int64_t lo = (int64_t)hr[1];
  // classes [lo, classes) back to the host
  unsigned long long* h = new unsigned long long[(size_t)(classes - lo) * 64];
  cudaError_t ce = cudaMemcpyAsync(h, limbs + lo * 64,
                                   sizeof(unsigned long long) * (size_t)(classes - lo) * 64,
                                   cudaMemcpyDeviceToHost, stream);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(stream);
  if (ce != cudaSuccess) {
    delete[] h;
    return cuda_fail(ce, "gs_count_weighted readback", __FILE__, __LINE__);
  }
  double X[8] = {0}, V[8] = {0};
  bool all_one = K == gr->m;
  for (int64_t c = lo; c < classes; ++c) {
    const unsigned long long* cl = h + (c - lo) * 64;
    bool any = false;
    for (int j = 0; j < 64 && !any; ++j) any = cl[j] != 0;
    if (!any) continue;
    double pi = scale * (double)c;
    if (pi > 1.0) pi = 1.0;
    if (pi < 1.0) all_one = false;
    for (int i = 0; i < 8; ++i) {
      const double s = i128_to_double(limb_value(cl + i * 4));
      const double s2 = (double)limb_value(cl + (8 + i) * 4);
      X[i] += s / pi;
      V[i] += (1.0 - pi) * s2 / (pi * pi);
    }
  }
  // exact integer totals when every edge was kept with pi = 1
  for (int i = 0; i < 8; ++i) {
    if (!(mask & bit[i])) continue;
    out->x[i] = X[i] / D[i];
    out->var[i] = V[i] / ((double)D[i] * D[i]);
    const double half = z * sqrt(out->var[i]);
    out->lb[i] = out->x[i] - half;
    out->ub[i] = out->x[i] + half;
    if (all_one) {
      u128 tot = 0;
      for (int64_t c = lo; c < classes; ++c) tot += limb_value(h + (c - lo) * 64 + i * 4);
      const i128 st = (i128)tot;
      if (st >= 0 && st % D[i] == 0 && st / D[i] <= (i128)UINT64_MAX) {
        out->exact[i] = (uint64_t)(st / D[i]);
        out->flags[i] |= GS_F_EXACT;
      }
    }
  }
  delete[] h;
  return GS_OK;
}

namespace gs {

// A bucket of keys with a common prefix that holds an order statistic: rank
// is its 0-based rank inside the bucket, size the bucket's keys.
struct RankBucket {
  KeyPrefix at;
  int64_t rank, size;
};

// Buckets of at most this many keys are read back and selected from on the
// host.
constexpr int64_t kBucketMost = 16384;

// The part of `b` whose next `bits` key bits hold its rank (h: their counts).
static gs_status narrow(RankBucket* b, const unsigned long long* h, int bits) {
  int64_t before = 0;
  int d = 0;
  for (; d < (1 << bits); ++d) {
    if (before + (int64_t)h[d] > b->rank) break;
    before += (int64_t)h[d];
  }
  if (d == (1 << bits)) {
    set_error("sampler key selection lost its rank");
    return GS_ECUDA;
  }
  b->rank -= before;
  b->at.prefix = (b->at.prefix << bits) | (uint64_t)d;
  b->at.above -= bits;
  b->size = (int64_t)h[d];
  return GS_OK;
}

// Boundaries of the k smallest keys for the cuts in c[0] and c[1] (k set; k =
// 0 and a cut that is already known are left alone). A histogram of the
// leading key bits, shared by both cuts, gives each one's bucket; buckets that
// are still large are split by further bits; the keys left are collected in
// one pass and selected from on the host. The digit-by-digit selection before
// took five passes and waits per cut (55 of the 223 launches of an adaptive
// estimate on R-MAT 18).
static gs_status rank_cuts(const gs_graph* gr, gs_workspace* ws, uint64_t seed,
                           unsigned long long* hist, RankCut* c[2], const bool known[2],
                           int64_t* launches, cudaStream_t stream) {
  const int64_t m = gr->m;
  constexpr int kBits = 11;
  std::vector<unsigned long long> h(kSelBins);
  auto histogram = [&](const KeyPrefix& p, int bits) -> gs_status {
    GS_CUDA(cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * kSelBins, stream));
    k_key_hist<<<grid_for(m, kThreads, 4), kThreads, 0, stream>>>(m, seed, p.prefix, p.above,
                                                                   p.above - bits, bits, hist);
    ++*launches;
    GS_CUDA(cudaMemcpyAsync(h.data(), hist, sizeof(unsigned long long) << bits,
                            cudaMemcpyDeviceToHost, stream));
    GS_CUDA(cudaStreamSynchronize(stream));
    return GS_OK;
  };
  RankBucket b[2];
  bool want[2];
  for (int j = 0; j < 2; ++j) {
    want[j] = !known[j] && c[j]->k > 0;
    if (!known[j] && c[j]->k <= 0) *c[j] = RankCut{0, 0, -1};
    b[j] = RankBucket{KeyPrefix{0, 53}, c[j]->k - 1, m};
  }
  if (!want[0] && !want[1]) return GS_OK;
  GS_TRY(histogram(KeyPrefix{0, 53}, kBits));
  for (int j = 0; j < 2; ++j)
    if (want[j]) GS_TRY(narrow(&b[j], h.data(), kBits));
  for (int j = 0; j < 2; ++j)
    while (want[j] && b[j].size > kBucketMost && b[j].at.above > 0) {
      const int bits = b[j].at.above < kBits ? b[j].at.above : kBits;
      GS_TRY(histogram(b[j].at, bits));
      GS_TRY(narrow(&b[j], h.data(), bits));
    }
  const int64_t n0 = want[0] ? b[0].size : 0, n1 = want[1] ? b[1].size : 0;
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 4,
                    Carve::bytes_for<unsigned long long>(2) + Carve::bytes_for<ulonglong2>(n0) +
                        Carve::bytes_for<ulonglong2>(n1),
                    stream, &base));
  Carve cv{(char*)base, 0};
  unsigned long long* cnt = cv.take<unsigned long long>(2);
  ulonglong2* d0 = cv.take<ulonglong2>(n0);
  ulonglong2* d1 = cv.take<ulonglong2>(n1);
  GS_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), stream));
  k_key_collect<<<grid_for(m, kThreads, 8), kThreads, 0, stream>>>(
      m, seed, want[0] ? b[0].at : KeyPrefix{0, 53}, want[1] ? b[1].at : KeyPrefix{0, 53}, d0, d1,
      cnt);
  ++*launches;
  std::vector<ulonglong2> keys((size_t)(n0 + n1));
  if (n0 > 0)
    GS_CUDA(cudaMemcpyAsync(keys.data(), d0, sizeof(ulonglong2) * (size_t)n0,
                            cudaMemcpyDeviceToHost, stream));
  if (n1 > 0)
    GS_CUDA(cudaMemcpyAsync(keys.data() + n0, d1, sizeof(ulonglong2) * (size_t)n1,
                            cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  for (int j = 0; j < 2; ++j) {
    if (!want[j]) continue;
    ulonglong2* first = keys.data() + (j == 0 ? 0 : n0);
    ulonglong2* nth = first + b[j].rank;
    std::nth_element(first, nth, first + b[j].size, [](const ulonglong2& x, const ulonglong2& y) {
      return x.x < y.x || (x.x == y.x && x.y < y.y);
    });
    c[j]->T = nth->x;
    c[j]->i_cut = (int64_t)nth->y;
  }
  return GS_OK;
}

// Edges ranked [k_lo, k_hi) by (key, i), in increasing canonical index,
// into d_pairs (device int32[2 (k_hi - k_lo)]) or, when d_pairs is NULL,
// into workspace slot 3 (*pairs_out).
gs_status sample_ranks(const gs_graph* gr, gs_workspace* ws, int64_t k_lo, int64_t k_hi,
                       uint64_t seed, int32_t* d_pairs, int32_t** pairs_out,
                       cudaStream_t stream, RankCut* cut) {
  const int64_t n = gr->dev.n, m = gr->m;
  if (pairs_out) *pairs_out = d_pairs;
  if (k_hi <= k_lo) return GS_OK;
  const int64_t tiles = (m + kSampTile - 1) / kSampTile;
  const size_t bytes = Carve::bytes_for<unsigned long long>(kSelBins) +
                       Carve::bytes_for<uint8_t>(m) +
                       Carve::bytes_for<int64_t>(tiles + 1) * 2 +
                       Carve::bytes_for<int64_t>(scan_tmp_elems(tiles));
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 2, bytes, stream, &base));
  Carve c{(char*)base, 0};
  unsigned long long* hist = c.take<unsigned long long>(kSelBins);
  uint8_t* keep = c.take<uint8_t>(m);
  int64_t* cnt = c.take<int64_t>(tiles + 1);
  int64_t* off = c.take<int64_t>(tiles + 1);
  int64_t* tmp = c.take<int64_t>(scan_tmp_elems(tiles));
  int64_t launches = 0;
  const bool known[2] = {cut != nullptr && k_lo > 0 && cut->k == k_lo, false};
  RankCut lo{k_lo, 0, -1}, hi{k_hi, 0, -1};
  if (known[0]) lo = *cut;
  RankCut* cuts[2] = {&lo, &hi};
  GS_TRY(rank_cuts(gr, ws, seed, hist, cuts, known, &launches, stream));
  if (cut != nullptr) *cut = hi;
  if (d_pairs == nullptr) {
    void* b3 = nullptr;
    GS_TRY(ws_reserve(ws, 3, Carve::bytes_for<int32_t>(2 * (k_hi - k_lo)), stream, &b3));
    d_pairs = (int32_t*)b3;
    if (pairs_out) *pairs_out = d_pairs;
  }
  k_fixed_flags<<<grid_for(m, kThreads, 8), kThreads, 0, stream>>>(m, seed, lo.T, lo.i_cut, hi.T,
                                                                    hi.i_cut, keep);
  k_flag_count<<<(unsigned)tiles, kThreads, 0, stream>>>(keep, m, cnt);
  GS_TRY(exclusive_scan_i64(cnt, off, tiles, tmp, stream));
  k_flag_write<<<(unsigned)tiles, kThreads, 0, stream>>>(gr->dev.col, gr->up_ptr, gr->edge_off,
                                                         nullptr, n, m, keep, off, d_pairs,
                                                         nullptr);
  launches += 3 + scan_launches(tiles);
  int64_t kept = 0;
  GS_CUDA(cudaMemcpyAsync(&kept, off + tiles, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  ws->launches_total += launches;
  if (kept != k_hi - k_lo) {
    set_error("sampler: selected %lld edges instead of %lld", (long long)kept,
              (long long)(k_hi - k_lo));
    return GS_ECUDA;
  }
  return GS_OK;
}

}  // namespace gs

extern "C" gs_status gs_sample_fixed(const gs_graph* gr, gs_workspace* ws, int64_t k,
                                     uint64_t seed, int32_t* d_pairs, void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || k < 0 || k > gr->m || (k > 0 && d_pairs == nullptr)) {
    set_error("gs_sample_fixed: invalid arguments (need 0 <= k <= m and an output)");
    return GS_EINVAL;
  }
  return sample_ranks(gr, ws, 0, k, seed, d_pairs, nullptr, stream);
}

extern "C" gs_status gs_sample_ranks(const gs_graph* gr, gs_workspace* ws, int64_t k_lo,
                                     int64_t k_hi, uint64_t seed, int32_t* d_pairs,
                                     void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || k_lo < 0 || k_hi < k_lo || k_hi > gr->m ||
      (k_hi > k_lo && d_pairs == nullptr)) {
    set_error("gs_sample_ranks: invalid arguments (need 0 <= k_lo <= k_hi <= m and an output)");
    return GS_EINVAL;
  }
  return sample_ranks(gr, ws, k_lo, k_hi, seed, d_pairs, nullptr, stream);
}
