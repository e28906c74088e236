// Edge-centric local counting over a sampled edge set J (Algorithms 2-4)
// and the exact fold of the per-edge numerators (Sec. 2.3).
//
// For an edge e = (u, v) with d_u <= d_v (ties: smaller id is u), let
// T = N(u) cap N(v), S_u = N(u) \ {v} \ T, S_v = N(v) \ {u} \ T. The paper's
// per-edge quantities are
//   t = |T|                                          (Algorithm 2)
//   k = adjacent pairs inside T                      (Algorithm 3)
//   q = pairs (w in S_u, r in S_v) with w ~ r        (Algorithm 4)
// For w in S_u the common neighbours of w and v are u, the members of T
// adjacent to w and the members of S_v adjacent to w, so with
// c(x, y) = |N(x) cap N(y)|:
//   q = sum_{w in S_u} (c(w, v) - 1) - sum_{r in T} (c(r, u) - 1) + 2k
// (sum_{w in S_u} |N(w) cap T| counted from the T side). Co-degrees of hub
// pairs, and of mid-degree x top-hub pairs, come from tables built at
// registration; the rest are computed by membership tests (see the item
// comment below).
//
// GPU structure (all work is flattened so that per-edge cost skew -- power
// law degrees -- does not serialise on one warp):
//   prep     one thread per pair: canonical orientation, edge check,
//            duplicate check, per-edge position count d_u (padded to 32
//            when 4-node work follows).
//   tri      each lane tests one x in N(u) for membership in N(v); ballots
//            give t and, for 4-node work (warps then take runs of chunks of
//            32 positions of one edge), a word of "x in T" flags per chunk.
//   compact  T lists written in order with their hub-matrix slots (by a warp,
//            a CTA or a lane per edge, see k_compact_T); edges with at least
//            kDenseMin matrix members in T whose dense-mode work (row groups
//            plus the other members' neighbour lists) is below their
//            sparse-mode tests are marked dense and get a T mask over matrix
//            slots.
//   cost     per chunk of 32 positions (items w = N(u)[i]): membership-test
//            count of each item (iterate the shorter list, test in the
//            longer); constant terms (the -1s, table co-degrees) added
//            directly; two ballots per chunk (items with tests, items a table
//            answered) for the 4-node pass; consecutive chunks with at most
//            32 items with tests in all form a pack.
//   quad     packs are cut into tasks of task_probes tests; warps take
//            runs of consecutive tasks from a counter; inside a task lanes
//            take consecutive tests (two per lane per iteration).
//   dense    in a dense edge segment A is counted by k_dense_pairs, in work
//            units of kDenseUnit T entries: pairs of dense-slot members by
//            matrix rows ANDed with the T mask, 128 bits at a time; for the
//            other members w, w's matrix neighbours (a bit of the mask, or,
//            past the dense slots, a search of T when above w) and w's
//            neighbours above w without a matrix slot (a search of T).
//   fold     per edge numerators N_i in 128-bit, block partial sums, one
//            final pass (or per-segment limb sums, k_fold_seg).
#include <string.h>

#include <algorithm>

#include "common.cuh"

namespace gs {

constexpr int kThreads = 256;
// k_chunk_cost: 6 CTAs per SM (at most 40 registers) hide more of its
// dependent loads than 4 do.
constexpr int kCostBlocksPerSm = 6;
constexpr int kQuadBlocksPerSm = 8;
constexpr unsigned kFull = 0xffffffffu;
// An edge whose T has at least this many hub-matrix members, and whose
// dense-mode work is the smaller, counts the pairs among them with
// word-parallel AND + popcount over hub-matrix rows.
constexpr int kDenseMin = 64;
constexpr unsigned long long kEmpty = ~0ull;
// Device counters of one count (CountBufs::stats): 0 triangle-pass tests,
// 1 4-node tests, 2 / 3 model bytes (3-node / 4-node part), 4 dense groups,
// 5 k_quad task counter, 6 dense edges, 7 k_dense_pairs unit counter,
// 8 k_chunk_cost chunk counter, 10 k_tri_chunks chunk counter, 9 tests of dense edges' members without a
// dense slot (k_dense_pairs).
constexpr int kStatSlots = 16;
// Chunks per run a k_chunk_cost warp takes from its counter, at most; also
// the most chunks a pack of k_quad spans (packs do not cross runs), at most 32.
constexpr int kCostGrab = 32;
static_assert(kCostGrab <= 32, "a pack's chunks are read by the lanes of a warp");
// The same for k_tri_chunks, whose chunks are cheap next to the search that
// begins a run (1M-vertex power-law graph exact: 38.2 / 34.6 / 32.3 / 33.3 ms
// at 16 / 32 / 128 / 512 chunks).
constexpr int kTriGrab = 128;
// Runs each warp should get to take from a counter: with fewer the work that
// is left over at the end is a large share of a warp's time, and a call with
// little work would leave most warps without a run (ER 2000/20000 exact:
// k_quad 396 us with runs of 32 tasks, which is 640 runs for 9728 warps).
constexpr int kRunsPerWarp = 8;
// Items per run when `total` items are shared by `warps` warps.
__device__ __forceinline__ int run_length(int64_t total, int64_t warps, int64_t most) {
  const int64_t r = total / (warps * kRunsPerWarp);
  return r < 1 ? 1 : (int)(r < most ? r : most);
}
// The same for chunks of positions, whose costs differ less than the search
// that begins a run costs: with few of them one run per warp, and no run of
// fewer than kRunsPerWarp chunks with more of them (58,000 to 467,000 chunks had
// runs of one to seven: triangle pass of 90,000 chunks 0.077 -> 0.040 ms, of
// 200,000 0.096 -> 0.058 on R-MAT 18, 0.105 -> 0.088 on the 1M-vertex power-law
// graph; cost pass 0.162 -> 0.128 and 0.220 -> 0.200 ms).
__device__ __forceinline__ int chunk_run_length(int64_t total, int64_t warps, int64_t most) {
  if (total <= warps * kRunsPerWarp) return (int)((total + warps - 1) / warps);
  return max(kRunsPerWarp, run_length(total, warps, most));
}
// Filter of a dense edge's T members without a matrix slot in k_dense_pairs:
// 2^15 bits, built when T has at most kTFilterMaxT entries.
constexpr int kTFilterWords = 1024;
constexpr int64_t kTFilterMaxT = 16384;
__device__ __forceinline__ uint32_t tfilter_hash(int32_t x) {
  return ((uint32_t)x * 2654435761u) >> 17;
}

// Membership tests per run of consecutive tasks a k_quad warp takes from
// the task counter (at least one task). Short runs keep the warps in a narrow
// window of the sample, whose lists and directories they share in L2; each
// run searches its place and sets up its packs anew. R-MAT 24 0.1%: 185 / 159
// / 144 / 138 / 143 ms at 512 / 1024 / 2048 / 4096 / 16384 tests; batch of
// 1024 graphs 60.6 / 58.8 / 57.9 / 57.6 / 59.6 ms.
constexpr int64_t kQuadGrabTests = 4096;
// Resident warps per SM of k_dense_pairs (at most 40 registers), in CTAs of
// 256 threads, or of 128 when there are many units: the five to seven barriers
// of a unit hold up the warps of a small CTA less, but a unit with long lists of
// other members is walked by fewer warps, so that only graphs whose adjacency
// entries have matrix slots for the most part take small CTAs. 4-node phase with
// 128 and with 256 threads, and the share of entries with slots: 1M-vertex
// power-law graph (0.54) 34,000 dense edges 1.90 and 1.82 ms, 68,000 3.21 and
// 3.29, 169,000 7.18 and 7.81, 1.7M 65.1 and 73.2; R-MAT 20 (0.69) 84,000 3.57
// and 3.82; R-MAT 22 (0.52) 34,000 8.12 and 7.78, 85,000 17.92 and 17.85, 169,000
// 32.8 and 34.1; R-MAT 24 (0.36) 32,000 65.4 and 60.3, 95,000 176 and 170,
// 317,000 549 and 542. The line lies at kManyDensePerCta dense edges per
// resident CTA of 256 (73,000 in all) and a share of 0.45.
constexpr int kDenseWarpsPerSm = 48;
constexpr int64_t kManyDensePerCta = 80;
constexpr double kSmallCtaShare = 0.45;
constexpr int kTriBlocksPerSm = 6;  // k_tri_chunks: at most 40 registers
// T entries per k_dense_pairs work unit (a heavy dense edge is split into
// several units so that small samples still fill the GPU).
constexpr int64_t kDenseUnit = 4 * kThreads;
// Matrix rows are at most this many 128-bit groups.
constexpr int kHubMatrixMaxGroups = (int)((kHubMatrixMax + 127) / 128);
// 32-bit words of a bitmap over those groups.
constexpr int kGroupWords = (kHubMatrixMaxGroups + 31) / 32;
// Cost of one 128-bit dense group against one membership test, in quarters
// (the dense-mode choice compares kGroupCost * groups with 4 * tests).
constexpr int kGroupCost = 4;

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}



__device__ __forceinline__ int64_t deg_of(const int64_t* __restrict__ row_ptr, int32_t v,
                                          int64_t* base) {
  int64_t s = __ldg(row_ptr + v), e = __ldg(row_ptr + v + 1);
  *base = s;
  return e - s;
}

// Last index e in [0, count) with off[e] <= p (off[0] = 0 <= p).
__device__ __forceinline__ int64_t last_le(const int64_t* __restrict__ off, int64_t count,
                                           int64_t p) {
  int64_t lo = 0, len = count;
  while (len > 1) {
    int64_t half = len >> 1;
    lo = (__ldg(off + lo + half) <= p) ? lo + half : lo;
    len -= half;
  }
  return lo;
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// ---------------------------------------------------------------- prep

__global__ void k_all_pairs(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                            const int64_t* __restrict__ up_ptr,
                            const int64_t* __restrict__ edge_off, int64_t n,
                            int32_t* __restrict__ pairs) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += warps) {
    int64_t s = up_ptr[u], e = row_ptr[u + 1], o = edge_off[u];
    for (int64_t p = s + lane; p < e; p += 32) {
      int64_t i = o + (p - s);
      pairs[2 * i] = (int32_t)u;
      pairs[2 * i + 1] = col[p];
    }
  }
}

__global__ void k_prep(DevGraph g, const int32_t* __restrict__ pairs, int64_t K, int pad,
                       unsigned long long* __restrict__ dup_table, int64_t dup_mask,
                       int2* __restrict__ uv, int64_t* __restrict__ len, DevError* err) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    int32_t x = pairs[2 * e], y = pairs[2 * e + 1];
    len[e] = 0;
    uv[e] = make_int2(0, 0);
    if (x < 0 || y < 0 || x >= g.n || y >= g.n || x == y) {
      raise_error(err, GS_EEDGE, e);
      continue;
    }
    int64_t bx, by;
    int64_t dx = deg_of(g.row_ptr, x, &bx), dy = deg_of(g.row_ptr, y, &by);
    bool x_small = dx < dy || (dx == dy && x < y);
    int32_t u = x_small ? x : y, v = x_small ? y : x;
    int64_t du = x_small ? dx : dy, bu = x_small ? bx : by;
    if (!sorted_contains(g.col + bu, du, v)) {
      raise_error(err, GS_EEDGE, e);
      continue;
    }
    if (dup_table != nullptr) {
      uint64_t key = ((uint64_t)(uint32_t)min(x, y) << 32) | (uint32_t)max(x, y);
      uint64_t h = mix64(key) & (uint64_t)dup_mask;
      for (int64_t probe = 0; probe <= dup_mask; ++probe) {
        unsigned long long prev = atomicCAS(dup_table + h, kEmpty, (unsigned long long)key);
        if (prev == kEmpty) break;
        if (prev == key) {
          raise_error(err, GS_EDUPSAMPLE, e);
          break;
        }
        h = (h + 1) & (uint64_t)dup_mask;
      }
    }
    uv[e] = make_int2(u, v);
    len[e] = pad ? ((du + 31) & ~(int64_t)31) : du;
  }
}

// ---------------------------------------------------------------- tri
// 3-node work alone: positions [0, P) of the concatenated N(u) lists are
// split into equal contiguous ranges of 32-position groups, one range per warp.
__global__ void __launch_bounds__(kThreads) k_tri(DevGraph g, const int2* __restrict__ uv,
                                                  const int64_t* __restrict__ off, int64_t K,
                                                  unsigned long long* __restrict__ t) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t P = __ldg(off + K);
  const int64_t groups = (P + 31) >> 5;
  const int64_t per = (groups + warps - 1) / warps;
  const int64_t g0 = warp * per, g1 = min(groups, g0 + per);
  if (g0 >= g1) return;
  int64_t e = last_le(off, K, g0 * 32);
  for (int64_t gi = g0; gi < g1; ++gi) {
    const int64_t p = gi * 32 + lane;
    int64_t le = e;
    while (le + 1 < K && __ldg(off + le + 1) <= p) ++le;
    bool hit = false;
    if (p < P) {
      int2 pr = uv[le];
      int64_t bu, bv;
      int64_t du = deg_of(g.row_ptr, pr.x, &bu), dv = deg_of(g.row_ptr, pr.y, &bv);
      int64_t i = p - __ldg(off + le);
      if (i < du) {
        int32_t x = __ldg(g.col + bu + i);
        const int32_t xs = g.col_hm != nullptr ? (int32_t)__ldg(g.col_hm + bu + i) : -2;
        hit = x != pr.y && adj_contains(g, pr.y, bv, dv, x, xs);
      }
    }
    const unsigned ball = __ballot_sync(kFull, hit);
    const unsigned grp = __match_any_sync(kFull, (unsigned long long)le);
    const int cnt = __popc(ball & grp);
    if (cnt && lane == __ffs(grp) - 1) atomicAdd(t + le, (unsigned long long)cnt);
    e = __shfl_sync(kFull, le, 31);
  }
}

// The triangle pass of the 4-node work (and of 3-node samples with long lists,
// see kLongLists; tbits is then NULL): positions padded to 32 per edge, so a
// chunk of 32 positions lies in one edge. Warps take runs of chunks from a
// counter; what an edge needs (N(u), and how "x in N(v)" is answered) is
// looked up when the edge changes, t is added once per edge and run, and the
// next chunk's elements are loaded before this chunk's answers are used.
// Looking all of it up for every position, as k_tri does for 3-node work alone: 1M-vertex power-law
// graph exact (5.6e9 positions): 47.2 -> 32.3 ms (with runs of 16 chunks 37.9,
// and 44.2 / 40.8 at 8 / 5 CTAs per SM instead of 6).
__global__ void __launch_bounds__(kThreads, kTriBlocksPerSm)
    k_tri_chunks(const __grid_constant__ DevGraph g, const int2* __restrict__ uv,
                 const int64_t* __restrict__ off, int64_t K, unsigned long long* __restrict__ t,
                 uint32_t* __restrict__ tbits, unsigned long long* __restrict__ counter) {
  const int lane = threadIdx.x & 31;
  const int64_t groups = __ldg(off + K) >> 5;  // padded: a multiple of 32
  const int grab =
      chunk_run_length(groups, (int64_t)gridDim.x * (kThreads / 32), (int64_t)kTriGrab);
  int64_t e = -1, first = 0, end = 0, bu = 0;
  int32_t du = 0, v = 0;
  EndSet sv{};
  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(counter, (unsigned long long)grab);
    const int64_t g0 = (int64_t)__shfl_sync(kFull, got, 0);
    if (g0 >= groups) break;
    const int64_t g1 = min(groups, g0 + grab);
    unsigned found = 0;  // of edge e in this run
    int32_t x = -1, xs = -1;
    bool loaded = false;
    for (int64_t gi = g0; gi < g1; ++gi) {
      const int64_t p0 = gi * 32;
      if (p0 < first || p0 >= end) {  // another edge: the next one, or a search
        if (found && lane == 0) atomicAdd(t + e, (unsigned long long)found);
        found = 0;
        e = p0 == end && e >= 0 ? e + 1 : last_le_warp(off, K, p0);
        first = __ldg(off + e);
        end = __ldg(off + e + 1);
        const int2 pr = uv[e];
        v = pr.y;
        du = (int32_t)deg_of(g.row_ptr, pr.x, &bu);
        int64_t bv;
        const int64_t dv = deg_of(g.row_ptr, v, &bv);
        sv = end_set(g, v, bv, dv);
        loaded = false;
      }
      const int64_t i = p0 - first + lane;
      if (!loaded) {
        x = i < du ? __ldg(g.col + bu + i) : -1;
        xs = sv.mrow != nullptr && i < du ? (int32_t)__ldg(g.col_hm + bu + i) : -1;
      }
      const int32_t y = x, ys = xs;
      loaded = gi + 1 < g1 && p0 + 32 < end;
      if (loaded) {
        x = i + 32 < du ? __ldg(g.col + bu + i + 32) : -1;
        xs = sv.mrow != nullptr && i + 32 < du ? (int32_t)__ldg(g.col_hm + bu + i + 32) : -1;
      }
      const unsigned ball = __ballot_sync(kFull, y >= 0 && y != v && set_has(sv, y, ys));
      if (tbits != nullptr && lane == 0) tbits[gi] = ball;
      found += __popc(ball);
    }
    if (found && lane == 0) atomicAdd(t + e, (unsigned long long)found);
  }
}

// 3-node work alone takes k_tri_chunks, on offsets padded by k_pad_lengths,
// from this many positions per edge and in all on; below, the padding or the
// look-ups per edge cost more than they save. R-MAT 22 5% (3.2M edges, 500
// positions each) 21.8 -> 15.5 ms, 1M-vertex power-law graph 5% (1.0M, 280) 3.0
// -> 2.2 ms; a uniform graph of mean degree 20 30% (1.2M, 17) 0.43 -> 0.54 ms
// and R-MAT 18 2% (30,000 edges) 0.15 -> 0.20 ms stay with k_tri.
constexpr int64_t kLongLists = 96;
constexpr int64_t kManyPositions = (int64_t)1 << 23;

__global__ void k_pad_lengths(const int64_t* __restrict__ off, int64_t K,
                              int64_t* __restrict__ len) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x)
    len[e] = (off[e + 1] - off[e] + 31) & ~(int64_t)31;
}

// Host launcher of the 3-node triangle pass for count_static.cu.
void launch_tri_unpadded(const DevGraph& g, const int2* uv, const int64_t* off, int64_t K,
                         unsigned long long* t, int blocks, cudaStream_t stream) {
  k_tri<<<blocks, kThreads, 0, stream>>>(g, uv, off, K, t);
}

// ---------------------------------------------------------------- compact T

constexpr int kCompactBlocksPerSm = 5;
// Lists of more than this many positions are compacted by a whole CTA: with
// few edges the longest list is the pass's tail; with many, warps are never
// short of edges and the CTA's barriers only cost. Compact phase at 1024 /
// 2048 / 4096 / no limit: adaptive estimation on R-MAT 18 (61 to 2,000 edges a
// pass) 2.46 / 2.57 / 2.59 / 2.90 ms the whole call; R-MAT 22 19,000 edges 0.34 /
// 0.32 / 0.34 / 1.50 ms, 64,000 0.69 / 0.66 / 0.64 / 2.6, 193,000 1.56 / 1.48 /
// 1.25 / 2.9, 1.9M 12.3 / 11.4 / 8.9 / 11.2; 1M-vertex power-law graph 100,000
// edges 0.54 / 0.46 / 0.52 / 1.81, 200,000 0.88 / 0.71 / 0.72 / 2.26, 1.0M 3.5 /
// 2.8 / 2.4 / 3.8, 2.0M 6.6 / 5.1 / 4.7 / 6.0, 5M 16.1 / 12.2 / 10.7 / 11.2,
// exact (20M) 65 / 49 / 42 / 35. Without a limit short lists go to single lanes
// (ER of mean degree 4, 4M edges 1.5 -> 0.13), so that begins at 2^21 already.
inline int64_t compact_long(int64_t K) {
  return K < (1 << 15) ? 1024 : K < (1 << 17) ? 2048 : K < (1 << 21) ? 4096 : INT64_MAX;
}

// What k_compact_T shares of the edges in work: one per warp, the first one's
// by the CTA.
struct CompactShared {
  uint32_t gbits[kThreads / 32][kGroupWords];  // member groups of an edge
  int32_t warp_n[kThreads / 32];
  long long part[kThreads / 32][4];
};

// T list of edge e by kWarps warps (1: the calling warp; else the CTA): T in
// order with its matrix slots, tpre per chunk, tdeg[e] = sum of the degrees of
// T's members (which only feeds the cost model statistics), and the choice of
// dense mode.
template <int kWarps>
__device__ __forceinline__ void compact_edge(const DevGraph& g, int64_t e, int32_t u,
                                             const int64_t* __restrict__ off,
                                             const int64_t* __restrict__ toff,
                                             const uint32_t* __restrict__ tbits, int32_t* T,
                                             int32_t* __restrict__ tpre, int16_t* T_hm,
                                             int64_t* __restrict__ tdeg,
                                             int32_t* __restrict__ mask_idx,
                                             unsigned long long* __restrict__ dense_counter,
                                             CompactShared& sh) {
  constexpr bool kCta = kWarps > 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int part = kCta ? wid : 0;
  auto sync = [&]() {
    if (kCta) __syncthreads();
    else __syncwarp();
  };
  int64_t bu;
  const int64_t du = deg_of(g.row_ptr, u, &bu);
  const int64_t words = (du + 31) >> 5, w0 = off[e] >> 5, t0 = toff[e];
  const int64_t D = g.hm_dense_words * 32;
  int64_t pos = t0;
  long long sum[4] = {0, 0, 0, 0};  // degrees, dense-slot members; then the choice's sums
  // 32 words of T bits per warp at a time, one per lane; then the words that
  // have members, four at a time so that their loads are in flight together
  for (int64_t wb0 = 0; wb0 < words; wb0 += 32 * kWarps) {
    const int64_t wb = wb0 + 32 * part;
    const uint32_t word = wb + lane < words ? __ldg(tbits + w0 + wb + lane) : 0u;
    int before = __popc(word);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(kFull, before, d);
      if (lane >= d) before += y;
    }
    int all = __shfl_sync(kFull, before, 31);
    before -= __popc(word);
    if (kCta) {
      if (lane == 0) sh.warp_n[wid] = all;
      __syncthreads();
      all = 0;
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        before += k < wid ? sh.warp_n[k] : 0;
        all += sh.warp_n[k];
      }
      __syncthreads();  // warp_n is rewritten by the next round
    }
    if (wb + lane < words) tpre[w0 + wb + lane] = (int32_t)(pos - t0) + before;
    const int64_t c0 = bu + wb * 32 + lane;
    for (unsigned nz = __ballot_sync(kFull, word != 0u); nz;) {
      int32_t x[4];
      int at[4];
      int16_t xs[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int k = nz ? __ffs(nz) - 1 : 0;
        const uint32_t wd = nz ? __shfl_sync(kFull, word, k) : 0u;
        const int bk = __shfl_sync(kFull, before, k);
        nz &= nz - 1;
        x[h] = -1;
        xs[h] = -1;
        at[h] = bk + __popc(wd & ((1u << lane) - 1u));
        if ((wd >> lane) & 1u) {
          x[h] = __ldg(g.col + c0 + k * 32);
          if (T_hm != nullptr) xs[h] = __ldg(g.col_hm + c0 + k * 32);
        }
      }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (x[h] < 0) continue;
        T[pos + at[h]] = x[h];
        if (T_hm != nullptr) {
          T_hm[pos + at[h]] = xs[h];
          sum[1] += xs[h] >= 0 && xs[h] < D;
        }
        sum[0] += __ldg(g.row_ptr + x[h] + 1) - __ldg(g.row_ptr + x[h]);
      }
    }
    pos += all;
  }
  // sums (of values >= 0) over the warp, or the CTA
  auto total = [&](int n) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n)
        sum[i] = __any_sync(kFull, sum[i] >= (1 << 26))
                     ? warp_sum<long long>(sum[i])
                     : (long long)__reduce_add_sync(kFull, (unsigned)sum[i]);
    if (kCta) {
      __syncthreads();
      if (lane == 0)
        for (int i = 0; i < n; ++i) sh.part[wid][i] = sum[i];
      __syncthreads();
      for (int i = 0; i < n; ++i) {
        sum[i] = 0;
        for (int k = 0; k < kWarps; ++k) sum[i] += sh.part[k][i];
      }
    }
  };
  total(2);
  const long long dsum = sum[0];
  bool dense_mode = false;
  if (T_hm != nullptr && sum[1] >= kDenseMin) {
    // segment-A work of this edge in either mode: sparse = tests over the
    // shorter of N(w) above w / T above w (estimated); dense = for each
    // dense-slot member, the 128-bit groups of the T mask that hold a
    // member and lie at or below its own (what k_dense_pairs reads), plus
    // the adjacency of the other members
    const int64_t te = pos - t0;
    uint32_t* gb = sh.gbits[kCta ? 0 : wid];
    const int first = kCta ? (int)threadIdx.x : lane;
    constexpr int kStep = 32 * kWarps;
    for (int w = first; w < kGroupWords; w += kStep) gb[w] = 0u;
    sync();  // also: the edge's T entries are visible to all its threads
    for (int64_t j = first; j < te; j += kStep) {
      const int xs = T_hm[t0 + j];
      if (xs >= 0 && xs < D) atomicOr(gb + (xs >> 12), 1u << ((xs >> 7) & 31));
    }
    sync();
    int gpre = lane < kGroupWords ? __popc(gb[lane]) : 0;  // groups in words <= lane
#pragma unroll
    for (int d = 1; d < kGroupWords; d <<= 1) {
      const int y = __shfl_up_sync(kFull, gpre, d);
      if (lane >= d) gpre += y;
    }
    sum[0] = sum[1] = sum[2] = 0;  // sparse, dense, groups
    for (int64_t j0 = 32 * part; j0 < te; j0 += kStep) {
      const int64_t j = j0 + lane;
      const int xs = j < te ? (int)T_hm[t0 + j] : -1;
      const int gw = __shfl_sync(kFull, gpre, xs >= 4096 ? (xs >> 12) - 1 : 0);
      if (j >= te) continue;
      const int32_t x = T[t0 + j];
      const int64_t dx = __ldg(g.row_ptr + x + 1) - __ldg(g.row_ptr + x);
      sum[0] += min(dx / 2, te - j - 1);  // about half of N(x) lies above x
      if (xs >= 0 && xs < D) {
        const int g0 = xs >> 7;
        sum[2] += (xs >= 4096 ? gw : 0) + __popc(gb[g0 >> 5] & (kFull >> (31 - (g0 & 31))));
      } else {  // k_dense_pairs walks its matrix and non-matrix-above lists
        sum[1] += g.mn_ptr != nullptr ? (__ldg(g.mn_ptr + x + 1) - __ldg(g.mn_ptr + x)) +
                                            (__ldg(g.nm_ptr + x + 1) - __ldg(g.nm_ptr + x))
                                      : dx;
      }
    }
    total(3);
    dense_mode = kGroupCost * sum[2] + 4 * sum[1] < 4 * sum[0];
  }
  if ((kCta ? (int)threadIdx.x : lane) == 0) {
    tdeg[e] = dsum;
    if (mask_idx != nullptr)
      mask_idx[e] = dense_mode ? (int32_t)atomicAdd(dense_counter, 1ull) : -1;
  }
  if (kCta) __syncthreads();  // sh is reused for the next edge
}

static_assert(kDenseMin > 32, "an edge of at most 32 positions is never dense");

// T lists of all edges: a warp per edge, then a CTA per edge with a long list
// (a list of 35,000 positions kept one warp busy for most of a small sample's
// pass: adaptive estimation on R-MAT 18, 149 us a pass before).
template <bool kLong>
__global__ void __launch_bounds__(kThreads, kCompactBlocksPerSm)
    k_compact_T(const __grid_constant__ DevGraph g, const int2* __restrict__ uv,
                const int64_t* __restrict__ off, const int64_t* __restrict__ toff, int64_t K,
                const uint32_t* __restrict__ tbits, int32_t* T, int32_t* __restrict__ tpre,
                int16_t* T_hm, int64_t* __restrict__ tdeg, int32_t* __restrict__ mask_idx,
                unsigned long long* __restrict__ dense_counter, int64_t long_list) {
  __shared__ CompactShared sh;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  if (!kLong) {
    // 32 edges per warp: a lane does an edge of at most 32 positions by itself
    // (it cannot be dense), the warp does the others one by one (a warp per
    // such edge left 31 lanes idle: batch of 1024 graphs 58 -> 50 ms)
    const int lane = threadIdx.x & 31;
    for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; b < K;
         b += warps * 32) {
      const int64_t e = b + lane;
      int32_t u = 0;
      int64_t bu = 0, du = 0;
      if (e < K) {
        u = uv[e].x;
        du = deg_of(g.row_ptr, u, &bu);
      }
      if (e < K && du <= 32) {
        const int64_t w = off[e] >> 5;
        uint32_t word = __ldg(tbits + w);
        int64_t at = toff[e], dsum = 0;
        tpre[w] = 0;
        for (; word; word &= word - 1, ++at) {
          const int64_t p = bu + __ffs(word) - 1;
          const int32_t x = __ldg(g.col + p);
          T[at] = x;
          if (T_hm != nullptr) T_hm[at] = __ldg(g.col_hm + p);
          dsum += __ldg(g.row_ptr + x + 1) - __ldg(g.row_ptr + x);
        }
        tdeg[e] = dsum;
        if (mask_idx != nullptr) mask_idx[e] = -1;
      }
      for (unsigned m = __ballot_sync(kFull, du > 32); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        compact_edge<1>(g, b + src, __shfl_sync(kFull, u, src), off, toff, tbits, T, tpre, T_hm,
                        tdeg, mask_idx, dense_counter, sh);
      }
    }
    return;
  }
  for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < K; e += warps) {
    const int32_t u = uv[e].x;
    if (__ldg(g.row_ptr + u + 1) - __ldg(g.row_ptr + u) <= long_list)
      compact_edge<1>(g, e, u, off, toff, tbits, T, tpre, T_hm, tdeg, mask_idx, dense_counter,
                      sh);
  }
  __syncthreads();
  // the CTA looks for long lists among edges that lie gridDim apart: in a sample
  // in edge order the edges of hubs with neighbouring ids follow one another
  // (R-MAT 20 1% with ids by degree: 0.80 ms by a warp per edge, 5.1 by the CTA
  // that had a hub's edges, 0.45 so)
  const int64_t step = gridDim.x;
  for (int64_t b = blockIdx.x; b < K; b += step * kThreads) {
    __shared__ uint32_t todo[kThreads / 32];
    const int64_t e = b + step * threadIdx.x;
    bool is_long = false;
    if (e < K) {
      const int32_t u = uv[e].x;
      is_long = __ldg(g.row_ptr + u + 1) - __ldg(g.row_ptr + u) > long_list;
    }
    const unsigned bal = __ballot_sync(kFull, is_long);
    if ((threadIdx.x & 31) == 0) todo[threadIdx.x >> 5] = bal;
    __syncthreads();
    for (int w = 0; w < kThreads / 32; ++w)
      for (unsigned m = todo[w]; m; m &= m - 1) {
        const int64_t el = b + step * (w * 32 + __ffs(m) - 1);
        compact_edge<kThreads / 32>(g, el, uv[el].x, off, toff, tbits, T, tpre, T_hm, tdeg,
                                    mask_idx, dense_counter, sh);
      }
    __syncthreads();  // todo is rewritten
  }
}

// Masks of T's hub-matrix members for dense edges: bit s of the edge's
// mask is set iff the member with matrix slot s is in T. One warp per edge.
__global__ void k_build_tmask(const int64_t* __restrict__ toff, const unsigned long long* __restrict__ t,
                              const int16_t* __restrict__ T_hm, const int32_t* __restrict__ mask_idx,
                              int64_t K, int64_t words, uint32_t* __restrict__ tmask,
                              int64_t* __restrict__ dense_e, int64_t* __restrict__ units) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < K; e += warps) {
    const int32_t idx = mask_idx[e];
    if (idx < 0) continue;
    if (lane == 0) {
      dense_e[idx] = e;
      units[idx] = ((int64_t)t[e] + kDenseUnit - 1) / kDenseUnit;
    }
    uint32_t* m = tmask + (int64_t)idx * words;
    for (int64_t w = lane; w < words; w += 32) m[w] = 0u;
    __syncwarp();
    const int64_t b = toff[e], len = (int64_t)t[e];
    for (int64_t i = lane; i < len; i += 32) {
      const int32_t s = T_hm[b + i];
      if (s >= 0 && s < words * 32) atomicOr(m + (s >> 5), 1u << (s & 31));
    }
  }
}

// Dense edge of every k_dense_pairs work unit: unit_idx[u] = mask index.
// One warp per dense edge.
__global__ void k_unit_fill(const int64_t* __restrict__ unit_off, int64_t ndense,
                            int32_t* __restrict__ unit_idx) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t idx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; idx < ndense;
       idx += warps)
    for (int64_t u = unit_off[idx] + lane; u < unit_off[idx + 1]; u += 32)
      unit_idx[u] = (int32_t)idx;
}

// Pairs of dense-slot members of T in the dense edges, and the pairs of T's
// other members, per work unit of kDenseUnit T entries (unit_off: exclusive
// scan of the units per dense edge, unit_idx: the dense edge of each unit); a
// CTA takes one unit at a time from a counter.
//   dense-slot pairs: the member of rank r in slot order (slot s) contributes
//   popcount(its matrix row AND the edge's T mask) over the bits below s, so
//   every adjacent pair of members counts once (k += 1, q += 2). Slots are in
//   decreasing degree, so T's members crowd in the low slots and the mask's
//   non-zero 128-bit groups at or below a member's own are few. A unit takes
//   the members of its kDenseUnit ranks, listed in slot order in shared
//   memory; eight lanes walk one member's groups (128 coalesced bytes of the
//   L2-resident matrix at a time), so a warp has four members of nearly equal
//   length in flight, eight with the second set.
//   other members (w without a dense slot among the unit's T entries): w's
//   matrix neighbours (a bit of the mask, or, past the dense slots, a search
//   of T when above w) and w's neighbours above w without a matrix slot (a
//   search of T behind a hashed filter).
template <int kDenseThreads>
__global__ void __launch_bounds__(kDenseThreads, kDenseWarpsPerSm * 32 / kDenseThreads)
    k_dense_pairs(const __grid_constant__ DevGraph g, const int64_t* __restrict__ toff,
                  const unsigned long long* __restrict__ t, const int32_t* __restrict__ T,
                  const int16_t* __restrict__ T_hm, const uint32_t* __restrict__ tmask,
                  const int64_t* __restrict__ dense_e, const int64_t* __restrict__ unit_off,
                  const int32_t* __restrict__ unit_idx, int64_t ndense, int need_q,
                  unsigned long long* __restrict__ k_out, unsigned long long* __restrict__ q,
                  unsigned long long* __restrict__ counter,
                  unsigned long long* __restrict__ tests,
                  unsigned long long* __restrict__ rest_tests) {
  constexpr int kWarps = kDenseThreads / 32;
  // the edge's T mask compacted to its non-zero 128-bit groups: smask[c] is
  // group sgrp[c], with sbase[c] members in the groups before it
  __shared__ uint4 smask[kHubMatrixMaxGroups];
  __shared__ uint16_t sgrp[kHubMatrixMaxGroups];
  __shared__ uint16_t sbase[kHubMatrixMaxGroups];
  __shared__ int wcnt[kWarps], wlen[kWarps];
  // the unit's dense-slot members in slot order: slot and compact group
  __shared__ uint16_t mslot[kDenseUnit];
  __shared__ uint8_t mgrp[kDenseUnit];
  // members without a dense slot among a warp's 32 T entries: vertex, list
  // offsets, matrix-neighbour count, start in the concatenation of the lists
  __shared__ int64_t ra[kDenseThreads], rb[kDenseThreads];
  __shared__ int32_t rw[kDenseThreads], rna[kDenseThreads], rst[kDenseThreads];
  // hashed filter of T's members without a matrix slot (what the
  // non-matrix lists search for): a clear bit means "not in T"
  __shared__ uint32_t tfilt[kTFilterWords];
  __shared__ unsigned long long part[kWarps][3];
  __shared__ int64_t cur;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t dense_words = g.hm_dense_words;
  const int G = (int)(dense_words / 4);  // 128-bit groups of the dense slots
  const int D = (int)(dense_words * 32);
  const unsigned below = (1u << lane) - 1u, upto = kFull >> (31 - lane);
  const int64_t units = __ldg(unit_off + ndense);
  if (threadIdx.x == 0) cur = (int64_t)atomicAdd(counter, 1ull);
  __syncthreads();
  for (;;) {
    const int64_t unit = cur;
    if (unit >= units) break;
    // the next unit's number, stored at the end of this one
    unsigned long long following = 0;
    if (threadIdx.x == 0) following = atomicAdd(counter, 1ull);
    const int64_t idx = __ldg(unit_idx + unit);
    const int64_t e = dense_e[idx];
    const uint4* m = reinterpret_cast<const uint4*>(tmask + idx * dense_words);
    const int64_t b = toff[e], te = (int64_t)t[e];
    const int64_t r0 = (unit - __ldg(unit_off + idx)) * kDenseUnit;
    const int32_t* Te = T + b;
    const int16_t* Ts = T_hm + b;
    int L = 0, M = 0;  // non-zero groups and members so far (the same in every thread)
    for (int i0 = 0; i0 < G; i0 += kDenseThreads) {
      const int i = i0 + threadIdx.x;
      const uint4 mv = i < G ? m[i] : make_uint4(0u, 0u, 0u, 0u);
      const int pc = __popc(mv.x) + __popc(mv.y) + __popc(mv.z) + __popc(mv.w);
      const unsigned bal = __ballot_sync(kFull, pc != 0);
      int incl = pc;
#pragma unroll
      for (int k = 1; k < 32; k <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, k);
        if (lane >= k) incl += y;
      }
      if (lane == 31) {
        wcnt[wid] = __popc(bal);
        wlen[wid] = incl;
      }
      __syncthreads();
      int at = L + __popc(bal & below), mb = M + incl - pc;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        at += w < wid ? wcnt[w] : 0;
        mb += w < wid ? wlen[w] : 0;
        L += wcnt[w];
        M += wlen[w];
      }
      if (pc) {
        smask[at] = mv;
        sgrp[at] = (uint16_t)i;
        sbase[at] = (uint16_t)mb;
      }
      __syncthreads();  // wcnt and wlen are rewritten by the next round
    }
    const bool others = (int64_t)M < te;
    const bool filt = others && te <= kTFilterMaxT;
    if (filt)
      for (int i = threadIdx.x; i < kTFilterWords; i += kDenseThreads) tfilt[i] = 0u;
    // members of rank [r0, r0 + kDenseUnit), a mask word per thread
    const int nmem = (int)min((int64_t)kDenseUnit, max((int64_t)0, (int64_t)M - r0));
    if (nmem > 0)
      for (int i = threadIdx.x; i < 4 * L; i += kDenseThreads) {
        const int c = i >> 2, w4 = i & 3;
        const uint4 mv = smask[c];
        uint32_t bits = w4 == 0 ? mv.x : w4 == 1 ? mv.y : w4 == 2 ? mv.z : mv.w;
        int64_t rank = (int64_t)sbase[c] - r0 + (w4 > 0 ? __popc(mv.x) : 0) +
                       (w4 > 1 ? __popc(mv.y) : 0) + (w4 > 2 ? __popc(mv.z) : 0);
        const int s0 = sgrp[c] * 128 + w4 * 32;
        for (; bits; bits &= bits - 1, ++rank)
          if (rank >= 0 && rank < nmem) {
            mslot[rank] = (uint16_t)(s0 + __ffs(bits) - 1);
            mgrp[rank] = (uint8_t)c;
          }
      }
    __syncthreads();
    if (filt)
      for (int64_t i = threadIdx.x; i < te; i += kDenseThreads)
        if (__ldg(Ts + i) < 0) {
          const uint32_t h = tfilter_hash(__ldg(Te + i));
          atomicOr(tfilt + (h >> 5), 1u << (h & 31u));
        }
    // dense-slot pairs: eight lanes per member, eight members per warp
    unsigned acc = 0, groups = 0;
    const int sub = lane >> 3, l8 = lane & 7;
    for (int m0 = wid * 8; m0 < nmem; m0 += kWarps * 8) {
      int p0[2], b0[2];
      const uint4* row[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = m0 + 2 * sub + h;
        const int s = r < nmem ? (int)mslot[r] : 0;
        p0[h] = r < nmem ? (int)mgrp[r] : -1;
        b0[h] = s & 127;
        row[h] = reinterpret_cast<const uint4*>(g.hm_bits + (int64_t)s * g.hm_words);
        groups += p0[h] + 1;  // the same in the eight lanes
      }
      const int last = max(p0[0], p0[1]);
      for (int c = l8; c <= last; c += 8) {
        const int gg = sgrp[c];
        const uint4 mk = smask[c];
        uint4 rv[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          rv[h] = c <= p0[h] ? ld_keep4(row[h] + gg) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t wd[4] = {rv[h].x & mk.x, rv[h].y & mk.y, rv[h].z & mk.z, rv[h].w & mk.w};
          if (c == p0[h]) {  // the member's own group: only the bits below its own
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) wd[q4] &= bits_below(b0[h] - 32 * q4);
          }
          acc += __popc(wd[0]) + __popc(wd[1]) + __popc(wd[2]) + __popc(wd[3]);
        }
      }
    }
    groups = l8 == 0 ? groups : 0u;
    // members without a dense slot: w's matrix neighbours x (a bit of the
    // mask below D; past D, x = hm_vertex[s] counts when above w and in T)
    // and w's neighbours above w without a matrix slot (counted when in T).
    // A warp walks the concatenation of these lists for 32 T entries.
    unsigned long long rtested = 0;
    if (others) {
      __syncthreads();  // the filter is complete
      const uint32_t* mask32 = tmask + idx * dense_words;
      const int64_t len = min(te, r0 + kDenseUnit);
      int64_t* wa = ra + wid * 32;
      int64_t* wb = rb + wid * 32;
      int32_t* wv = rw + wid * 32;
      int32_t* wna = rna + wid * 32;
      int32_t* wst = rst + wid * 32;
      for (int64_t c0 = r0 + (int64_t)wid * 32; c0 < len; c0 += kDenseThreads) {
        int32_t w = -1, na = 0, nb = 0;
        int64_t a0 = 0, n0 = 0;
        const int64_t j = c0 + lane;
        if (j < len) {
          const int xs = __ldg(Ts + j);
          if (!(xs >= 0 && xs < D)) {
            w = __ldg(Te + j);
            a0 = __ldg(g.mn_ptr + w);
            na = (int32_t)(__ldg(g.mn_ptr + w + 1) - a0);
            n0 = __ldg(g.nm_ptr + w);
            nb = (int32_t)(__ldg(g.nm_ptr + w + 1) - n0);
          }
        }
        const unsigned nz = __ballot_sync(kFull, na + nb > 0);
        if (nz == 0) continue;
        // start of the list in the concatenation; lane i then keeps the start
        // of the i-th list (the total past the lists)
        int32_t start = na + nb;
#pragma unroll
        for (int k = 1; k < 32; k <<= 1) {
          const int32_t y = __shfl_up_sync(kFull, start, k);
          if (lane >= k) start += y;
        }
        const int32_t total = __shfl_sync(kFull, start, 31);
        __syncwarp();  // the previous entries are no longer read
        if (na + nb > 0) {
          const int at = __popc(nz & below);
          wa[at] = a0;
          wb[at] = n0;
          wv[at] = w;
          wna[at] = na;
          wst[at] = start - (na + nb);
        }
        __syncwarp();
        const int cnt = __popc(nz);
        start = lane < cnt ? wst[lane] : total;
        for (int32_t p = 0; p < total; p += 32) {
          const int j0 = __popc(__ballot_sync(kFull, start <= p)) - 1;
          const int32_t ds = start - p;
          const unsigned marks = __reduce_or_sync(kFull, ds > 0 && ds < 32 ? 1u << ds : 0u);
          const int k = min(j0 + __popc(marks & upto), cnt - 1);
          const int32_t o = p + lane - __shfl_sync(kFull, start, k);
          if (p + lane < total) {
            bool hit;
            if (o < wna[k]) {
              const int sx = __ldg(g.mn_slot + wa[k] + o);
              if (sx < D) {
                hit = ((__ldg(mask32 + (sx >> 5)) >> (sx & 31)) & 1u) != 0;
              } else {
                const int32_t x = __ldg(g.hm_vertex + sx);
                hit = x > wv[k] && sorted_contains(Te, te, x);
              }
            } else {
              const int32_t x = __ldg(g.nm_col + wb[k] + (o - wna[k]));
              const uint32_t h = tfilter_hash(x);
              hit = (!filt || ((tfilt[h >> 5] >> (h & 31u)) & 1u) != 0) &&
                    sorted_contains(Te, te, x);
            }
            acc += hit ? 1u : 0u;
          }
        }
        rtested += lane == 0 ? total : 0;
      }
    }
    unsigned long long acc64 = warp_sum<unsigned long long>(acc);
    rtested = warp_sum<unsigned long long>(rtested);
    const unsigned long long gsum = warp_sum<unsigned long long>(groups);
    if (lane == 0) {
      part[wid][0] = acc64;
      part[wid][1] = gsum;
      part[wid][2] = rtested;
    }
    if (threadIdx.x == 0) cur = (int64_t)following;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long sk = 0, sg = 0, sr = 0;
      for (int w = 0; w < kWarps; ++w) {
        sk += part[w][0];
        sg += part[w][1];
        sr += part[w][2];
      }
      if (sk) {
        atomicAdd(k_out + e, sk);
        if (need_q) atomicAdd(q + e, 2 * sk);
      }
      if (sg) atomicAdd(tests, sg);
      if (sr) atomicAdd(rest_tests, sr);
    }
    // the masks, lists and part are reused for the next unit, whose first
    // writes to them follow a barrier or are this thread's own
  }
}

// ---------------------------------------------------------------- items
// One item per position of a 32-position chunk: w = N(u)[i], w != v.
// With T = N(u) cap N(v) and c(x, y) = |N(x) cap N(y)|, the 4-node terms are
//   k = sum_{w in T} |N(w) cap T, above w|                 (each pair once)
//   q = sum_{w in S_u} (c(w, v) - 1) - sum_{r in T} (c(r, u) - 1) + 2k
// The second line is sum_{w in S_u} (|N(w) cap N(v)| - |N(w) cap T| - 1)
// with sum_{w in S_u} |N(w) cap T| = sum_{r in T} (c(r, u) - 1) - 2k
// (count the pairs (r in T, w in N(u) \ {v}) with r ~ w from the r side).
// Each item carries up to two segments of membership tests:
//   A (w in T):  x over the shorter of N(w) above w / T above w, tested in
//                the other; a hit is one 4-clique pair: k += 1, q += 2.
//   B (c(w, o)): o = u for w in T, o = v for w in S_u; x over the shorter
//                adjacency, tested in the longer; q -= 1 / q += 1 per hit.
//                Skipped (constant term instead) when the co-degree table
//                holds c(w, o).
// The searched side is a vertex y's adjacency (set_search) or a T list.
struct Seg {
  const int32_t* it;    // iterated list (its matrix slots lie beside it)
  const int32_t* sl;    // searched list
  int32_t sslot;        // matrix slot of y, or -1
  int32_t sbm;          // bitmap slot of y (>= 0), -2 - s when y has a
                        // bucket directory with shift s, else -1
  int32_t slen;         // length of sl, or (sbm < -1) the first entry of
                        // y's directory in g.dir
  int32_t cnt;          // number of tests
};

// Segment A of an item w in T (k_quad) counts the pairs above w. In a dense
// edge no item has a segment A: k_dense_pairs counts all of that edge's
// pairs.

struct EdgeCtx {
  int64_t e;
  int32_t u, v;
  int64_t bu, du, bv, dv;
  int64_t te, toff;
  const uint32_t* tmask;  // this edge's T mask (dense edges), else NULL
};

// What the cost pass keeps of an edge: the endpoints' lists, and for each end
// o of its co-degree queries c(w, o) (o = u for w in T, o = v for w in S_u)
// the row of a small graph's co-degree block shifted so that w's entry is
// row[w] (NULL without a block), the table slot and the mid x big column.
struct CostEdge {
  int64_t e, first, end;  // edge, its positions [first, end)
  int64_t bu, te;
  int32_t v, du, dv;
  bool dense;
  const uint8_t *row_u, *row_v;
  int32_t slot_u, slot_v, col_u, col_v;
};

__device__ __forceinline__ const uint8_t* block_row(const DevGraph& g, int32_t o) {
  const int64_t r = __ldg(g.cg_row + o);
  return r >= 0 ? g.cg + (r - __ldg(g.dm_first + o)) : nullptr;
}

__device__ __forceinline__ void load_edge(const DevGraph& g, const int2* __restrict__ uv,
                                          const unsigned long long* __restrict__ t,
                                          const int64_t* __restrict__ toff,
                                          const int32_t* __restrict__ mask_idx,
                                          const uint32_t* __restrict__ tmask, int64_t e,
                                          EdgeCtx& c) {
  const int32_t mi = mask_idx != nullptr ? mask_idx[e] : -1;
  c.tmask = mi >= 0 ? tmask + (int64_t)mi * g.hm_dense_words : nullptr;
  int2 pr = uv[e];
  c.e = e;
  c.u = pr.x;
  c.v = pr.y;
  c.du = deg_of(g.row_ptr, pr.x, &c.bu);
  c.dv = deg_of(g.row_ptr, pr.y, &c.bv);
  c.te = (int64_t)t[e];
  c.toff = toff[e];
}

// c(w, o) + 1 from the co-degree table when both are table hubs or from the
// mid x big table when one is a mid vertex and the other a big hub; 0 when
// neither can answer (the +1 marks a present entry). sw, so: table slots (-1
// none, <= -2 a mid row); co: o's mid x big column (-1 none).
__device__ __forceinline__ uint32_t table_codeg(const DevGraph& g, int32_t w, int32_t sw,
                                                int32_t so, int32_t co) {
  if (sw >= 0 && so >= 0) {
    const int32_t lo = min(sw, so), hi = max(sw, so);
    const uint16_t c = ld_once16(g.tb_codeg + tb_index(lo, hi, g.tb_count));
    if (c != 0xFFFFu) return (uint32_t)c + 1u;
    if (g.tb_giant != nullptr) {  // a pair of giants
      const int32_t ga = __ldg(g.tb_giant + lo), gb = __ldg(g.tb_giant + hi);
      if (ga >= 0 && gb >= 0) return __ldg(g.tb_giant_codeg + (int64_t)ga * g.tb_giants + gb) + 1u;
    }
    return 0;  // a true co-degree of 65,535 is left to the tests
  }
  if (g.md_codeg != nullptr && (sw < -1 || so < -1) && (sw >= 0 || so >= 0)) {
    // one mid vertex (slot -2 - row), one table vertex that may be big
    const int32_t col = sw >= 0 ? __ldg(g.bg_slot + w) : co;
    if (col >= 0)
      return (uint32_t)ld_once16(g.md_codeg + (int64_t)(-2 - min(sw, so)) * g.bg_count + col) + 1u;
  }
  return 0;
}

// sslot value marking a searched vertex whose adjacency is a dense bit-matrix
// row: sl then points at the row and sbm holds the first vertex of the block.
constexpr int32_t kDenseRow = -3;

// The searched side of a segment: vertex y's adjacency, answered by its
// dense row, the hub-pair matrix, its bitmap, or a halving search.
__device__ __forceinline__ void set_search(const DevGraph& g, int32_t y, int64_t by, int64_t dy,
                                           Seg& s) {
  s.sl = g.col + by;
  s.slen = (int32_t)dy;
  if (g.dm_row != nullptr) {
    const int64_t r = __ldg(g.dm_row + y);
    if (r >= 0) {
      s.sslot = kDenseRow;
      s.sl = reinterpret_cast<const int32_t*>(g.dm_bits + r);
      s.sbm = __ldg(g.dm_first + y);
      return;
    }
  }
  s.sslot = table_slot(g, y);
  s.sbm = bitmap_slot(g, y);
  if (s.sbm < 0 && g.dir_at != nullptr) {
    const int64_t at = __ldg(g.dir_at + y);
    if (at >= 0) {
      s.slen = (int32_t)at;
      s.sbm = -2 - (g.id_bits - dir_log2(dy, g.id_bits));
    }
  }
}

// Segment for c(w, o): iterate the shorter adjacency, test in the longer.
__device__ __forceinline__ void codeg_segment(const DevGraph& g, int32_t w, int64_t bw, int64_t dw,
                                              int32_t o, int64_t bo, int64_t dob, Seg& s) {
  if (dw <= dob) {
    s.it = g.col + bw;
    s.cnt = (int32_t)dw;
    set_search(g, o, bo, dob, s);
  } else {
    s.it = g.col + bo;
    s.cnt = (int32_t)dob;
    set_search(g, w, bw, dw, s);
  }
}

// Tests of item i of an edge (segment A + segment B) and its constant q
// term, for the cost pass (the 4-node pass re-derives the segments in
// setup_item). The table slot of w comes from beside the adjacency when
// the graph has it, so the table read does not wait for a gather.
struct ItemCost {
  int32_t a, b;    // tests of segments A and B
  int32_t qconst;  // constant q contribution (a co-degree is below n < 2^31)
  bool tabled;     // a co-degree table answered segment B
};

// Most items are in S_u and answered by a table: for those only the element,
// its table slot and the table entry are read; degrees are read by the rest.
// w: the item's vertex (-1: no item), sw: its table slot (-1 without tables).
__device__ __forceinline__ ItemCost item_cost(const DevGraph& g, const CostEdge& c, int32_t w,
                                              int32_t sw, uint32_t tword,
                                              const int32_t* __restrict__ tpre, int lane,
                                              bool need_q) {
  ItemCost r{0, 0, 0, false};
  if (w < 0 || w == c.v) return r;
  const bool in_t = (tword >> lane) & 1u;
  if (need_q) {
    // segment B: -(c(w, u) - 1) for w in T, c(w, v) - 1 for w in S_u
    const uint8_t* row = in_t ? c.row_u : c.row_v;
    uint32_t tc = 0;
    if (row != nullptr) {
      const uint32_t b = __ldg(row + w);
      if (b < 255u) tc = b + 1u;
    }
    if (tc == 0 && g.tb_slot != nullptr) {
      if (g.col_tb == nullptr) sw = __ldg(g.tb_slot + w);
      tc = table_codeg(g, w, sw, in_t ? c.slot_u : c.slot_v, in_t ? c.col_u : c.col_v);
    }
    r.tabled = tc != 0;
    if (tc != 0) {
      r.qconst = in_t ? 2 - (int32_t)tc : (int32_t)tc - 2;
    } else {
      r.qconst = in_t ? 1 : -1;
      r.b = (int32_t)min(__ldg(g.row_ptr + w + 1) - __ldg(g.row_ptr + w),
                         (int64_t)(in_t ? c.du : c.dv));
    }
  }
  if (in_t && !c.dense) {
    // |N(w) above w cap T above w|: the shorter side is iterated (in a dense
    // edge segment A is k_dense_pairs' work)
    const int64_t tg = c.te - (__ldg(tpre) + __popc(tword & ((1u << lane) - 1u))) - 1;
    if (tg > 0) r.a = (int32_t)min(__ldg(g.row_ptr + w + 1) - __ldg(g.up_ptr + w), tg);
  }
  return r;
}


// Chunk costs: membership tests per chunk and the number of tasks it needs.
// Also adds the constant part of q. Bound by the latency of the table reads
// (two bytes of a random sector per item); cost phase of the 1M-vertex
// power-law graph exact: 131 -> 114 ms when the items a table answers stopped
// reading their degrees and the sums went to 32-bit warp reductions, 110 ms
// with one addition to q per edge and run. Loading the next chunk's elements
// ahead spilled at 40 registers (119 ms) and gave 112 ms at 64.
__global__ void __launch_bounds__(kThreads, kCostBlocksPerSm)
    k_chunk_cost(DevGraph g, const int2* __restrict__ uv, const int64_t* __restrict__ off, int64_t K,
                 const unsigned long long* __restrict__ t, const uint32_t* __restrict__ tbits,
                 const int32_t* __restrict__ tpre, const int32_t* __restrict__ mask_idx,
                 int need_q, int64_t task_probes, int64_t* __restrict__ task_cnt,
                 uint32_t* __restrict__ cbits, unsigned long long* __restrict__ q,
                 unsigned long long* __restrict__ stats) {
  unsigned long long tests = 0;
  const int lane = threadIdx.x & 31;
  const int64_t P = __ldg(off + K);
  const int64_t groups = P >> 5;  // padded: P is a multiple of 32
  CostEdge c;
  c.e = -1;
  c.first = c.end = 0;
  c.row_u = c.row_v = nullptr;
  c.slot_u = c.slot_v = c.col_u = c.col_v = -1;
  // runs of consecutive chunks from a counter (chunks differ in cost: table
  // answers, hub edges)
  const int grab =
      chunk_run_length(groups, (int64_t)gridDim.x * (kThreads / 32), (int64_t)kCostGrab);
  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(stats + 8, (unsigned long long)grab);
    const int64_t g0 = (int64_t)__shfl_sync(kFull, got, 0);
    if (g0 >= groups) break;
    const int64_t g1 = min(groups, g0 + grab);
    // packs: consecutive chunks of the run with at most 32 live items in all,
    // so that k_quad sets up a warp's worth of items at a time; a pack's
    // tasks are counted at its first chunk
    int64_t head = g0, pcost = 0, qsum = 0;  // qsum: constant of edge c.e in this run
    int plive = 0;
    for (int64_t gi = g0; gi < g1; ++gi) {
      const int64_t p0 = gi * 32;
      if (p0 < c.first || p0 >= c.end) {  // another edge: the next one, or a search
        if (qsum != 0 && lane == 0) atomicAdd(q + c.e, (unsigned long long)qsum);
        qsum = 0;
        c.e = p0 == c.end && c.e >= 0 ? c.e + 1 : last_le(off, K, p0);
        c.first = __ldg(off + c.e);
        c.end = __ldg(off + c.e + 1);
        const int2 pr = uv[c.e];
        c.v = pr.y;
        c.du = (int32_t)deg_of(g.row_ptr, pr.x, &c.bu);
        c.dv = (int32_t)(__ldg(g.row_ptr + pr.y + 1) - __ldg(g.row_ptr + pr.y));
        c.te = (int64_t)t[c.e];
        c.dense = mask_idx != nullptr && mask_idx[c.e] >= 0;
        if (g.cg_row != nullptr) {
          c.row_u = block_row(g, pr.x);
          c.row_v = block_row(g, pr.y);
        }
        if (g.tb_slot != nullptr) {
          c.slot_u = __ldg(g.tb_slot + pr.x);
          c.slot_v = __ldg(g.tb_slot + pr.y);
        }
        if (g.bg_slot != nullptr) {
          c.col_u = __ldg(g.bg_slot + pr.x);
          c.col_v = __ldg(g.bg_slot + pr.y);
        }
      }
      const int64_t i = p0 + lane - c.first, at = c.bu + i;
      const int32_t w = i < c.du ? __ldg(g.col + at) : -1;
      const int32_t sw = g.col_tb != nullptr && i < c.du ? __ldg(g.col_tb + at) : -1;
      const uint32_t tword = __ldg(tbits + gi);
      const ItemCost it = item_cost(g, c, w, sw, tword, tpre + gi, lane, need_q);
      const unsigned live = __ballot_sync(kFull, (it.a | it.b) != 0);
      const unsigned tabled = __ballot_sync(kFull, it.tabled);
      if (lane == 0) reinterpret_cast<uint2*>(cbits)[gi] = make_uint2(live, tabled);
      // sums over the warp, in 32 bits while every term is far from them
      constexpr int32_t kSmall = 1 << 24;
      const bool wide = __any_sync(kFull, it.a > kSmall || it.b > kSmall || it.qconst > kSmall ||
                                              it.qconst < -kSmall);
      int64_t cost, qc;
      if (wide) {
        cost = warp_sum<int64_t>((int64_t)it.a + it.b);
        qc = warp_sum<int64_t>(it.qconst);
      } else {
        cost = __reduce_add_sync(kFull, it.a + it.b);
        qc = __reduce_add_sync(kFull, it.qconst);
      }
      if (plive + __popc(live) > 32) {
        if (lane == 0) task_cnt[head] = (pcost + task_probes - 1) / task_probes;
        head = gi;
        pcost = 0;
        plive = 0;
      }
      pcost += cost;
      plive += __popc(live);
      if (lane == 0) {
        if (gi != head) task_cnt[gi] = 0;
        tests += cost;
      }
      qsum += qc;
    }
    if (qsum != 0 && lane == 0) atomicAdd(q + c.e, (unsigned long long)qsum);
    if (lane == 0) task_cnt[head] = (pcost + task_probes - 1) / task_probes;
  }
  if (lane == 0 && tests) atomicAdd(stats + 1, (unsigned long long)tests);
}

// ---------------------------------------------------------------- quad

// Membership of x in a directory bucket p[0..len): short buckets (the usual
// case: 2 to 4 entries) are compared entry by entry with independent loads.
__device__ __forceinline__ bool bucket_contains(const int32_t* __restrict__ p, int32_t len,
                                                int32_t x) {
  if (len <= 4) {
    bool f = false;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < len) f |= __ldg(p + k) == x;
    return f;
  }
  return sorted_contains(p, len, x);
}

// The items of the pack a warp works on, field by field so that lanes that
// read different items hit different banks (60 bytes per item: eight CTAs of
// 256 items take 120 KB of shared memory, which leaves the rest of the SM's
// 256 KB to the L1 cache that the membership tests depend on). Only items
// with tests are kept, in order of position. [0] is segment A, [1] segment B.
// The matrix slots of an iterated list are found beside it (col_hm for
// adjacency lists, T_hm for T).
struct WarpItems {
  const int32_t* it[2][32];
  const int32_t* sl[2][32];
  int32_t sbm[2][32];
  int32_t slen[2][32];
  int32_t ca[32];       // tests of segment A; its hits count +1 in k, +2 in q
  int16_t sslot[2][32];
  int16_t bsign[32];    // segment B adds it to q per hit
  uint16_t who[32];     // chunk of the pack (high bits) and bit of each item
};
static_assert(sizeof(WarpItems) == 60 * 32, "WarpItems size");

// Item set-up of k_quad, out of line: it runs once per pack and its
// temporaries would otherwise raise the register count of the test loop.
// Derives the same segments as item_cost counts for position i of edge e
// (bit `bit` of its chunk, an item with tests), with the cost pass's word on
// whether a table answered segment B in place of the table reads, and stores each field to place `at` of the
// warp's item arrays as soon as it is known (only the segments that have
// tests are written; a segment with no tests is never read). Returns the
// item's test count.
__device__ __noinline__ int64_t setup_item(const DevGraph& g, const int2* __restrict__ uv,
                                           const unsigned long long* __restrict__ t,
                                           const int64_t* __restrict__ toff,
                                           const int32_t* __restrict__ mask_idx,
                                           const uint32_t* __restrict__ tmask, int64_t e,
                                           const int32_t* __restrict__ T, int64_t i,
                                           uint32_t tword, int32_t tbase, int bit, bool need_q,
                                           bool tabled, WarpItems* wi, int at) {
  EdgeCtx c;
  load_edge(g, uv, t, toff, mask_idx, tmask, e, c);
  int32_t ca = 0, cb = 0, bsign = 0;
  if (i < c.du) {
    const int32_t w = __ldg(g.col + c.bu + i);
    if (w != c.v) {
      const bool in_t = (tword >> bit) & 1u;
      int64_t bw;
      const int64_t dw = deg_of(g.row_ptr, w, &bw);
      if (in_t && c.tmask != nullptr) {
        // dense edge: segment A is done by k_dense_pairs
      } else if (in_t) {
        const int64_t iw = tbase + __popc(tword & ((1u << bit) - 1u));
        const int64_t tg = c.te - iw - 1;
        const int64_t upw = __ldg(g.up_ptr + w);
        const int64_t dup = bw + dw - upw;
        if (dup <= tg) {
          wi->it[0][at] = g.col + upw;
          wi->sl[0][at] = T + c.toff + iw + 1;
          wi->slen[0][at] = (int32_t)tg;
          wi->sslot[0][at] = -1;
          wi->sbm[0][at] = -1;
          ca = (int32_t)dup;
        } else {
          Seg sa;
          set_search(g, w, bw, dw, sa);
          wi->it[0][at] = T + c.toff + iw + 1;
          wi->sl[0][at] = sa.sl;
          wi->slen[0][at] = sa.slen;
          wi->sslot[0][at] = (int16_t)sa.sslot;
          wi->sbm[0][at] = sa.sbm;
          ca = (int32_t)tg;
        }
      }
      if (need_q) {
        // segment B: c(w, u) for w in T (q -= 1 per hit), c(w, v) for w in
        // S_u (q += 1 per hit), unless a co-degree table answered it
        bsign = in_t ? -1 : 1;
        if (!tabled) {
          Seg sb;
          if (in_t) codeg_segment(g, w, bw, dw, c.u, c.bu, c.du, sb);
          else codeg_segment(g, w, bw, dw, c.v, c.bv, c.dv, sb);
          wi->it[1][at] = sb.it;
          wi->sl[1][at] = sb.sl;
          wi->slen[1][at] = sb.slen;
          wi->sslot[1][at] = (int16_t)sb.sslot;
          wi->sbm[1][at] = sb.sbm;
          cb = sb.cnt;
        }
      }
    }
  }
  wi->ca[at] = ca;
  wi->bsign[at] = bsign;
  return (int64_t)ca + cb;
}

// One side of a membership test, as loaded so far: a word and a bit to test
// (matrix, bitmap, dense row), the bounds of a directory bucket, or nothing
// yet (a halving search is left).
struct Probe {
  uint32_t word, bit;
  int how;  // 0 search, 1 word, 2 bucket
};

// First loads of the test "x in the searched set". xs: x's matrix slot, -1
// when it has none; kMayMatrix false: the set has no matrix row (sslot < 0).
template <bool kMayMatrix>
__device__ __forceinline__ Probe probe_begin(const DevGraph& g, int sslot, int32_t sbm,
                                             const int32_t* sl, int32_t slen, int32_t x,
                                             int32_t xs) {
  Probe p{0u, 0u, 0};
  if (kMayMatrix && sslot >= 0 && xs >= 0) {
    p.word = ld_keep(g.hm_bits + (int64_t)sslot * g.hm_words + (xs >> 5));
    p.bit = xs & 31;
    p.how = 1;
  } else if (sslot == kDenseRow) {
    const int32_t lx = x - sbm;
    p.word = __ldg(reinterpret_cast<const uint32_t*>(sl) + (lx >> 5));
    p.bit = lx & 31;
    p.how = 1;
  } else if (sbm >= 0) {
    p.word = __ldg(g.bm_bits + (int64_t)sbm * g.bm_words + (x >> 5));
    p.bit = x & 31;
    p.how = 1;
  } else if (sbm < -1) {
    const uint32_t* d = g.dir + (uint32_t)slen + (uint32_t)(x >> (-2 - sbm));
    p.word = __ldg(d);
    p.bit = __ldg(d + 1);
    p.how = 2;
  }
  return p;
}

__device__ __forceinline__ bool probe_end(const Probe& p, const int32_t* sl, int32_t slen,
                                          int32_t x) {
  return p.how == 1   ? ((p.word >> p.bit) & 1u) != 0
         : p.how == 2 ? bucket_contains(sl + p.word, (int32_t)(p.bit - p.word), x)
                      : sorted_contains(sl, slen, x);
}

// Matrix slots beside an iterated list: col_hm for an adjacency list, T_hm
// for a T list (NULL without a matrix).
__device__ __forceinline__ const int16_t* slots_beside(const DevGraph& g, const int32_t* it,
                                                       const int32_t* T, const int16_t* T_hm) {
  if (T_hm == nullptr) return nullptr;
  const size_t pc = (size_t)(it - g.col);
  return pc < (size_t)g.nnz ? g.col_hm + pc : T_hm + (it - T);
}

// The 4-node membership tests. A pack is up to 32 items with tests from
// consecutive chunks (of one edge or several); its tests (the items' segments
// A and B in order) are one index space, cut into tasks of task_probes tests.
// A warp walks a task from test r on in one of two ways:
//   run   the next 64 or more tests belong to one segment: its descriptor is
//         the same in every lane, so the set searched and the way it answers
//         are chosen once per run, and lanes take consecutive elements, two
//         each per step;
//   mixed otherwise, 64 tests of several items: each lane finds the item of
//         its two tests from bit masks of the item starts among those 64
//         (one warp reduction per 32), and reads its descriptor.
// Lane i owns item i: it counts the item's hits from the hit ballots, whose
// bits [start, end) are the item's tests, and adds them to the item's edge.
//
// Why packs: a chunk of 32 positions has few items left after the tables
// (3.8 on the 1M-vertex power-law graph, 11 on R-MAT 24), so setting up one
// chunk at a time left most lanes idle in the set-up, which was most of the
// work there (850 of 1390 warp instructions per chunk). Eight CTAs per SM at
// 32 registers, some spilled, hide more latency than six at 40 (R-MAT 24
// 0.1%: 151 against 160 ms; 1M-vertex power-law exact 456 against 457 ms).
// The look for a run is left out where no item of the pack has one: a uniform
// graph's items have a few dozen tests, and the look and the hit masks made the
// phase slower than five shuffles per test had been (ER of mean degree 20 / 40,
// 4M edges exact 13.3 / 50.5 -> 12.3 / 46.9 ms).
__global__ void __launch_bounds__(kThreads, kQuadBlocksPerSm)
    k_quad(const __grid_constant__ DevGraph g, const int2* __restrict__ uv, const int64_t* __restrict__ off, int64_t K,
           const unsigned long long* __restrict__ t, const int64_t* __restrict__ toff,
           const uint32_t* __restrict__ tbits, const int32_t* __restrict__ tpre,
           const uint32_t* __restrict__ cbits,
           const int32_t* __restrict__ T, const int16_t* __restrict__ T_hm,
           const int32_t* __restrict__ mask_idx, const uint32_t* __restrict__ tmask,
           const int64_t* __restrict__ task_off,
           int64_t groups, int need_k, int need_q, int64_t task_probes,
           unsigned long long* __restrict__ k_out,
           unsigned long long* __restrict__ q,
           unsigned long long* __restrict__ task_counter) {
  __shared__ WarpItems items[kThreads / 32];
  const int lane = threadIdx.x & 31;
  const unsigned upto = kFull >> (31 - lane);
  WarpItems* my = items + (threadIdx.x >> 5);
  // warps take runs of consecutive tasks from a counter: tasks differ in
  // cost (a pack with few tests still pays a whole item set-up, tests
  // differ in latency), so fixed per-warp ranges left a long tail
  const int grab = run_length(__ldg(task_off + groups), (int64_t)gridDim.x * (kThreads / 32),
                              max((int64_t)1, kQuadGrabTests / task_probes));
  for (;;) {
    unsigned long long got = 0;
    if (lane == 0) got = atomicAdd(task_counter, (unsigned long long)grab);
    int64_t task = (int64_t)__shfl_sync(kFull, got, 0);
    int left = (int)min((int64_t)grab, __ldg(task_off + groups) - task);
    if (left <= 0) break;
    int64_t gi = last_le_warp(task_off, groups, task);
    int64_t e0 = last_le_warp(off, K, gi * 32);
    while (left > 0) {
      // the tasks of this run that lie in the pack at chunk gi
      while (__ldg(task_off + gi + 1) <= task) ++gi;
      while (e0 + 1 < K && __ldg(off + e0 + 1) <= gi * 32) ++e0;
      int here = (int)min((int64_t)left, __ldg(task_off + gi + 1) - task);
      left -= here;
      // lane c: chunk gi + c of the pack (up to the next chunk with tasks of
      // its own) and the items with tests in it
      uint2 cb = make_uint2(0u, 0u);
      bool own = false;
      if (lane < kCostGrab && gi + lane < groups) {
        cb = __ldg(reinterpret_cast<const uint2*>(cbits) + gi + lane);
        own = lane > 0 && __ldg(task_off + gi + lane + 1) > __ldg(task_off + gi + lane);
      }
      const unsigned heads = __ballot_sync(kFull, own);
      if (heads && lane >= __ffs(heads) - 1) cb.x = 0u;
      int upto_c = __popc(cb.x);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(kFull, upto_c, d);
        if (lane >= d) upto_c += y;
      }
      const int live = __shfl_sync(kFull, upto_c, 31);
      __syncwarp();  // the previous pack's descriptors are no longer read
      for (unsigned bits = cb.x, k = upto_c - __popc(cb.x); bits; bits &= bits - 1, ++k) {
        const int b = __ffs(bits) - 1;
        my->who[k] = (uint16_t)((lane << 6) | (((cb.y >> b) & 1u) << 5) | b);
      }
      __syncwarp();
      // lane i: the set-up of item i
      int64_t e = e0, mine = 0;
      if (lane < live) {
        const int who = my->who[lane];
        const int64_t gc = gi + (who >> 6);
        while (e + 1 < K && __ldg(off + e + 1) <= gc * 32) ++e;
        mine = setup_item(g, uv, t, toff, mask_idx, tmask, e, T,
                          gc * 32 + (who & 31) - __ldg(off + e), __ldg(tbits + gc),
                          __ldg(tpre + gc), who & 31, need_q, ((who >> 5) & 1) != 0, my, lane);
      }
      __syncwarp();
      int64_t start = mine;  // first test of the item; the total past the items
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        int64_t y = __shfl_up_sync(kFull, start, d);
        if (lane >= d) start += y;
      }
      const int64_t ctotal = __shfl_sync(kFull, start, 31);
      start -= mine;
      unsigned long long acc_a = 0, acc_b = 0;  // hits of the lane's item
      const bool runs = __any_sync(
          kFull, lane < live && (my->ca[lane] >= 64 || mine - my->ca[lane] >= 64));
      for (; here > 0; --here, ++task) {
        const int64_t lo = (task - __ldg(task_off + gi)) * task_probes;
        const int32_t len = (int32_t)min(ctotal - lo, task_probes);
        // item starts relative to the task's first test, in 32 bits: clamping
        // keeps their order and never touches the item that holds a test of
        // this task (it starts less than one item's tests before lo)
        const int32_t srel = (int32_t)max(min(start - lo, task_probes), (int64_t)INT32_MIN + 1);
        // segment B of the item starts at sb, the item ends at se
        const int32_t sb =
            (int32_t)max(min(start - lo + (lane < live ? my->ca[lane] : 0), task_probes),
                         (int64_t)INT32_MIN + 1);
        const int32_t sd = __shfl_down_sync(kFull, srel, 1);
        const int32_t se = lane < 31 ? min(sd, len) : len;
        for (int32_t r = 0; r < len;) {
          // item of test r: the last one that starts at or before it (lanes
          // past the items hold the total, which is at or past len)
          const int j0 = 31 - __clz(__ballot_sync(kFull, srel <= r));
          if (runs) {  // some segment has 64 tests
            const int32_t sj = __shfl_sync(kFull, srel, j0);
            const int32_t sbj = __shfl_sync(kFull, sb, j0);
            const int32_t sej = __shfl_sync(kFull, se, j0);
            const int sg = r >= sbj ? 1 : 0;
            const int32_t end = sg ? sej : min(sbj, len);
            if (end - r >= 64) {
              const int32_t* it = my->it[sg][j0] + (r - (sg ? sbj : sj)) + lane;
              const int32_t* sl = my->sl[sg][j0];
              const int32_t sbm = my->sbm[sg][j0], slen = my->slen[sg][j0];
              const int sslot = my->sslot[sg][j0];
              unsigned hits = 0;
              const int32_t n = (end - r) & ~63;
              r += n;
              if (sslot >= 0) {
                const int16_t* hs = slots_beside(g, it, T, T_hm);
                for (int32_t i = 0; i < n; i += 64) {
                  const int32_t x0 = __ldg(it + i), x1 = __ldg(it + i + 32);
                  int32_t s0, s1;
                  if (hs != nullptr) {
                    s0 = __ldg(hs + i);
                    s1 = __ldg(hs + i + 32);
                  } else {
                    s0 = __ldg(g.hm_slot + x0);
                    s1 = __ldg(g.hm_slot + x1);
                  }
                  const Probe p0 = probe_begin<true>(g, sslot, sbm, sl, slen, x0, s0);
                  const Probe p1 = probe_begin<true>(g, sslot, sbm, sl, slen, x1, s1);
                  hits += probe_end(p0, sl, slen, x0);
                  hits += probe_end(p1, sl, slen, x1);
                }
              } else {
                for (int32_t i = 0; i < n; i += 64) {
                  const int32_t x0 = __ldg(it + i), x1 = __ldg(it + i + 32);
                  const Probe p0 = probe_begin<false>(g, sslot, sbm, sl, slen, x0, -1);
                  const Probe p1 = probe_begin<false>(g, sslot, sbm, sl, slen, x1, -1);
                  hits += probe_end(p0, sl, slen, x0);
                  hits += probe_end(p1, sl, slen, x1);
                }
              }
              hits = __reduce_add_sync(kFull, hits);
              if (lane == j0) {
                if (sg) acc_b += hits;
                else acc_a += hits;
              }
              continue;
            }
          }
          // item starts among the next 64 tests: bit b of m0 / m1 = test r + b
          // / r + 32 + b begins an item (items have tests, so starts differ)
          const int32_t ds = srel - r;
          const unsigned m0 = __reduce_or_sync(kFull, ds > 0 && ds < 32 ? 1u << ds : 0u);
          const unsigned m1 =
              __reduce_or_sync(kFull, ds >= 32 && ds < 64 ? 1u << (ds - 32) : 0u);
          int j[2], seg[2];
          int32_t x[2], xs[2];
          bool act[2];
          j[0] = min(j0 + __popc(m0 & upto), 31);
          j[1] = min(j0 + __popc(m0) + __popc(m1 & upto), 31);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int32_t rr = r + 32 * h + lane;
            const int32_t bj = __shfl_sync(kFull, sb, j[h]);
            int32_t o = rr - __shfl_sync(kFull, srel, j[h]);
            act[h] = rr < len;
            seg[h] = 0;
            x[h] = 0;
            xs[h] = -1;
            if (act[h]) {
              if (rr >= bj) {
                seg[h] = 1;
                o = rr - bj;
              }
              const int32_t* it = my->it[seg[h]][j[h]] + o;
              x[h] = __ldg(it);
              if (my->sslot[seg[h]][j[h]] >= 0) {
                const int16_t* hs = slots_beside(g, it, T, T_hm);
                xs[h] = hs != nullptr ? (int32_t)__ldg(hs) : __ldg(g.hm_slot + x[h]);
              }
            }
          }
          Probe p[2];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (act[h])
              p[h] = probe_begin<true>(g, my->sslot[seg[h]][j[h]], my->sbm[seg[h]][j[h]],
                                       my->sl[seg[h]][j[h]], my->slen[seg[h]][j[h]], x[h], xs[h]);
          unsigned hit[2];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            hit[h] = __ballot_sync(
                kFull,
                act[h] && probe_end(p[h], my->sl[seg[h]][j[h]], my->slen[seg[h]][j[h]], x[h]));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int32_t rh = r + 32 * h;
            const unsigned below_b = bits_below(sb - rh);
            acc_a += __popc(hit[h] & below_b & ~bits_below(srel - rh));
            acc_b += __popc(hit[h] & bits_below(se - rh) & ~below_b);
          }
          r += 64;
        }
      }
      // the lanes' counts to their edges: one addition when the pack lies in
      // one edge
      long long dq = 0;
      if (lane < live)
        dq = (need_q ? 2 * (long long)acc_a : 0) + (long long)my->bsign[lane] * (long long)acc_b;
      const int64_t e_last = __shfl_sync(kFull, e, live - 1);
      if (e_last == e0) {
        acc_a = warp_sum<unsigned long long>(acc_a);
        dq = warp_sum<long long>(dq);
        if (lane != 0) acc_a = 0, dq = 0;
      }
      if (acc_a) atomicAdd(k_out + e, acc_a);
      if (dq) atomicAdd(q + e, (unsigned long long)dq);
    }
  }
}

// ---------------------------------------------------------------- fold

typedef unsigned __int128 u128;
typedef __int128 i128;

__device__ __forceinline__ u128 shfl_down_u128(u128 v, int o) {
  unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
  lo = __shfl_down_sync(kFull, lo, o);
  hi = __shfl_down_sync(kFull, hi, o);
  return ((u128)hi << 64) | lo;
}

// Per-edge numerators (order 3,4,7,8,9,10,11,12) and 128-bit block sums:
// part[block][0..7] = sum N_i (two's complement), part[block][8..15] = sum N_i^2.
__global__ void __launch_bounds__(kThreads)
    k_fold(DevGraph g, const int2* __restrict__ uv, int64_t K,
           const unsigned long long* __restrict__ t, const unsigned long long* __restrict__ k2,
           const unsigned long long* __restrict__ q, const int64_t* __restrict__ tdeg,
           const int64_t* __restrict__ nbr_degsum, int need_k, int need_q,
           int64_t* __restrict__ per_edge, u128* __restrict__ part,
           unsigned long long* __restrict__ stats) {
  u128 acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0;
  unsigned long long tri_tests = 0, model = 0, model4 = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < K;
       e += (int64_t)gridDim.x * blockDim.x) {
    int2 pr = uv[e];
    int64_t bu, bv;
    const i128 du = deg_of(g.row_ptr, pr.x, &bu), dv = deg_of(g.row_ptr, pr.y, &bv);
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
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      acc[i] += (u128)N[i];
      u128 m = (u128)(N[i] < 0 ? -N[i] : N[i]);
      acc[8 + i] += m * m;
    }
    // streaming cost model B(e) of Algorithms 2-4 (statistics only)
    tri_tests += (unsigned long long)du;
    model += 24 + 4 * (unsigned long long)(du + dv);
    if (tdeg != nullptr) {
      const long long td = tdeg[e];
      unsigned long long B4 = 0;
      if (need_k) B4 += 8 * (unsigned long long)tt + 4 * (unsigned long long)td;
      if (need_q) {
        long long su = (long long)(8 * a) + 4 * (nbr_degsum[pr.x] - (long long)dv - td);
        long long sv = (long long)(8 * b) + 4 * (nbr_degsum[pr.y] - (long long)du - td);
        B4 += (unsigned long long)(su < sv ? su : sv);
      }
      model4 += B4;
    }
    if (per_edge != nullptr) {
      per_edge[3 * e] = (int64_t)tt;
      per_edge[3 * e + 1] = (int64_t)kk;
      per_edge[3 * e + 2] = (int64_t)qq;
    }
  }
  __shared__ u128 red[kThreads / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    u128 v = acc[i];
    for (int o = 16; o > 0; o >>= 1) v += shfl_down_u128(v, o);
    if (lane == 0) red[warp][i] = v;
  }
  tri_tests = warp_sum<unsigned long long>(tri_tests);
  model = warp_sum<unsigned long long>(model);
  model4 = warp_sum<unsigned long long>(model4);
  if (lane == 0) {
    atomicAdd(stats + 0, tri_tests);
    atomicAdd(stats + 2, model);
    if (model4) atomicAdd(stats + 3, model4);
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    u128 s = 0;
    for (int w = 0; w < kThreads / 32; ++w) s += red[w][threadIdx.x];
    part[(int64_t)blockIdx.x * 16 + threadIdx.x] = s;
  }
}

// Sums of the block partials, a warp per value (one thread per value walked
// hundreds of dependent loads: 12 to 40 us; exact integers, any order).
__global__ void __launch_bounds__(512) k_fold_final(const u128* __restrict__ part, int blocks,
                                                    unsigned long long* __restrict__ out) {
  const int lane = threadIdx.x & 31, value = threadIdx.x >> 5;
  u128 s = 0;
  for (int b = lane; b < blocks; b += 32) s += part[(int64_t)b * 16 + value];
  for (int o = 16; o > 0; o >>= 1) s += shfl_down_u128(s, o);
  if (lane == 0) {
    out[2 * value] = (unsigned long long)s;
    out[2 * value + 1] = (unsigned long long)(s >> 64);
  }
}


// Per-segment exact sums. Edges [seg_off[s], seg_off[s+1]) form segment s
// (one graph of a batch, one request of a serving step). Each of the 16
// values (8 sums in two's complement, 8 sums of squares) is accumulated as
// four 32-bit limbs in 64-bit counters: a limb sum stays below 2^64 for
// fewer than 2^32 additions, so the 128-bit total is recovered exactly.
// Lanes of a warp are reduced per segment first (segmented shuffle scan).
__global__ void __launch_bounds__(kThreads)
    k_fold_seg(DevGraph g, const int2* __restrict__ uv, int64_t K,
               const unsigned long long* __restrict__ t, const unsigned long long* __restrict__ k2,
               const unsigned long long* __restrict__ q, const int64_t* __restrict__ seg_off,
               int64_t nseg, unsigned long long* __restrict__ limbs) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < K;
       base += stride) {
    const int64_t e = base + lane;
    int64_t seg = -1;
    u128 val[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) val[i] = 0;
    if (e < K) {
      seg = last_le(seg_off, nseg, e);
      int2 pr = uv[e];
      int64_t bu, bv;
      const i128 du = deg_of(g.row_ptr, pr.x, &bu), dv = deg_of(g.row_ptr, pr.y, &bv);
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
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        val[i] = (u128)N[i];
        u128 m = (u128)(N[i] < 0 ? -N[i] : N[i]);
        val[8 + i] = m * m;
      }
    }
    // segmented inclusive scan over the warp (segments are contiguous)
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int64_t sd = __shfl_up_sync(kFull, seg, d);
      const bool take = lane >= d && sd == seg;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        unsigned long long lo = __shfl_up_sync(kFull, (unsigned long long)val[i], d);
        unsigned long long hi = __shfl_up_sync(kFull, (unsigned long long)(val[i] >> 64), d);
        if (take) val[i] += ((u128)hi << 64) | lo;
      }
    }
    const int64_t next = __shfl_down_sync(kFull, seg, 1);
    const bool tail = seg >= 0 && (lane == 31 || next != seg);
    if (tail) {
      unsigned long long* dst = limbs + seg * 64;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          const unsigned long long limb = (unsigned long long)((val[i] >> (32 * l)) & 0xffffffffu);
          if (limb) atomicAdd(dst + i * 4 + l, limb);
        }
      }
    }
  }
}

// Recombines the limbs: sums[s][i] = sum_l limb_l << 32 l (mod 2^128), as
// (low, high) 64-bit words.
__global__ void k_fold_seg_final(const unsigned long long* __restrict__ limbs, int64_t nseg,
                                 unsigned long long* __restrict__ sums) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < nseg * 16;
       x += (int64_t)gridDim.x * blockDim.x) {
    u128 s = 0;
#pragma unroll
    for (int l = 0; l < 4; ++l) s += (u128)limbs[x * 4 + l] << (32 * l);
    sums[2 * x] = (unsigned long long)s;
    sums[2 * x + 1] = (unsigned long long)(s >> 64);
  }
}

}  // namespace gs

// =================================================================== host side
namespace gs {

// 8 triangle-pass CTAs per SM (k_tri, 32 registers; k_tri_chunks takes at most
// kTriBlocksPerSm) and tasks of 512 tests.
Tuning default_tuning() { return Tuning{8, kQuadBlocksPerSm, 512, 1, kHubDenseSlots}; }

int quad_blocks_limit() { return kQuadBlocksPerSm; }

DevGraph graph_view(const gs_graph* gr, const Tuning& tu) {
  DevGraph g = gr->dev;
  g.hm_dense_words =
      g.hm_bits != nullptr ? std::min(g.hm_words, std::max<int64_t>(tu.dense_slots, 0) / 128 * 4)
                           : 0;
  if (!tu.use_hubs) {
    g.bm_slot = nullptr;
    g.bm_bits = nullptr;
    g.bm_count = 0;
    g.tb_slot = nullptr;
    g.tb_codeg = nullptr;
    g.tb_giant = nullptr;
    g.tb_count = 0;
    g.hm_slot = nullptr;
    g.hm_bits = nullptr;
    g.col_hm = nullptr;
    g.mn_ptr = nullptr;
    g.mn_slot = nullptr;
    g.nm_ptr = nullptr;
    g.nm_col = nullptr;
    g.hm_vertex = nullptr;
    g.bg_slot = nullptr;
    g.md_codeg = nullptr;
    g.dir_at = nullptr;
    g.dir = nullptr;
    g.col_tb = nullptr;
    g.cg = nullptr;
    g.cg_row = nullptr;
  }
  return g;
}

size_t count_front_bytes(int64_t K, bool all_edges, bool check_dup, int64_t nseg) {
  int64_t dup_cap = 1;
  while (dup_cap < 2 * K) dup_cap <<= 1;
  const int fold_blocks = grid_for(K, kThreads, 2);
  return Carve::bytes_for<DevError>(1) + Carve::bytes_for<unsigned long long>(32) +
         Carve::bytes_for<unsigned long long>(kStatSlots) +
         (all_edges ? Carve::bytes_for<int32_t>(2 * K) : 0) + Carve::bytes_for<int2>(K) +
         Carve::bytes_for<int64_t>(K + 1) * 2 + Carve::bytes_for<unsigned long long>(K) * 3 +
         Carve::bytes_for<int64_t>(K) + Carve::bytes_for<int32_t>(K) +
         Carve::bytes_for<int64_t>(scan_tmp_elems(K + 1)) +
         (check_dup ? Carve::bytes_for<unsigned long long>(dup_cap) : 0) +
         Carve::bytes_for<u128>((int64_t)fold_blocks * 16) +
         (nseg > 0 ? Carve::bytes_for<unsigned long long>(nseg * 64) +
                         Carve::bytes_for<unsigned long long>(nseg * 32)
                   : 0);
}

void carve_front(void* base, int64_t K, bool all_edges, bool check_dup, int64_t nseg,
                 CountBufs& b) {
  Carve c{(char*)base, 0};
  int64_t dup_cap = 1;
  while (dup_cap < 2 * K) dup_cap <<= 1;
  b.K = K;
  b.dup_cap = dup_cap;
  b.fold_blocks = grid_for(K, kThreads, 2);
  b.err = c.take<DevError>(1);
  b.sums = c.take<unsigned long long>(32);
  b.stats = c.take<unsigned long long>(kStatSlots);
  b.pairs_all = all_edges ? c.take<int32_t>(2 * K) : nullptr;
  b.uv = c.take<int2>(K);
  b.off = c.take<int64_t>(K + 1);
  b.toff = c.take<int64_t>(K + 1);
  b.t = c.take<unsigned long long>(K);
  b.k2 = c.take<unsigned long long>(K);
  b.q = c.take<unsigned long long>(K);
  b.tdeg = c.take<int64_t>(K);
  b.mask_idx = c.take<int32_t>(K);
  b.tmp0 = c.take<int64_t>(scan_tmp_elems(K + 1));
  b.dup = check_dup ? c.take<unsigned long long>(dup_cap) : nullptr;
  b.part = c.take<u128>((int64_t)b.fold_blocks * 16);
  b.nseg = nseg;
  b.limbs = nseg > 0 ? c.take<unsigned long long>(nseg * 64) : nullptr;
  b.seg_sums = nseg > 0 ? c.take<unsigned long long>(nseg * 32) : nullptr;
}

size_t count_mid_bytes(int64_t P) {
  const int64_t groups = (P + 31) / 32;
  return Carve::bytes_for<uint32_t>(groups) + Carve::bytes_for<int32_t>(groups) +
         Carve::bytes_for<uint32_t>(2 * groups) +
         Carve::bytes_for<int64_t>(groups + 1) +
         Carve::bytes_for<int64_t>(scan_tmp_elems(groups + 1));
}

void carve_mid(void* base, int64_t P, CountBufs& b) {
  Carve c{(char*)base, 0};
  b.P = P;
  b.groups = (P + 31) / 32;
  b.tbits = c.take<uint32_t>(b.groups);
  b.tpre = c.take<int32_t>(b.groups);
  b.cbits = c.take<uint32_t>(2 * b.groups);
  b.task_off = c.take<int64_t>(b.groups + 1);
  b.tmp1 = c.take<int64_t>(scan_tmp_elems(b.groups + 1));
}

// Bytes from b.err to the end of b.stats.
constexpr size_t kFrontWords = 512 + sizeof(unsigned long long) * kStatSlots;

// memsets + (all-pair enumeration) + prep + position scan. No host sync.
int64_t launch_front(const gs_graph* gr, const DevGraph& g, const int32_t* pairs, bool four,
                     CountBufs& b, cudaStream_t stream) {
  int64_t launches = 0;
  const int64_t K = b.K;
  // err, sums and stats in one fill; t, k2 and q (carved one behind the other)
  // in another
  cudaMemsetAsync(b.err, 0, kFrontWords, stream);
  cudaMemsetAsync(b.t, 0,
                  four ? (size_t)((char*)(b.q + K) - (char*)b.t) : sizeof(unsigned long long) * K,
                  stream);
  if (b.dup != nullptr) cudaMemsetAsync(b.dup, 0xff, sizeof(unsigned long long) * b.dup_cap, stream);
  if (pairs == nullptr) {
    k_all_pairs<<<grid_for(g.n * 32, kThreads, 8), kThreads, 0, stream>>>(
        g.row_ptr, g.col, gr->up_ptr, gr->edge_off, g.n, b.pairs_all);
    pairs = b.pairs_all;
    ++launches;
  }
  k_prep<<<grid_for(K, kThreads, 8), kThreads, 0, stream>>>(g, pairs, K, four ? 1 : 0, b.dup,
                                                            b.dup_cap - 1, b.uv, b.off, b.err);
  exclusive_scan_i64(b.off, b.off, K, b.tmp0, stream);
  return launches + 1 + scan_launches(K);
}

int64_t launch_tri(const DevGraph& g, bool four, const Tuning& tu, CountBufs& b,
                   cudaStream_t stream) {
  const int sms = sm_count(), grid = sms * tu.tri_blocks_per_sm;
  // no more CTAs than are resident: a small call gives each of their warps a run
  const int chunk_grid = sms * std::min(tu.tri_blocks_per_sm, kTriBlocksPerSm);
  if (four) {
    k_tri_chunks<<<chunk_grid, kThreads, 0, stream>>>(g, b.uv, b.off, b.K, b.t, b.tbits,
                                                      b.stats + 10);
  } else if (b.P >= kManyPositions && b.P >= kLongLists * b.K) {
    // toff is free in 3-node work: the padded offsets
    k_pad_lengths<<<grid_for(b.K, kThreads, 8), kThreads, 0, stream>>>(b.off, b.K, b.toff);
    exclusive_scan_i64(b.toff, b.toff, b.K, b.tmp0, stream);
    k_tri_chunks<<<chunk_grid, kThreads, 0, stream>>>(g, b.uv, b.toff, b.K, b.t, nullptr,
                                                      b.stats + 10);
    return 2 + scan_launches(b.K);
  } else {
    k_tri<<<grid, kThreads, 0, stream>>>(g, b.uv, b.off, b.K, b.t);
  }
  return 1;
}

int64_t launch_scan_t(CountBufs& b, cudaStream_t stream) {
  exclusive_scan_i64((const int64_t*)b.t, b.toff, b.K, b.tmp0, stream);
  return scan_launches(b.K);
}

// T lists (and their matrix slots) in order; marks dense edges (mask index
// from the counter stats[6]). T must hold b.toff[K] entries. No host sync.
int64_t launch_compact(const DevGraph& g, CountBufs& b, cudaStream_t stream) {
  int16_t* T_hm = g.col_hm != nullptr ? b.T_hm : nullptr;
  const int64_t long_list = compact_long(b.K);
  if (long_list == INT64_MAX)
    k_compact_T<false><<<grid_for(b.K * 32, kThreads, 8), kThreads, 0, stream>>>(
        g, b.uv, b.off, b.toff, b.K, b.tbits, b.T, b.tpre, T_hm, b.tdeg, b.mask_idx, b.stats + 6,
        long_list);
  else
    k_compact_T<true><<<grid_for(b.K * kThreads, kThreads, 8), kThreads, 0, stream>>>(
        g, b.uv, b.off, b.toff, b.K, b.tbits, b.T, b.tpre, T_hm, b.tdeg, b.mask_idx, b.stats + 6,
        long_list);
  return 1;
}

// T masks of the dense edges (b.ndense of them). No host sync.
int64_t launch_tmask(const DevGraph& g, CountBufs& b, cudaStream_t stream) {
  if (b.ndense <= 0 || g.col_hm == nullptr) return 0;
  k_build_tmask<<<grid_for(b.K * 32, kThreads, 8), kThreads, 0, stream>>>(
      b.toff, b.t, b.T_hm, b.mask_idx, b.K, g.hm_dense_words, b.tmask, b.dense_e, b.unit_off);
  exclusive_scan_i64(b.unit_off, b.unit_off, b.ndense, b.unit_tmp, stream);
  k_unit_fill<<<grid_for(b.ndense * 32, kThreads, 8), kThreads, 0, stream>>>(b.unit_off, b.ndense,
                                                                              b.unit_idx);
  return 2 + scan_launches(b.ndense);
}

// Pairs among the matrix members of T in the dense edges (k_dense_pairs).
// No host sync.
int64_t launch_dense(const DevGraph& g, bool need_q, CountBufs& b, cudaStream_t stream) {
  if (b.ndense <= 0 || g.col_hm == nullptr) return 0;
  auto go = [&](auto kernel, int threads) {
    kernel<<<sm_count() * (kDenseWarpsPerSm * 32 / threads), threads, 0, stream>>>(
        g, b.toff, b.t, b.T, b.T_hm, b.tmask, b.dense_e, b.unit_off, b.unit_idx, b.ndense,
        need_q ? 1 : 0, b.k2, b.q, b.stats + 7, b.stats + 4, b.stats + 9);
  };
  const int64_t resident = (int64_t)sm_count() * (kDenseWarpsPerSm * 32 / 256);
  if (b.ndense >= kManyDensePerCta * resident &&
      (double)g.mn_total >= kSmallCtaShare * (double)g.nnz)
    go(k_dense_pairs<128>, 128);
  else go(k_dense_pairs<256>, 256);
  return 1;
}

// Chunk costs and the task scan. No host sync.
int64_t launch_cost(const DevGraph& g, bool need_k, bool need_q, const Tuning& tu, CountBufs& b,
                    cudaStream_t stream) {
  (void)need_k;  // every item's segment A feeds both k and q
  const int32_t* mi = g.col_hm != nullptr ? b.mask_idx : nullptr;
  k_chunk_cost<<<sm_count() * kCostBlocksPerSm, kThreads, 0, stream>>>(
      g, b.uv, b.off, b.K, b.t, b.tbits, b.tpre, mi, need_q, tu.task_probes, b.task_off, b.cbits,
      b.q, b.stats);
  exclusive_scan_i64(b.task_off, b.task_off, b.groups, b.tmp1, stream);
  return 1 + scan_launches(b.groups);
}

// The 4-node membership tests (k_quad). No host sync.
int64_t launch_quad(const DevGraph& g, bool need_k, bool need_q, const Tuning& tu, CountBufs& b,
                    cudaStream_t stream) {
  const int sms = sm_count();
  const int qb = tu.quad_blocks_per_sm < 1 ? 1
                 : tu.quad_blocks_per_sm > kQuadBlocksPerSm ? kQuadBlocksPerSm
                                                            : tu.quad_blocks_per_sm;
  k_quad<<<sms * qb, kThreads, 0, stream>>>(g, b.uv, b.off, b.K, b.t, b.toff, b.tbits, b.tpre,
                                            b.cbits, b.T,
                                            g.col_hm != nullptr ? b.T_hm : nullptr,
                                            g.col_hm != nullptr ? b.mask_idx : nullptr, b.tmask,
                                            b.task_off, b.groups, need_k, need_q,
                                            tu.task_probes, b.k2, b.q, b.stats + 5);
  return 1;
}

int64_t launch_fold(const gs_graph* gr, const DevGraph& g, bool four, bool need_k, bool need_q,
                    int64_t* per_edge, CountBufs& b, cudaStream_t stream) {
  k_fold<<<b.fold_blocks, kThreads, 0, stream>>>(g, b.uv, b.K, b.t, four ? b.k2 : nullptr,
                                                  four ? b.q : nullptr, four ? b.tdeg : nullptr,
                                                  gr->nbr_degsum, need_k, need_q, per_edge, b.part,
                                                  b.stats);
  k_fold_final<<<1, 512, 0, stream>>>(b.part, b.fold_blocks, b.sums);
  return 2;
}

int64_t launch_fold_seg(const DevGraph& g, bool four, const int64_t* seg_off, CountBufs& b,
                        cudaStream_t stream) {
  cudaMemsetAsync(b.limbs, 0, sizeof(unsigned long long) * b.nseg * 64, stream);
  k_fold_seg<<<grid_for(b.K, kThreads, 4), kThreads, 0, stream>>>(
      g, b.uv, b.K, b.t, four ? b.k2 : nullptr, four ? b.q : nullptr, seg_off, b.nseg, b.limbs);
  k_fold_seg_final<<<grid_for(b.nseg * 16, 256, 4), 256, 0, stream>>>(b.limbs, b.nseg,
                                                                       b.seg_sums);
  return 2;
}

static gs_status error_status(const DevError& h, const char* what) {
  if (h.code != 0) {
    const char* kind = h.code == GS_EDUPSAMPLE ? "edge sampled twice"
                       : h.code == GS_EEDGE    ? "sampled pair is out of range or not an edge"
                                               : "invalid input";
    set_error("%s: %s (pair %lld)", what, kind, (long long)h.index);
    return h.code;
  }
  return GS_OK;
}

gs_status fetch_error(DevError* d_err, cudaStream_t stream, const char* what) {
  DevError h;
  GS_CUDA(cudaMemcpyAsync(&h, d_err, sizeof(h), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  return error_status(h, what);
}

void store_sums(const unsigned long long* h, uint32_t mask, gs_sums* out) {
  static const uint32_t bit[8] = {GS_G3, GS_G4, GS_G7, GS_G8, GS_G9, GS_G10, GS_G11, GS_G12};
  for (int i = 0; i < 8; ++i) {
    if (!(mask & bit[i])) continue;
    out->sum[i][0] = h[2 * i];
    out->sum[i][1] = h[2 * i + 1];
    out->sumsq[i][0] = h[2 * (8 + i)];
    out->sumsq[i][1] = h[2 * (8 + i) + 1];
  }
}

// Up to this many positions the T lists (6 bytes an entry) get room for every
// position instead of a wait for their size.
constexpr int64_t kSmallPositions = 1 << 20;

// Full counting run with host synchronisation for sizing (gs_count and the
// sizing pass of the batched and served paths). seg_off != NULL selects the
// per-segment fold (results in b.seg_sums) instead of the single sum.
gs_status count_run(const gs_graph* gr, gs_workspace* ws, const int32_t* d_pairs, int64_t K,
                    uint32_t mask, bool check_dup, int64_t* d_per_edge, const int64_t* seg_off,
                    int64_t nseg, const Tuning& tu, CountBufs& b, cudaStream_t stream,
                    const char* what) {
  const bool need_k = (mask & (GS_G7 | GS_G8 | GS_G9 | GS_G11)) != 0;
  const bool need_q = (mask & (GS_G10 | GS_G12)) != 0;
  const bool four = need_k || need_q;
  const bool all_edges = d_pairs == nullptr;
  const DevGraph g = graph_view(gr, tu);
  int64_t launches = 0;
  struct Timer {
    gs_workspace* ws;
    cudaStream_t s;
    void start(int p) {
      if (ws->timing) cudaEventRecord(ws->ev[2 * p], s);
    }
    void stop(int p) {
      if (ws->timing) cudaEventRecord(ws->ev[2 * p + 1], s);
    }
  } timer{ws, stream};

  void* base0 = nullptr;
  GS_TRY(ws_reserve(ws, 0, count_front_bytes(K, all_edges, check_dup, seg_off ? nseg : 0), stream,
                    &base0));
  carve_front(base0, K, all_edges, check_dup, seg_off ? nseg : 0, b);
  timer.start(0);
  launches += launch_front(gr, g, d_pairs, four, b, stream);
  timer.stop(0);
  GS_CUDA(cudaGetLastError());
  void* staged = nullptr;
  GS_TRY(ws_staging(ws, &staged));
  DevError* h_err = (DevError*)staged;
  int64_t* h_val = (int64_t*)((char*)staged + 256);
  GS_CUDA(cudaMemcpyAsync(h_val, b.off + K, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaMemcpyAsync(h_err, b.err, sizeof(DevError), cudaMemcpyDeviceToHost, stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  const int64_t P = *h_val;
  ws->launches_total += launches;
  const gs_status es = error_status(*h_err, what);
  if (es != GS_OK) return es;

  void* base1 = nullptr;
  GS_TRY(ws_reserve(ws, 1, four ? count_mid_bytes(P) : 256, stream, &base1));
  if (four) {
    carve_mid(base1, P, b);
  } else {
    b.P = P;
    b.groups = (P + 31) / 32;
    b.tbits = nullptr;
  }
  int64_t more = 0;
  timer.start(1);
  more += launch_tri(g, four, tu, b, stream);
  timer.stop(1);
  GS_CUDA(cudaGetLastError());
  b.tsum = 0;
  if (four) {
    timer.start(2);
    more += launch_scan_t(b, stream);
    if (P <= kSmallPositions) {
      b.tsum = P;  // every T entry is a position: room for all, and no wait
    } else {
      GS_CUDA(
          cudaMemcpyAsync(h_val, b.toff + K, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
      GS_CUDA(cudaStreamSynchronize(stream));
      b.tsum = *h_val;
    }
    void* base2 = nullptr;
    GS_TRY(ws_reserve(ws, 2,
                      Carve::bytes_for<int32_t>(b.tsum) + Carve::bytes_for<int16_t>(b.tsum),
                      stream, &base2));
    Carve c2{(char*)base2, 0};
    b.T = c2.take<int32_t>(b.tsum);
    b.T_hm = c2.take<int16_t>(b.tsum);
    more += launch_compact(g, b, stream);
    b.ndense = 0;
    if (g.col_hm != nullptr && g.hm_dense_words > 0) {  // without a matrix no edge is dense
      GS_CUDA(cudaMemcpyAsync(h_val, b.stats + 6, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
      GS_CUDA(cudaStreamSynchronize(stream));
      b.ndense = *h_val;
    }
    b.tmask = nullptr;
    b.dense_e = nullptr;
    if (b.ndense > 0) {
      void* base4 = nullptr;
      GS_TRY(ws_reserve(ws, 4,
                        Carve::bytes_for<uint32_t>(b.ndense * g.hm_dense_words) +
                            Carve::bytes_for<int64_t>(b.ndense) +
                            Carve::bytes_for<int64_t>(b.ndense + 1) +
                            Carve::bytes_for<int64_t>(scan_tmp_elems(b.ndense + 1)) +
                            Carve::bytes_for<int32_t>(b.tsum / kDenseUnit + b.ndense),
                        stream, &base4));
      Carve c4{(char*)base4, 0};
      b.tmask = c4.take<uint32_t>(b.ndense * g.hm_dense_words);
      b.dense_e = c4.take<int64_t>(b.ndense);
      b.unit_off = c4.take<int64_t>(b.ndense + 1);
      b.unit_tmp = c4.take<int64_t>(scan_tmp_elems(b.ndense + 1));
      // units of an edge: ceil(t / kDenseUnit) <= t / kDenseUnit + 1
      b.unit_idx = c4.take<int32_t>(b.tsum / kDenseUnit + b.ndense);
    }
    timer.stop(2);
    timer.start(3);
    more += launch_tmask(g, b, stream);
    more += launch_cost(g, need_k, need_q, tu, b, stream);
    timer.stop(3);
    timer.start(4);
    more += launch_quad(g, need_k, need_q, tu, b, stream);
    more += launch_dense(g, need_q, b, stream);
    timer.stop(4);
    GS_CUDA(cudaGetLastError());
  } else {
    for (int ph = 2; ph <= 4; ++ph) {
      timer.start(ph);
      timer.stop(ph);
    }
  }
  timer.start(5);
  if (seg_off != nullptr)
    more += launch_fold_seg(g, four, seg_off, b, stream);
  else
    more += launch_fold(gr, g, four, need_k, need_q, d_per_edge, b, stream);
  timer.stop(5);
  GS_CUDA(cudaGetLastError());
  ws->launches_total += more;
  ws->stats.launches = launches + more;
  return GS_OK;
}

}  // namespace gs

// =================================================================== C ABI
using namespace gs;

static const uint32_t kKnownMask = GS_CONNECTED;

extern "C" gs_status gs_count(const gs_graph* gr, gs_workspace* ws, const int32_t* d_pairs,
                              int64_t K, uint32_t mask, int64_t* d_per_edge, gs_sums* h_sums,
                              void* stream_) {
  cudaStream_t stream = (cudaStream_t)stream_;
  if (gr == nullptr || ws == nullptr || h_sums == nullptr || K < 0 || mask == 0 ||
      (mask & ~kKnownMask) != 0) {
    set_error("gs_count: invalid arguments (mask must be a non-empty subset of GS_CONNECTED)");
    return GS_EINVAL;
  }
  memset(h_sums, 0, sizeof(*h_sums));
  h_sums->k = K;
  h_sums->m = gr->m;
  h_sums->mask = mask;
  memset(&ws->stats, 0, sizeof(ws->stats));
  ws->stats.k = K;
  if (K == 0) return GS_OK;  // empty sample (d_pairs is not read)
  if (d_pairs == nullptr && K != gr->m) {
    set_error("gs_count: with d_pairs = NULL, k must equal the edge count %lld", (long long)gr->m);
    return GS_EINVAL;
  }
  const Tuning tu = ws->has_tuning ? ws->tuning : default_tuning();
  if (d_pairs == nullptr && d_per_edge == nullptr && (mask & ~(uint32_t)GS_THREE_NODE) == 0 &&
      gr->out_col != nullptr && tu.use_hubs) {
    // every edge, triangles and 2-stars only: triangles listed once through
    // the oriented lists (same per-edge t, sums independent of the order)
    unsigned long long h[32], hs[8];
    int64_t nl = 0;
    GS_TRY(count_tri_oriented(gr, ws, h, hs, &nl, stream));
    store_sums(h, mask, h_sums);
    gs_stats& st = ws->stats;
    st.k = K;
    st.tri_tests = (int64_t)hs[0];
    st.model_bytes = hs[2];
    st.model_tri_bytes = hs[2];
    st.launches = nl;
    ws->launches_total += nl;
    st.timed = ws->timing;
    if (ws->timing) {
      float* ms[6] = {&st.ms_prep, &st.ms_tri, &st.ms_compact, &st.ms_cost, &st.ms_quad,
                      &st.ms_fold};
      for (int ph = 0; ph < 6; ++ph)
        cudaEventElapsedTime(ms[ph], ws->ev[2 * ph], ws->ev[2 * ph + 1]);
    }
    return GS_OK;
  }
  CountBufs b;
  GS_TRY(count_run(gr, ws, d_pairs, K, mask, d_pairs != nullptr, d_per_edge, nullptr, 0, tu, b,
                   stream, "gs_count"));
  const bool four = (mask & (GS_G7 | GS_G8 | GS_G9 | GS_G10 | GS_G11 | GS_G12)) != 0;
  void* staged = nullptr;
  GS_TRY(ws_staging(ws, &staged));
  // err (unused here), sums and stats, then the task and T totals
  unsigned long long* h = (unsigned long long*)((char*)staged + 256);
  unsigned long long* hs = (unsigned long long*)((char*)staged + 512);
  int64_t* h_val = (int64_t*)((char*)staged + kFrontWords);
  h_val[0] = h_val[1] = 0;
  GS_CUDA(cudaMemcpyAsync(staged, b.err, kFrontWords, cudaMemcpyDeviceToHost, stream));
  if (four) {
    GS_CUDA(cudaMemcpyAsync(h_val, b.task_off + b.groups, sizeof(int64_t), cudaMemcpyDeviceToHost,
                            stream));
    GS_CUDA(cudaMemcpyAsync(h_val + 1, b.toff + K, sizeof(int64_t), cudaMemcpyDeviceToHost,
                            stream));
  }
  GS_CUDA(cudaStreamSynchronize(stream));
  const int64_t ntasks = h_val[0];
  store_sums(h, mask, h_sums);
  gs_stats& st = ws->stats;
  st.k = K;
  st.tri_tests = (int64_t)hs[0];
  st.dense_edges = (int64_t)hs[6];
  st.quad_tests = (int64_t)(hs[1] + hs[4] + hs[9]);
  st.dense_groups = (int64_t)hs[4];
  st.model_bytes = hs[2] + hs[3];
  st.model_tri_bytes = hs[2];
  st.model_quad_bytes = hs[3];
  st.t_sum = h_val[1];
  st.tasks = ntasks;
  st.timed = ws->timing;
  if (ws->timing) {
    float* ms[6] = {&st.ms_prep, &st.ms_tri, &st.ms_compact, &st.ms_cost, &st.ms_quad, &st.ms_fold};
    for (int ph = 0; ph < 6; ++ph) cudaEventElapsedTime(ms[ph], ws->ev[2 * ph], ws->ev[2 * ph + 1]);
  }
  return GS_OK;
}

extern "C" gs_status gs_workspace_set_tuning(gs_workspace* ws, int tri_blocks_per_sm,
                                             int quad_blocks_per_sm, int64_t task_probes,
                                             int use_hubs) {
  if (ws == nullptr || tri_blocks_per_sm < 1 || tri_blocks_per_sm > 8 || quad_blocks_per_sm < 1 ||
      quad_blocks_per_sm > kQuadBlocksPerSm || task_probes < 32 || task_probes > (1 << 20)) {
    set_error("gs_workspace_set_tuning: out-of-range parameter (tri 1..8, quad 1..%d, task "
              "32..2^20)",
              kQuadBlocksPerSm);
    return GS_EINVAL;
  }
  const int64_t ds = ws->has_tuning ? ws->tuning.dense_slots : kHubDenseSlots;
  ws->tuning = Tuning{tri_blocks_per_sm, quad_blocks_per_sm, task_probes, use_hubs ? 1 : 0, ds};
  ws->has_tuning = 1;
  return GS_OK;
}

extern "C" gs_status gs_workspace_set_dense_slots(gs_workspace* ws, int64_t slots) {
  if (ws == nullptr || slots < 0) {
    set_error("gs_workspace_set_dense_slots: null workspace or negative slot count");
    return GS_EINVAL;
  }
  if (!ws->has_tuning) ws->tuning = default_tuning();
  ws->tuning.dense_slots = slots;
  ws->has_tuning = 1;
  return GS_OK;
}
