// Exact triangle counts of every edge for the 3-node pass over all edges
// (gs_count with J = E, mask within G3 | G4, no per-edge output).
//
// Algorithm 2 gives every edge e its t = |N(u) cap N(v)|; over all edges
// the same integers follow from listing every triangle once. Edges are
// oriented from the lower to the higher (degree, id) endpoint, so out-lists
// N+(x) are short (at most about sqrt(2M) long; 1,761 on R-MAT scale 24).
// A triangle {u, v, x} with u < v < x in that order is found once: at the
// oriented edge u -> v as x in N+(u) cap N+(v). It adds one to t of its
// three edges:
//   (v, x): counted in shared memory per entry of N+(v), flushed once;
//   (u, v): summed over the warp that scans N+(u), one atomic per edge;
//   (u, x): one global atomic per triangle.
// Work is grouped by the middle vertex v: a CTA stages N+(v) in a
// shared-memory hash table and streams N+(u) (coalesced) for a chunk of v's
// in-neighbours u, so a membership test is a shared-memory probe instead of
// a random DRAM access. The per-edge t are folded in edge order of the
// out-lists (the sums do not depend on the order): N3 = t,
// N4 = d_u + d_v - 2 - 2t, their sums and sums of squares in 128 bits.
#include <string.h>

#include "common.cuh"

namespace gs {

// count.cu: final pass over the 128-bit block partials.
__global__ void k_fold_final(const unsigned __int128* __restrict__ part, int blocks,
                             unsigned long long* __restrict__ out);

namespace {

constexpr int kThreads = 256;
constexpr unsigned kFull = 0xffffffffu;
constexpr int64_t kInChunk = 256;      // in-neighbours per work unit
constexpr int32_t kMaxOutDegree = 4096;  // larger out-lists: the general pass
// Resident CTAs per SM (as far as shared memory allows).
constexpr int kOrientBlocksPerSm = 8;
// Out-list entries a lane loads before it probes them (loads in flight).
constexpr int kProbeBatch = 4;

typedef unsigned __int128 u128;

__device__ __forceinline__ bool ranks_above(int64_t dx, int32_t x, int64_t dv, int32_t v) {
  return dx > dv || (dx == dv && x > v);
}

// Out- and in-degree of every vertex (one warp per vertex).
__global__ void k_orient_count(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                               int64_t n, int64_t* __restrict__ dplus, int64_t* __restrict__ dminus,
                               unsigned long long* __restrict__ maxd) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  unsigned long long mx = 0;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    const int64_t dv = row_ptr[v + 1] - row_ptr[v];
    unsigned up = 0;
    for (int64_t p = row_ptr[v] + lane; p < row_ptr[v + 1]; p += 32) {
      const int32_t x = col[p];
      up += ranks_above(__ldg(row_ptr + x + 1) - __ldg(row_ptr + x), x, dv, (int32_t)v);
    }
    up = __reduce_add_sync(kFull, up);
    if (lane == 0) {
      dplus[v] = up;
      dminus[v] = dv - up;
      mx = up > mx ? up : mx;
    }
  }
  if (lane == 0 && mx) atomicMax(maxd, mx);
}

// Out-list (higher-ranked neighbours) and in-list (lower-ranked ones) of
// every vertex, both in increasing id (one warp per vertex). Lists longer than
// a warp have several steps' loads in flight, as a hub's list is the kernel's
// tail; the others are one step (2M vertices of mean degree 4: 0.23 ms with one
// step for all, 0.50 with four, 0.22 so).
__global__ void __launch_bounds__(kThreads, 8)
    k_orient_fill(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int64_t n,
                  const int64_t* __restrict__ out_ptr, const int64_t* __restrict__ in_ptr,
                  int32_t* __restrict__ out_col, int32_t* __restrict__ in_col) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    const int64_t begin = row_ptr[v], end = row_ptr[v + 1], dv = end - begin;
    int64_t o = out_ptr[v], i = in_ptr[v];
    // one step: x = -1 past the list
    auto place = [&](int32_t x, bool up) {
      const unsigned bu = __ballot_sync(kFull, x >= 0 && up);
      const unsigned bd = __ballot_sync(kFull, x >= 0 && !up);
      if (x >= 0 && up) out_col[o + __popc(bu & below)] = x;
      if (x >= 0 && !up) in_col[i + __popc(bd & below)] = x;
      o += __popc(bu);
      i += __popc(bd);
    };
    if (dv <= 32) {
      const int32_t x = lane < dv ? col[begin + lane] : -1;
      const int64_t d = x >= 0 ? __ldg(row_ptr + x + 1) - __ldg(row_ptr + x) : 0;
      place(x, ranks_above(d, x, dv, (int32_t)v));
      continue;
    }
    constexpr int kDeep = 4;
    for (int64_t p0 = begin + lane; p0 - lane < end; p0 += 32 * kDeep) {
      int32_t x[kDeep], d[kDeep];  // degrees are below 2^31
#pragma unroll
      for (int h = 0; h < kDeep; ++h) x[h] = p0 + 32 * h < end ? col[p0 + 32 * h] : -1;
#pragma unroll
      for (int h = 0; h < kDeep; ++h)
        d[h] = x[h] >= 0 ? (int32_t)(__ldg(row_ptr + x[h] + 1) - __ldg(row_ptr + x[h])) : 0;
#pragma unroll
      for (int h = 0; h < kDeep; ++h) place(x[h], ranks_above(d[h], x[h], dv, (int32_t)v));
    }
  }
}

// in_pos[j]: the out-list position of v in N+(u) for the in-edge u -> v
// stored at in_col[j] (halving search of the short out-list). Warps take equal
// contiguous ranges of the m in-edges: a hub's in-list, which one warp walked
// before, was the tail of the kernel (1.3 of the 28 ms of a 100k-vertex graph's
// registration). The vertex of each is found as last_le_lanes says.
__global__ void k_orient_in_pos(const int64_t* __restrict__ out_ptr,
                                const int32_t* __restrict__ out_col,
                                const int64_t* __restrict__ in_ptr,
                                const int32_t* __restrict__ in_col, int64_t n, int64_t m,
                                uint32_t* __restrict__ in_pos) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int64_t per = ((m + 31) / 32 + warps - 1) / warps * 32;
  const int64_t j0 = warp * per, j1 = min(m, j0 + per);
  if (j0 >= j1) return;
  int64_t v = last_le_warp(in_ptr, n, j0);  // the vertex whose in-list holds the position
  for (int64_t jb = j0; jb < j1; jb += 32) {
    const int64_t j = jb + lane;
    v = last_le_lanes(in_ptr, n, v, min(j, j1 - 1));
    if (j < j1) {
      const int32_t u = in_col[j];
      int64_t lo = out_ptr[u], len = out_ptr[u + 1] - lo;
      while (len > 1) {
        const int64_t half = len >> 1;
        lo = (__ldg(out_col + lo + half) <= (int32_t)v) ? lo + half : lo;
        len -= half;
      }
      in_pos[j] = (uint32_t)lo;
    }
    v = __shfl_sync(kFull, v, 31);
  }
}

// Work units: ceil(d-(v) / kInChunk) per vertex with a non-empty out-list.
__global__ void k_orient_units(const int64_t* __restrict__ out_ptr,
                               const int64_t* __restrict__ in_ptr, int64_t n,
                               int64_t* __restrict__ units) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t dp = out_ptr[v + 1] - out_ptr[v], dm = in_ptr[v + 1] - in_ptr[v];
    units[v] = dp > 0 ? (dm + kInChunk - 1) / kInChunk : 0;
  }
}

// Hash table of N+(v): buckets of four keys. A bucket is filled in order, so a
// key that is not among a bucket's four is in the next one only if the fourth
// is taken. kSlotsWanted slots per entry are taken as far as kTableSlots go,
// which lets eight CTAs share an SM; an out-list too long for that gets at
// least kSlotsLeast per entry. R-MAT 22 (out-lists of up to 1,100): 42.5 / 39.1
// / 37.4 ms at 3 / 4 / 6 slots wanted; 39.4 / 39.1 / 44.3 ms with 2560 / 3328 /
// 4096 table slots (four wanted).
constexpr int64_t kTableSlots = 3328;
constexpr int64_t kSlotsWanted = 6, kSlotsLeast = 2;
__host__ __device__ __forceinline__ int table_buckets(int64_t out_degree) {
  int64_t s = kSlotsWanted * out_degree;
  if (s > kTableSlots) s = kSlotsLeast * out_degree > kTableSlots ? kSlotsLeast * out_degree : kTableSlots;
  return (int)(s < 64 ? 16 : (s + 3) / 4);
}
__device__ __forceinline__ int bucket_of(int32_t x, int buckets) {
  return (int)__umulhi((uint32_t)x * 2654435761u, (uint32_t)buckets);
}

// Triangles by middle vertex (see the file comment). Persistent CTAs take
// units from a counter; dynamic shared memory holds the hash table of
// N+(v): keys (int32, -1 empty) and one word per slot holding the out-list
// position of x (low 16 bits) and the count of (v, x) (high 16 bits: at
// most kInChunk per unit).
//
// Bound by instruction issue (84% of the cycles; a probe walked its chain of
// single slots as long as the longest of 32 lanes, 100 warp instructions per 32
// probes). Buckets of four keys are read in one load, and a second bucket is
// rarely needed. R-MAT 22, 14.4e9 probes: 53.3 -> 34.8 ms.
__global__ void __launch_bounds__(kThreads, kOrientBlocksPerSm)
    k_tri_oriented(const int64_t* __restrict__ out_ptr, const int32_t* __restrict__ out_col,
                   const int64_t* __restrict__ in_ptr, const int32_t* __restrict__ in_col,
                   const uint32_t* __restrict__ in_pos, const int64_t* __restrict__ unit_off,
                   int64_t n, int max_buckets, unsigned int* __restrict__ tplus,
                   unsigned long long* __restrict__ counter,
                   unsigned long long* __restrict__ probes) {
  extern __shared__ int4 keys4[];
  int32_t* keys = reinterpret_cast<int32_t*>(keys4);
  uint32_t* slotw = reinterpret_cast<uint32_t*>(keys4 + max_buckets);
  __shared__ int64_t cur;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t U = __ldg(unit_off + n);
  unsigned long long my_probes = 0;
  for (;;) {
    if (threadIdx.x == 0) cur = (int64_t)atomicAdd(counter, 1ull);
    __syncthreads();
    const int64_t unit = cur;
    if (unit >= U) break;
    int64_t lo = 0, len = n;  // vertex owning the unit
    while (len > 1) {
      const int64_t half = len >> 1;
      lo = (__ldg(unit_off + lo + half) <= unit) ? lo + half : lo;
      len -= half;
    }
    const int32_t v = (int32_t)lo;
    const int64_t ob = out_ptr[v], od = out_ptr[v + 1] - ob;
    const int64_t j0 = in_ptr[v] + (unit - __ldg(unit_off + v)) * kInChunk;
    const int64_t j1 = min(in_ptr[v + 1], j0 + kInChunk);
    const int nb = table_buckets(od);  // this unit's table
    for (int s = threadIdx.x; s < nb; s += kThreads) keys4[s] = make_int4(-1, -1, -1, -1);
    __syncthreads();
    for (int64_t i = threadIdx.x; i < od; i += kThreads) {
      const int32_t x = out_col[ob + i];
      int b = bucket_of(x, nb), j = 0;
      while (atomicCAS(keys + 4 * b + j, -1, x) != -1)
        if (++j == 4) {
          j = 0;
          b = b + 1 == nb ? 0 : b + 1;
        }
      slotw[4 * b + j] = (uint32_t)i;  // position, count 0
    }
    __syncthreads();
    for (int64_t j = j0 + wid; j < j1; j += kThreads / 32) {
      const int32_t u = in_col[j];
      const int64_t ub = out_ptr[u], ud = out_ptr[u + 1] - ub;
      unsigned hits = 0;
      for (int64_t i0 = lane; i0 < ud; i0 += 32 * kProbeBatch) {
        int32_t xb[kProbeBatch];
#pragma unroll
        for (int q = 0; q < kProbeBatch; ++q)
          xb[q] = i0 + 32 * q < ud ? __ldg(out_col + ub + i0 + 32 * q) : -1;
#pragma unroll
        for (int q = 0; q < kProbeBatch; ++q) {
          const int32_t x = xb[q];
          if (x < 0) continue;
          int b = bucket_of(x, nb), at = -1;
          for (;;) {
            const int4 k = keys4[b];
            if (k.x == x) at = 0;
            if (k.y == x) at = 1;
            if (k.z == x) at = 2;
            if (k.w == x) at = 3;
            if (at >= 0 || k.w == -1) break;
            b = b + 1 == nb ? 0 : b + 1;
          }
          if (at >= 0) {
            ++hits;
            atomicAdd(slotw + 4 * b + at, 1u << 16);
            atomicAdd(tplus + ub + i0 + 32 * q, 1u);  // edge (u, x)
          }
        }
      }
      my_probes += (unsigned long long)(ud > lane ? (ud - lane + 31) / 32 : 0);
      hits = __reduce_add_sync(kFull, hits);
      if (lane == 0 && hits) atomicAdd(tplus + in_pos[j], hits);  // edge (u, v)
    }
    __syncthreads();
    for (int s = threadIdx.x; s < 4 * nb; s += kThreads) {
      const uint32_t w = slotw[s];
      if (keys[s] != -1 && (w >> 16) != 0) atomicAdd(tplus + ob + (w & 0xffffu), w >> 16);  // (v, x)
    }
    __syncthreads();  // the table and cur are reused for the next unit
  }
  my_probes = __reduce_add_sync(kFull, (unsigned)min(my_probes, 0xffffffffull));
  if (lane == 0 && my_probes) atomicAdd(probes, my_probes);
}

// N3 = t, N4 = d_u + d_v - 2 - 2t per oriented edge; 128-bit block sums in
// the layout of k_fold (order 3, 4, 7, ..., 12, then the squares).
__global__ void __launch_bounds__(kThreads)
    k_fold_oriented(const int64_t* __restrict__ row_ptr, const int64_t* __restrict__ out_ptr,
                    const int32_t* __restrict__ out_col, const unsigned int* __restrict__ tplus,
                    int64_t n, u128* __restrict__ part, unsigned long long* __restrict__ stats) {
  u128 s3 = 0, s4 = 0, q3 = 0, q4 = 0;
  unsigned long long model = 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < n; u += warps) {
    const int64_t du = row_ptr[u + 1] - row_ptr[u];
    for (int64_t p = out_ptr[u] + lane; p < out_ptr[u + 1]; p += 32) {
      const int32_t v = out_col[p];
      const int64_t dv = __ldg(row_ptr + v + 1) - __ldg(row_ptr + v);
      const uint64_t t = tplus[p];
      const uint64_t n4 = (uint64_t)(du + dv - 2) - 2 * t;
      s3 += t;
      s4 += n4;
      q3 += (u128)t * t;
      q4 += (u128)n4 * n4;
      model += 24 + 4 * (unsigned long long)(du + dv);
    }
  }
  __shared__ u128 red[kThreads / 32][4];
  u128 v4[4] = {s3, s4, q3, q4};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    u128 x = v4[i];
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long lo = (unsigned long long)x, hi = (unsigned long long)(x >> 64);
      lo = __shfl_down_sync(kFull, lo, o);
      hi = __shfl_down_sync(kFull, hi, o);
      x += ((u128)hi << 64) | lo;
    }
    if (lane == 0) red[wid][i] = x;
  }
  for (int o = 16; o > 0; o >>= 1) model += __shfl_xor_sync(kFull, model, o);
  if (lane == 0 && model) atomicAdd(stats + 2, model);
  __syncthreads();
  if (threadIdx.x < 16) {
    u128 s = 0;
    const int k = threadIdx.x;
    const int src = k == 0 ? 0 : k == 1 ? 1 : k == 8 ? 2 : k == 9 ? 3 : -1;
    if (src >= 0)
      for (int w = 0; w < kThreads / 32; ++w) s += red[w][src];
    part[(int64_t)blockIdx.x * 16 + k] = s;
  }
}

}  // namespace

// Oriented out- and in-lists for the exact 3-node pass (registration).
// Skipped (the general pass serves) when the graph has 2^31 or more edges
// or an out-list longer than kMaxOutDegree.
gs_status build_oriented(gs_graph* g, cudaStream_t stream) {
  const int64_t n = g->dev.n, m = g->m;
  if (n == 0 || m == 0 || m >= ((int64_t)1 << 31)) return GS_OK;
  int64_t* dp = nullptr;
  int64_t* dm = nullptr;
  int64_t* tmp = nullptr;
  unsigned long long* d_max = nullptr;
  auto release = [&]() {
    cudaFree(dp);
    cudaFree(dm);
    cudaFree(tmp);
    cudaFree(d_max);
  };
  if (cudaMalloc(&dp, sizeof(int64_t) * (size_t)(n + 1)) != cudaSuccess ||
      cudaMalloc(&dm, sizeof(int64_t) * (size_t)(n + 1)) != cudaSuccess ||
      cudaMalloc(&tmp, sizeof(int64_t) * (size_t)scan_tmp_elems(n + 1)) != cudaSuccess ||
      cudaMalloc(&d_max, sizeof(unsigned long long)) != cudaSuccess) {
    release();
    cudaGetLastError();
    return GS_OK;  // no room: the general pass serves
  }
  cudaMemsetAsync(d_max, 0, sizeof(unsigned long long), stream);
  k_orient_count<<<grid_for(n * 32, kThreads, 8), kThreads, 0, stream>>>(
      g->dev.row_ptr, g->dev.col, n, dp, dm, d_max);
  unsigned long long hmax = 0;
  cudaMemcpyAsync(&hmax, d_max, sizeof(hmax), cudaMemcpyDeviceToHost, stream);
  cudaError_t e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) {
    release();
    return cuda_fail(e, "oriented lists", __FILE__, __LINE__);
  }
  if ((int64_t)hmax > kMaxOutDegree) {
    release();
    return GS_OK;
  }
  bool ok = cudaMalloc(&g->out_ptr, sizeof(int64_t) * (size_t)(n + 1)) == cudaSuccess &&
            cudaMalloc(&g->in_ptr, sizeof(int64_t) * (size_t)(n + 1)) == cudaSuccess &&
            cudaMalloc(&g->out_col, sizeof(int32_t) * (size_t)m) == cudaSuccess &&
            cudaMalloc(&g->in_col, sizeof(int32_t) * (size_t)m) == cudaSuccess &&
            cudaMalloc(&g->in_pos, sizeof(uint32_t) * (size_t)m) == cudaSuccess &&
            cudaMalloc(&g->orient_units, sizeof(int64_t) * (size_t)(n + 1)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    release();
    cudaFree(g->out_ptr);
    cudaFree(g->in_ptr);
    cudaFree(g->out_col);
    cudaFree(g->in_col);
    cudaFree(g->in_pos);
    cudaFree(g->orient_units);
    g->out_ptr = g->in_ptr = g->orient_units = nullptr;
    g->out_col = g->in_col = nullptr;
    g->in_pos = nullptr;
    return GS_OK;
  }
  gs_status s = exclusive_scan_i64(dp, g->out_ptr, n, tmp, stream);
  if (s == GS_OK) s = exclusive_scan_i64(dm, g->in_ptr, n, tmp, stream);
  if (s == GS_OK) {
    k_orient_fill<<<grid_for(n * 32, kThreads, 8), kThreads, 0, stream>>>(
        g->dev.row_ptr, g->dev.col, n, g->out_ptr, g->in_ptr, g->out_col, g->in_col);
    k_orient_in_pos<<<grid_for(m, kThreads, 8), kThreads, 0, stream>>>(
        g->out_ptr, g->out_col, g->in_ptr, g->in_col, n, m, g->in_pos);
    k_orient_units<<<grid_for(n, kThreads, 8), kThreads, 0, stream>>>(g->out_ptr, g->in_ptr, n,
                                                                       g->orient_units);
    s = exclusive_scan_i64(g->orient_units, g->orient_units, n, tmp, stream);
  }
  e = cudaStreamSynchronize(stream);
  release();
  if (s != GS_OK) return s;
  if (e != cudaSuccess) return cuda_fail(e, "oriented lists", __FILE__, __LINE__);
  g->max_out_degree = (int64_t)hmax;
  return GS_OK;
}

// The exact 3-node pass over every edge through the oriented lists: sums in
// the layout of gs_count's (32 words: 8 sums and 8 sums of squares, low and
// high) in d_sums, statistics in d_stats. Needs build_oriented's lists.
gs_status count_tri_oriented(const gs_graph* g, gs_workspace* ws, unsigned long long* h_sums,
                             unsigned long long* h_stats, int64_t* launches, cudaStream_t stream) {
  const int64_t n = g->dev.n, m = g->m;
  const int buckets = table_buckets(g->max_out_degree);
  const size_t smem = (size_t)buckets * 4 * 2 * sizeof(int32_t);
  const int fold_blocks = grid_for(n * 32, kThreads, 2);
  void* base = nullptr;
  GS_TRY(ws_reserve(ws, 0,
                    Carve::bytes_for<unsigned int>(m) + Carve::bytes_for<unsigned long long>(8) +
                        Carve::bytes_for<unsigned long long>(32) +
                        Carve::bytes_for<u128>((int64_t)fold_blocks * 16),
                    stream, &base));
  Carve c{(char*)base, 0};
  unsigned int* tplus = c.take<unsigned int>(m);
  unsigned long long* stats = c.take<unsigned long long>(8);
  unsigned long long* sums = c.take<unsigned long long>(32);
  u128* part = c.take<u128>((int64_t)fold_blocks * 16);
  if (ws->timing) cudaEventRecord(ws->ev[0], stream);
  GS_CUDA(cudaMemsetAsync(tplus, 0, sizeof(unsigned int) * (size_t)m, stream));
  GS_CUDA(cudaMemsetAsync(stats, 0, sizeof(unsigned long long) * 8, stream));
  if (ws->timing) cudaEventRecord(ws->ev[1], stream);
  static bool attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    GS_CUDA(cudaFuncSetAttribute(k_tri_oriented, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((size_t)table_buckets(kMaxOutDegree) * 4 * 2 * sizeof(int32_t))));
    attr_set[dev] = true;
  }
  if (ws->timing) cudaEventRecord(ws->ev[2], stream);
  k_tri_oriented<<<sm_count() * kOrientBlocksPerSm, kThreads, smem, stream>>>(
      g->out_ptr, g->out_col, g->in_ptr, g->in_col, g->in_pos, g->orient_units, n, buckets, tplus,
      stats + 7, stats + 0);
  if (ws->timing)
    for (int ev = 3; ev <= 10; ++ev) cudaEventRecord(ws->ev[ev], stream);  // phases 2-4 empty
  GS_CUDA(cudaGetLastError());
  k_fold_oriented<<<fold_blocks, kThreads, 0, stream>>>(g->dev.row_ptr, g->out_ptr, g->out_col,
                                                        tplus, n, part, stats);
  k_fold_final<<<1, 512, 0, stream>>>(part, fold_blocks, sums);
  if (ws->timing) cudaEventRecord(ws->ev[11], stream);
  GS_CUDA(cudaGetLastError());
  GS_CUDA(cudaMemcpyAsync(h_sums, sums, sizeof(unsigned long long) * 32, cudaMemcpyDeviceToHost,
                          stream));
  GS_CUDA(cudaMemcpyAsync(h_stats, stats, sizeof(unsigned long long) * 8, cudaMemcpyDeviceToHost,
                          stream));
  GS_CUDA(cudaStreamSynchronize(stream));
  *launches = 5;
  return GS_OK;
}

}  // namespace gs
