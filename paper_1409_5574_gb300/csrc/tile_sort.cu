// Counting sort of particles by the 32 x 32-cell tile of the 2D Yee grid that
// holds them and by cell inside each tile, and the work list of the tile-staged
// gather kernel: one item per chunk of at most kChunk particles of one tile.  In
// cell order the lanes of a warp read the same or neighbouring stencil values
// of the staged tile (broadcasts instead of shared-memory bank conflicts).
// Particles keep their ids (pid array), so the Philox streams and ledger
// entries follow them.  The order inside a cell depends on atomic timing;
// results per particle do not.
#include <cuda_runtime.h>
#include <stdint.h>

#include "prad_internal.h"

namespace prad {

namespace {

// (v - v0) inv reduced to [0, n), with every rounding fixed.  Several kernels
// find a particle's cell and must agree to the bit: a block reserves its run
// of a tile from one count and fills it from another, so two contractions of
// these products and sums would write beyond the run.
__device__ __forceinline__ float wrapped(float v, float v0, float inv, float n) {
  const float c = __fmul_rn(__fsub_rn(v, v0), inv);
  return __fmaf_rn(-n, floor(__fdiv_rn(c, n)), c);
}
__device__ __forceinline__ double wrapped(double v, double v0, double inv, double n) {
  const double c = __dmul_rn(__dsub_rn(v, v0), inv);
  return __fma_rn(-n, floor(__ddiv_rn(c, n)), c);
}

// The grid cell (ix, iy) that holds (x, y): periodic, clamped (also for NaN)
// into range.
template <typename R>
__device__ __forceinline__ int2 cell_xy(R x, R y, int nx, int ny, R x0, R y0, R inv_dx,
                                        R inv_dy) {
  const R fx = static_cast<R>(nx), fy = static_cast<R>(ny);
  const R xi = wrapped(x, x0, inv_dx, fx), yi = wrapped(y, y0, inv_dy, fy);
  int ix = static_cast<int>(fmin(fmax(xi, R(0)), fx - R(1)));
  int iy = static_cast<int>(fmin(fmax(yi, R(0)), fy - R(1)));
  ix = ix < 0 ? 0 : (ix >= nx ? nx - 1 : ix);
  iy = iy < 0 ? 0 : (iy >= ny ? ny - 1 : iy);
  return make_int2(ix, iy);
}

template <typename R>
__device__ __forceinline__ int tile_of(R x, R y, int nx, int ny, int ntx, R x0, R y0,
                                       R inv_dx, R inv_dy) {
  const int2 c = cell_xy(x, y, nx, ny, x0, y0, inv_dx, inv_dy);
  return (c.y / kTile) * ntx + (c.x / kTile);
}

// The cell's index inside its tile, row-major (0 .. kTile^2 - 1).
template <typename R>
__device__ __forceinline__ int cell_in_tile(R x, R y, int nx, int ny, R x0, R y0, R inv_dx,
                                            R inv_dy) {
  const int2 c = cell_xy(x, y, nx, ny, x0, y0, inv_dx, inv_dy);
  return (c.y % kTile) * kTile + (c.x % kTile);
}

// Warp-aggregated increment of counter[t] for every valid lane: lanes of the
// warp with the same tile form one group, its first lane adds the group's
// size with one atomic, and each lane receives base + its rank in the group.
// Particles stay nearly tile-ordered between sorts, so a warp usually holds
// one or two tiles: one or two atomics per 32 particles instead of 32 on the
// same counter.  Warp-collective (every lane calls it).
__device__ __forceinline__ unsigned int warp_claim(unsigned int* counter, int t, bool valid) {
  const int lane = threadIdx.x & 31;
  const unsigned vmask = __ballot_sync(0xffffffffu, valid);
  unsigned int slot = 0u;
  if (valid) {
    const unsigned peers = __match_any_sync(vmask, t);
    const int leader = __ffs(peers) - 1;
    const int rank = __popc(peers & ((1u << lane) - 1u));
    unsigned int base = 0u;
    if (lane == leader) base = atomicAdd(counter + t, static_cast<unsigned int>(__popc(peers)));
    slot = __shfl_sync(peers, base, leader) + static_cast<unsigned int>(rank);
  }
  return slot;
}

// Grid-stride over warps of 32 consecutive particles (every lane of a warp
// takes the same number of iterations).
template <typename R>
__global__ void k_tile_count(const R* __restrict__ x, const R* __restrict__ y, int64_t n,
                             int nx, int ny, int ntx, R x0, R y0, R inv_dx, R inv_dy,
                             unsigned int* __restrict__ counts) {
  const int lane = threadIdx.x & 31;
  const int64_t wstride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t w0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + (threadIdx.x & ~31);
       w0 < n; w0 += wstride) {
    const int64_t i = w0 + lane;
    const bool valid = i < n;
    const int t = valid ? tile_of(x[i], y[i], nx, ny, ntx, x0, y0, inv_dx, inv_dy) : 0;
    (void)warp_claim(counts, t, valid);
  }
}

// One block: exclusive scan of the tile counts (starts, scatter cursors) and
// of the per-tile chunk counts (work list offsets); writes the work list.
// Warp w owns a contiguous run of tiles and reads it 32 at a time, so counts,
// starts and cursors are touched in whole lines (one tile per thread and
// iteration; with a run of tiles per thread 16384 tiles took 27 us, now 7).
constexpr int kScanThreads = 1024;

__device__ __forceinline__ unsigned int warp_inclusive(unsigned int v, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int u = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += u;
  }
  return v;
}

// sparse > 0 (binned gather): with fewer than `sparse` particles per occupied
// tile there is no tile work, and the gate lets the plain kernel run instead;
// so too with at least `ordered` > 0 particles near the one before them
// (k_bin_count's last counter).
__global__ void __launch_bounds__(kScanThreads)
    k_tile_scan(const unsigned int* __restrict__ counts, int ntiles,
                unsigned int* __restrict__ starts, unsigned int* __restrict__ cursor,
                int4* __restrict__ work, unsigned int* __restrict__ work_count,
                unsigned int chunk, unsigned int sparse, unsigned int ordered) {
  constexpr int kWarps = kScanThreads / 32;
  __shared__ unsigned int s_sum[kWarps], s_chunks[kWarps], s_used[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = ((ntiles + kWarps - 1) / kWarps + 31) / 32 * 32;
  const int lo = warp * per, hi = min(lo + per, ntiles);
  unsigned int sum = 0, chunks = 0, used = 0;
#pragma unroll 4
  for (int t0 = lo; t0 < hi; t0 += 32) {
    const unsigned int c = t0 + lane < hi ? counts[t0 + lane] : 0u;
    sum += c;
    chunks += (c + chunk - 1) / chunk;
    used += c != 0u;
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  chunks = __reduce_add_sync(0xffffffffu, chunks);
  used = __reduce_add_sync(0xffffffffu, used);
  if (lane == 0) {
    s_sum[warp] = sum;
    s_chunks[warp] = chunks;
    s_used[warp] = used;
  }
  __syncthreads();
  if (warp == 0) {
    const unsigned int a = s_sum[lane], b = s_chunks[lane];
    const unsigned int ia = warp_inclusive(a, lane), ib = warp_inclusive(b, lane);
    const unsigned int tiles = __reduce_add_sync(0xffffffffu, s_used[lane]);
    s_sum[lane] = ia - a;
    s_chunks[lane] = ib - b;
    if (lane == 31) {
      starts[ntiles] = ia;
      const bool none = (sparse != 0u && ia < static_cast<uint64_t>(sparse) * tiles) ||
                        (ordered != 0u && counts[ntiles] >= ordered);
      work_count[0] = none ? 0u : ib;
      work_count[1] = none ? 1u : 0u;
    }
  }
  __syncthreads();
  unsigned int run = s_sum[warp], wrun = s_chunks[warp];
#pragma unroll 4
  for (int t0 = lo; t0 < hi; t0 += 32) {
    const int t = t0 + lane;
    const unsigned int c = t < hi ? counts[t] : 0u;
    const unsigned int k = (c + chunk - 1) / chunk;
    const unsigned int ic = warp_inclusive(c, lane), ik = warp_inclusive(k, lane);
    const unsigned int first = run + ic - c;
    if (t < hi) {
      starts[t] = first;
      cursor[t] = first;
    }
    unsigned int w = wrun + ik - k;
    for (unsigned int f = 0; f < c; f += chunk) {
      const unsigned int e = f + chunk < c ? f + chunk : c;
      work[w++] = make_int4(t, static_cast<int>(first + f), static_cast<int>(first + e), 0);
    }
    run += __shfl_sync(0xffffffffu, ic, 31);
    wrun += __shfl_sync(0xffffffffu, ik, 31);
  }
}

template <typename R>
struct Arrays7 {
  R* p[7];  // x y z ux uy uz w (z may be null)
};

template <typename R>
__global__ void k_tile_scatter(const Arrays7<R> src, const Arrays7<R> dst,
                               const uint32_t* __restrict__ pid, uint32_t* __restrict__ pid_out,
                               int64_t n, int nx, int ny, int ntx, R x0, R y0, R inv_dx,
                               R inv_dy, unsigned int* __restrict__ cursor) {
  const int lane = threadIdx.x & 31;
  const int64_t wstride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t w0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + (threadIdx.x & ~31);
       w0 < n; w0 += wstride) {
    const int64_t i = w0 + lane;
    const bool valid = i < n;
    const int t =
        valid ? tile_of(src.p[0][i], src.p[1][i], nx, ny, ntx, x0, y0, inv_dx, inv_dy) : 0;
    const unsigned int d = warp_claim(cursor, t, valid);
    if (valid) {
#pragma unroll
      for (int k = 0; k < 7; ++k)
        if (src.p[k]) dst.p[k][d] = src.p[k][i];
      pid_out[d] = pid[i];
    }
  }
}

// Second pass, one block per tile: the tile's particles (a contiguous range
// of the tile-sorted scratch copy) are ordered by cell with a shared-memory
// histogram of the tile's kTile^2 cells, and written back to the caller's
// arrays.  The cell is computed with the same arithmetic as the tile, so
// every particle stays inside its tile's range.
constexpr int kCellThreads = kTile * kTile;

template <typename R>
__global__ void __launch_bounds__(kCellThreads)
    k_cell_scatter(const Arrays7<R> src, const Arrays7<R> dst,
                   const uint32_t* __restrict__ pid_src, uint32_t* __restrict__ pid_dst,
                   const unsigned int* __restrict__ starts, int nx, int ny, R x0, R y0,
                   R inv_dx, R inv_dy) {
  __shared__ unsigned int s_cnt[kCellThreads];
  __shared__ unsigned int s_warp[kCellThreads / 32];
  const unsigned int a = starts[blockIdx.x], b = starts[blockIdx.x + 1];
  if (a == b) return;  // the whole block leaves: no barrier is left waiting
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  s_cnt[tid] = 0u;
  __syncthreads();
  for (unsigned int i = a + tid; i < b; i += kCellThreads)
    atomicAdd(s_cnt + cell_in_tile(src.p[0][i], src.p[1][i], nx, ny, x0, y0, inv_dx, inv_dy),
              1u);
  __syncthreads();
  // exclusive scan of the cell counts: within warps, then over the warp sums
  const unsigned int c = s_cnt[tid];
  unsigned int v = c;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned int u = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += u;
  }
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  if (warp == 0) {
    unsigned int w = s_warp[lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned int u = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += u;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  s_cnt[tid] = (warp > 0 ? s_warp[warp - 1] : 0u) + v - c;  // cursor of cell tid
  __syncthreads();
  for (unsigned int i = a + tid; i < b; i += kCellThreads) {
    const int cl = cell_in_tile(src.p[0][i], src.p[1][i], nx, ny, x0, y0, inv_dx, inv_dy);
    const unsigned int d = a + atomicAdd(s_cnt + cl, 1u);
#pragma unroll
    for (int k = 0; k < 7; ++k)
      if (src.p[k]) dst.p[k][d] = src.p[k][i];
    pid_dst[d] = pid_src[i];
  }
}

// ---------------------------------------------------------------------------
// FP32, binning: a copy of the state in that order, on which the tile-staged
// kernel runs.  It goes back to where it came from (particles that stay in
// the caller's order) or, for the sorted path, in its own order, both streams
// of whole lines.  The caller's arrays are only ever streamed; the scattered
// side is the copy, whose particles are one 32-byte sector each.  (Gathering the seven arrays through an index in
// the push itself cost 0.25 ns per particle and launch on 8M particles in
// random order; now 2^21 particles in random order take 13 us to count, 6 to
// scan, 27 + 28 to place by tile and cell, 39 to copy and 26 to write back,
// beside 1014 us for 25 steps of the push: 7.98 ms with the plain gather,
// 1.38 ms so.)  Block b owns the contiguous
// particles [n b / B, n (b + 1) / B); the tile counters of its particles sit
// in shared memory (SM) so that a tile costs a block one global atomic, not
// one per warp that meets it; grids of more than kBinTiles tiles count in
// global memory.
// ---------------------------------------------------------------------------
constexpr int kBinThreads = 512;
constexpr int kBinTiles = 16384;  // 64 KB of shared counters

struct BinGeom {
  int nx, ny, ntx, ntiles;
  float x0, y0, inv_dx, inv_dy;
};

__device__ __forceinline__ uint2 bin_of(const BinGeom& g, float x, float y) {
  const int2 c = cell_xy(x, y, g.nx, g.ny, g.x0, g.y0, g.inv_dx, g.inv_dy);
  return make_uint2(static_cast<unsigned>((c.y / kTile) * g.ntx + (c.x / kTile)),
                    static_cast<unsigned>((c.y % kTile) * kTile + (c.x % kTile)));
}

// An increment of tile t's counter by every valid lane and the slot it got.
// Shared counters: one add for a warp inside one tile, else one per lane
// (grouping the lanes of a warp by tile costs more than the adds when the
// caller's order is random); global ones: one add per tile of the warp.
template <bool SM>
__device__ __forceinline__ unsigned int bin_claim(unsigned int* cnt, unsigned int t, bool valid) {
  if constexpr (!SM) return warp_claim(cnt, static_cast<int>(t), valid);
  const int lane = threadIdx.x & 31;
  unsigned int d = 0u;
  const unsigned int t0 = __shfl_sync(0xffffffffu, t, 0);  // (by every lane, valid or not)
  const bool same = valid && t == t0;
  if (__all_sync(0xffffffffu, same)) {
    if (lane == 0) d = atomicAdd(cnt + t, 32u);
    return __shfl_sync(0xffffffffu, d, 0) + lane;
  }
  if (valid) d = atomicAdd(cnt + t, 1u);
  return d;
}

// Counts of this block's particles by tile, added into cnt.
template <bool SM>
__device__ __forceinline__ void bin_count_range(const BinGeom& g, const float* __restrict__ x,
                                                const float* __restrict__ y, int64_t lo,
                                                int64_t hi, unsigned int* cnt) {
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int64_t w0 = lo + (threadIdx.x & ~31); w0 < hi; w0 += kBinThreads) {
    const int64_t i = w0 + lane;
    const bool valid = i < hi;
    const unsigned t = valid ? bin_of(g, x[i], y[i]).x : 0u;
    (void)bin_claim<SM>(cnt, t, valid);
  }
}

// near > 0: how many particles lie within that many cells, in x and in y, of
// the one before them in the caller's order (a warp's first counts as one) is
// added to counts[g.ntiles]: in an order of cells nearly all, in a random one
// few, and the plain gather's loads meet in L1 where they do.
template <bool SM>
__global__ void __launch_bounds__(kBinThreads)
    k_bin_count(const BinGeom g, const float* __restrict__ x, const float* __restrict__ y,
                int64_t n, unsigned int* __restrict__ counts, int near) {
  extern __shared__ unsigned int s_tile[];
  const int64_t lo = n * blockIdx.x / gridDim.x, hi = n * (blockIdx.x + 1) / gridDim.x;
  if (near > 0) {
    const int lane = threadIdx.x & 31;
    unsigned int mine = 0u;
#pragma unroll 4
    for (int64_t w0 = lo + (threadIdx.x & ~31); w0 < hi; w0 += kBinThreads) {
      const int64_t i = w0 + lane;
      const int2 c = i < hi ? cell_xy(x[i], y[i], g.nx, g.ny, g.x0, g.y0, g.inv_dx, g.inv_dy)
                            : make_int2(0, 0);
      const int px = __shfl_up_sync(0xffffffffu, c.x, 1);
      const int py = __shfl_up_sync(0xffffffffu, c.y, 1);
      mine += i < hi && (lane == 0 || (abs(c.x - px) <= near && abs(c.y - py) <= near));
    }
    mine = __reduce_add_sync(0xffffffffu, mine);
    if (lane == 0 && mine) atomicAdd(counts + g.ntiles, mine);
  }
  if constexpr (SM) {
    for (int t = threadIdx.x; t < g.ntiles; t += kBinThreads) s_tile[t] = 0u;
    __syncthreads();
    bin_count_range<true>(g, x, y, lo, hi, s_tile);
    __syncthreads();
    for (int t = threadIdx.x; t < g.ntiles; t += kBinThreads)
      if (s_tile[t]) atomicAdd(counts + t, s_tile[t]);
  } else {
    bin_count_range<false>(g, x, y, lo, hi, counts);
  }
}

// Keys (particle, cell) into tile order.  SM: the block counts its particles
// again, reserves its run of every tile it meets with one atomic, and places
// them with shared cursors.
template <bool SM>
__global__ void __launch_bounds__(kBinThreads)
    k_bin_scatter(const BinGeom g, const float* __restrict__ x, const float* __restrict__ y,
                  int64_t n, unsigned int* __restrict__ cursor,
                  const unsigned int* __restrict__ gate, uint2* __restrict__ keys) {
  if (*gate) return;
  extern __shared__ unsigned int s_tile[];
  const int64_t lo = n * blockIdx.x / gridDim.x, hi = n * (blockIdx.x + 1) / gridDim.x;
  if constexpr (SM) {
    for (int t = threadIdx.x; t < g.ntiles; t += kBinThreads) s_tile[t] = 0u;
    __syncthreads();
    bin_count_range<true>(g, x, y, lo, hi, s_tile);
    __syncthreads();
    for (int t = threadIdx.x; t < g.ntiles; t += kBinThreads)
      if (s_tile[t]) s_tile[t] = atomicAdd(cursor + t, s_tile[t]);
    __syncthreads();
  }
  unsigned int* cur = SM ? s_tile : cursor;
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int64_t w0 = lo + (threadIdx.x & ~31); w0 < hi; w0 += kBinThreads) {
    const int64_t i = w0 + lane;
    const bool valid = i < hi;
    const uint2 b = valid ? bin_of(g, x[i], y[i]) : make_uint2(0u, 0u);
    const unsigned int d = bin_claim<SM>(cur, b.x, valid);
    if (valid) keys[d] = make_uint2(static_cast<unsigned>(i), b.y);
  }
}

// One block per tile: the slots of the tile's particles in cell order.
__global__ void __launch_bounds__(kBinThreads)
    k_bin_cells(const uint2* __restrict__ keys, uint32_t* __restrict__ slot,
                const unsigned int* __restrict__ starts, const unsigned int* __restrict__ gate) {
  if (*gate) return;
  constexpr int kCells = kTile * kTile;
  static_assert(kCells == 2 * kBinThreads, "two cells per thread");
  __shared__ unsigned int s_cnt[kCells];
  __shared__ unsigned int s_warp[kBinThreads / 32];
  const unsigned int a = starts[blockIdx.x], b = starts[blockIdx.x + 1];
  if (a == b) return;  // the whole block leaves
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  s_cnt[tid] = 0u;
  s_cnt[tid + kBinThreads] = 0u;
  __syncthreads();
#pragma unroll 4
  for (unsigned int k = a + tid; k < b; k += kBinThreads) atomicAdd(s_cnt + keys[k].y, 1u);
  __syncthreads();
  // exclusive scan, thread tid holding cells 2 tid and 2 tid + 1
  const unsigned int c0 = s_cnt[2 * tid], c1 = s_cnt[2 * tid + 1];
  const unsigned int v = warp_inclusive(c0 + c1, lane);
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  if (warp == 0) {
    const unsigned int w = warp_inclusive(lane < kBinThreads / 32 ? s_warp[lane] : 0u, lane);
    if (lane < kBinThreads / 32) s_warp[lane] = w;
  }
  __syncthreads();
  const unsigned int e0 = (warp > 0 ? s_warp[warp - 1] : 0u) + v - c0 - c1;
  s_cnt[2 * tid] = e0;
  s_cnt[2 * tid + 1] = e0 + c0;
  __syncthreads();
#pragma unroll 4
  for (unsigned int k = a + tid; k < b; k += kBinThreads) {
    const uint2 q = keys[k];
    slot[q.x] = a + atomicAdd(s_cnt + q.y, 1u);
  }
}

// The state to its slots, and back.
__global__ void __launch_bounds__(256)
    k_bin_pack(const StepParams<float> P, const uint32_t* __restrict__ slot,
               const unsigned int* __restrict__ gate, float4* __restrict__ aos) {
  if (*gate) return;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < P.n;
       i += stride) {
    const size_t d = slot[i];
    const uint32_t id = P.pid ? P.pid[i] : P.pid0 + static_cast<uint32_t>(i);
    aos[2 * d] = make_float4(P.x[i], P.y[i], P.z ? P.z[i] : 0.0f, P.ux[i]);
    aos[2 * d + 1] = make_float4(P.uy[i], P.uz[i], P.w[i], __uint_as_float(id));
  }
}
// (z and w do not change on the grid)
__global__ void __launch_bounds__(256)
    k_bin_unpack(const StepParams<float> P, const uint32_t* __restrict__ slot,
                 const unsigned int* __restrict__ gate, const float4* __restrict__ aos) {
  if (*gate) return;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < P.n;
       i += stride) {
    const size_t d = slot[i];
    const float4 a = aos[2 * d], b = aos[2 * d + 1];
    P.x[i] = a.x;
    P.y[i] = a.y;
    P.ux[i] = a.w;
    P.uy[i] = b.x;
    P.uz[i] = b.y;
  }
}

// The copy back in its own order: the caller's particles reordered.
__global__ void __launch_bounds__(256)
    k_bin_unsort(const StepParams<float> P, const float4* __restrict__ aos,
                 float* __restrict__ w, uint32_t* __restrict__ pid) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < P.n;
       i += stride) {
    const float4 a = aos[2 * i], b = aos[2 * i + 1];
    P.x[i] = a.x;
    P.y[i] = a.y;
    if (P.z) P.z[i] = a.z;
    P.ux[i] = a.w;
    P.uy[i] = b.x;
    P.uz[i] = b.y;
    w[i] = b.z;
    pid[i] = __float_as_uint(b.w);
  }
}

int stream_grid(int64_t n, int num_sms) {
  const int64_t want = (n + 255) / 256, cap = 8 * static_cast<int64_t>(num_sms);
  return static_cast<int>(want < cap ? want : cap);
}

}  // namespace

cudaError_t launch_tile_bin(const StepParams<float>& p, const BinBuffers& b, int chunk, bool sparse,
                            int near, int num_sms, cudaStream_t s) {
  const int64_t n = p.n;
  const float *x = p.x, *y = p.y;
  const unsigned int* gated = b.work_count + 1;  // (written by the scan)
  BinGeom g;
  g.nx = p.nx;
  g.ny = p.ny;
  g.ntx = (p.nx + kTile - 1) / kTile;
  g.ntiles = b.ntiles;
  g.x0 = p.x0;
  g.y0 = p.y0;
  g.inv_dx = p.inv_dx;
  g.inv_dy = p.inv_dy;
  cudaError_t e = cudaMemsetAsync(b.counts, 0, sizeof(unsigned int) * (b.ntiles + 1), s);
  if (e != cudaSuccess) return e;
  const bool sm = b.ntiles <= kBinTiles;
  const size_t dyn = sm ? sizeof(unsigned int) * b.ntiles : 0;
  if (dyn > 48 * 1024) {
    if ((e = cudaFuncSetAttribute(k_bin_count<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kBinTiles * 4)) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(k_bin_scatter<true>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kBinTiles * 4)) != cudaSuccess)
      return e;
  }
  // blocks: three per SM (64 KB of counters each at most), fewer for sets
  // that would leave a block less than 2048 particles
  const int64_t want = (n + 2047) / 2048;
  const int grid = static_cast<int>(want < 3 * num_sms ? want : 3 * num_sms);
  if (sm)
    k_bin_count<true><<<grid, kBinThreads, dyn, s>>>(g, x, y, n, b.counts, near);
  else
    k_bin_count<false><<<grid, kBinThreads, 0, s>>>(g, x, y, n, b.counts, near);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_tile_scan<<<1, kScanThreads, 0, s>>>(b.counts, b.ntiles, b.starts, b.cursor, b.work,
                                          b.work_count, static_cast<unsigned int>(chunk),
                                          sparse ? kBinSparse : 0u,
                                          near > 0 ? static_cast<unsigned int>(n / 2 + 1) : 0u);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (sm)
    k_bin_scatter<true><<<grid, kBinThreads, dyn, s>>>(g, x, y, n, b.cursor, gated, b.keys);
  else
    k_bin_scatter<false><<<grid, kBinThreads, 0, s>>>(g, x, y, n, b.cursor, gated, b.keys);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_bin_cells<<<b.ntiles, kBinThreads, 0, s>>>(b.keys, b.slot, b.starts, gated);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_bin_pack<<<stream_grid(n, num_sms), 256, 0, s>>>(p, b.slot, gated, b.aos);
  return cudaGetLastError();
}

cudaError_t launch_tile_unbin(const StepParams<float>& p, const BinBuffers& b, int num_sms,
                              cudaStream_t s) {
  k_bin_unpack<<<stream_grid(p.n, num_sms), 256, 0, s>>>(p, b.slot, b.work_count + 1, b.aos);
  return cudaGetLastError();
}

cudaError_t launch_tile_unsort(const StepParams<float>& p, const BinBuffers& b, float* w,
                               uint32_t* pid, int num_sms, cudaStream_t s) {
  k_bin_unsort<<<stream_grid(p.n, num_sms), 256, 0, s>>>(p, b.aos, w, pid);
  return cudaGetLastError();
}

// The FP64 sort (its records are too long for the sectors the binning moves).
template <typename R>
cudaError_t launch_tile_sort(R* arr[7], uint32_t* pid, int64_t n, const SortBuffers& b,
                             int nx, int ny, double x0, double y0, double inv_dx,
                             double inv_dy, int chunk, cudaStream_t s) {
  const int ntx = (nx + kTile - 1) / kTile;
  cudaError_t e = cudaMemsetAsync(b.counts, 0, sizeof(unsigned int) * b.ntiles, s);
  if (e != cudaSuccess) return e;
  const int block = 256;
  const int64_t want = (n + block - 1) / block;
  const int grid = static_cast<int>(want < 8192 ? (want > 0 ? want : 1) : 8192);
  k_tile_count<R><<<grid, block, 0, s>>>(arr[0], arr[1], n, nx, ny, ntx, R(x0), R(y0),
                                         R(inv_dx), R(inv_dy), b.counts);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_tile_scan<<<1, kScanThreads, 0, s>>>(b.counts, b.ntiles, b.starts, b.cursor, b.work,
                                          b.work_count, static_cast<unsigned int>(chunk), 0u,
                                          0u);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  Arrays7<R> srcp, dstp;
  for (int k = 0; k < 7; ++k) {
    srcp.p[k] = arr[k];
    dstp.p[k] = arr[k] ? static_cast<R*>(b.tmp[k]) : nullptr;
  }
  k_tile_scatter<R><<<grid, block, 0, s>>>(srcp, dstp, pid, b.tmp_pid, n, nx, ny, ntx, R(x0),
                                           R(y0), R(inv_dx), R(inv_dy), b.cursor);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // back into the caller's arrays, in cell order inside each tile
  k_cell_scatter<R><<<b.ntiles, kCellThreads, 0, s>>>(dstp, srcp, b.tmp_pid, pid, b.starts, nx,
                                                      ny, R(x0), R(y0), R(inv_dx), R(inv_dy));
  return cudaGetLastError();
}

template cudaError_t launch_tile_sort<double>(double* [7], uint32_t*, int64_t,
                                              const SortBuffers&, int, int, double, double,
                                              double, double, int, cudaStream_t);

}  // namespace prad
