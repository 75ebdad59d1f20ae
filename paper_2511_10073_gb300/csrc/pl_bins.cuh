// Bin rows of the augmented graph as the transpose of the cells' window
// blocks (Sec. V, bin virtual nodes; the column-free storage of the bin
// hints follows the Laplacian-sparsification outlook of Sec. IX).
//
// A hint cell i in bin b' stores the weights of its detection window as W
// slots, slot s = (dy + hy) (2 hx + 1) + (dx + hx) for the window bin
// b' + (dx, dy).  The row of bin node b therefore holds, for every slot s whose
// source bin b' = b - (dx_s, dy_s) lies in the grid, the cells of b''s hint
// bucket with weight w_s(i).  No entry of a bin row is stored: its sums are
// formed from the bucket lists and the window blocks.
//
// The hint cells of each bucket (ascending id) are cut into chunks of
// kBinChunk; a warp per chunk forms, for every slot, the chunk's double-float
// sum (exact products for the filter, weights and positive weights for the
// degrees), each lane over its cells in order and then a fixed tree over the
// lanes, so every partial is a fixed function of the inputs.  The row of bin b adds, slot by slot, the
// partials of that slot's source-bucket chunks (bin_row_chunks).
#pragma once

#include "pl_common.cuh"

namespace pl {

// 4 warps a CTA, each on its own chunks: a CTA of 8 K registers fits beside
// the refinement product's short-row kernel held to 5 CTAs per SM, so the bin
// rows run beside the short rows instead of after them
constexpr int kBinThreads = 128;
constexpr int kBinPer = 8;         // hint cells per lane
constexpr int kBinChunk = 32 * kBinPer;  // hint cells per chunk (one warp)

struct BinGeo {
  int nbx, nby, hx, hy, W;  // bin grid, window half widths, slots per window
  int NB;
};

// Offset (dx, dy) of slot s of a window.
__device__ __forceinline__ void slot_off(const BinGeo &B, int s, int *dx, int *dy) {
  const int wx = 2 * B.hx + 1;
  *dy = s / wx - B.hy;
  *dx = s % wx - B.hx;
}


template <int WT>
__device__ __forceinline__ float bw_load(const void *bw, size_t k) {
  if (WT == 0) return reinterpret_cast<const float *>(bw)[k];
  return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short *>(bw)[k] << 16);
}

// Per chunk and slot, a float4 partial: with DEG, (sum w, sum of positive w)
// as two double-floats; otherwise (sum w x_i, sum w y_i) with exact products.
// A warp per chunk: lane j takes the chunk's cells j, j + 32, ... (all their
// loads in flight together); per slot, each lane adds its cells in order and
// a fixed tree adds the lanes, so every partial is a fixed function of the
// inputs.  bwq: the chunks' window blocks, slot-major within a chunk (slot t
// of the chunk's i-th cell at (c W + t) kBinChunk + i), so each slot is read
// as consecutive weights; x: coordinates of every node (the cells' ones are
// gathered).  The chunk count is bchunk[NB];
// the grid may be any size.
// Slots t0 .. t0 + NT - 1 of chunk c with the partials of all of them
// reduced over the warp at once (warp_rs_df): value 2 t of the slot group is
// the first double-float of slot t0 + t, value 2 t + 1 the second.  The same
// sums, bit for bit, as a warp_sum_df per slot and value.  CUT: stop after the
// nu of a lane's kBinPer places that hold cells (the same in every lane; places
// beyond would only add zeros).
template <int WT, bool DEG, int NT, bool CUT>
__device__ __forceinline__ void bin_slot_group(const void *bwq, size_t wbase, const bool *cv, int nu,
                                               const float2 *xi, float4 *part, size_t pbase, int t0) {
  const int lane = threadIdx.x & 31;
  dfl v[2 * NT];
#pragma unroll
  for (int t = 0; t < NT; ++t) {
    float w[kBinPer];
#pragma unroll
    for (int u = 0; u < kBinPer; ++u)
      w[u] = cv[u] ? bw_load<WT>(bwq, wbase + (size_t)(t0 + t) * kBinChunk + lane + 32 * u) : 0.f;
    dfl a{0.f, 0.f}, e{0.f, 0.f};
#pragma unroll
    for (int u = 0; u < kBinPer; ++u) {
      if (CUT && u >= nu) break;
      if (DEG) {
        df_add(a, w[u]);
        if (w[u] > 0.f) df_add(e, w[u]);
      } else {
        df_add_prod(a, w[u], xi[u].x);
        df_add_prod(e, w[u], xi[u].y);
      }
    }
    v[2 * t] = a;
    v[2 * t + 1] = e;
  }
  int pos = 0, cnt = 2 * NT;
  warp_rs_df<2 * NT, 16>(v, pos, cnt);
  if (cnt == 1) {
    const dfl r = df_norm(v[0]);
    reinterpret_cast<float2 *>(part)[(pbase + t0 + (pos >> 1)) * 2 + (pos & 1)] = make_float2(r.hi, r.lo);
  }
}

// Chunk c's partials (a warp).  NS: the window is known to have 9 slots, or 1 (0:
// any number); FIVE: nine are taken as groups of five and four.
template <int WT, bool DEG, int NS, bool FIVE = false>
__device__ __forceinline__ void bin_chunk(const BinGeo &B, const int32_t *bchunk,
                                          const int32_t *cown, const int64_t *boff,
                                          const uint32_t *blist, const void *bwq,
                                          const float2 *x, float4 *part, long long c) {
  const int lane = threadIdx.x & 31;
  const int b = cown[c];
  const long long k0 = boff[2 * b] + (long long)(c - bchunk[b]) * kBinChunk;
  const long long k1 = boff[2 * b + 1];
  uint32_t kp[kBinPer];  // list positions (below 2^31: movable cells)
  bool cv[kBinPer];
  uint32_t ci[kBinPer];
#pragma unroll
  for (int u = 0; u < kBinPer; ++u) {
    kp[u] = (uint32_t)(k0 + lane + 32LL * u);
    cv[u] = k0 + lane + 32LL * u < k1;
    ci[u] = (!DEG && cv[u]) ? blist[kp[u]] : 0u;
  }
  float2 xi[kBinPer];
#pragma unroll
  for (int u = 0; u < kBinPer; ++u) xi[u] = (!DEG && cv[u]) ? x[ci[u]] : make_float2(0.f, 0.f);
  const size_t wbase = (size_t)c * B.W * kBinChunk;
  const int nu = (int)((min(k1 - k0, (long long)kBinChunk) + 31) / 32);
  const size_t pb = (size_t)c * B.W;
  if (NS == 1) {  // fewer than 20 bins
    bin_slot_group<WT, DEG, 1, true>(bwq, wbase, cv, nu, xi, part, pb, 0);
    return;
  }
  if (NS == 9) {  // the 3 x 3 window of 20 to 39 bins: mostly full chunks
    // (three groups of three in a rolled loop; groups of five and four spill when
    // unrolled, and hold in 64 registers only alone in their kernel and rolled)
    if (FIVE) {
#pragma unroll 1
      for (int t0 = 0; t0 < 9; t0 += 5) {
        if (t0 == 0) bin_slot_group<WT, DEG, 5, false>(bwq, wbase, cv, nu, xi, part, pb, 0);
        else bin_slot_group<WT, DEG, 4, false>(bwq, wbase, cv, nu, xi, part, pb, 5);
      }
      return;
    }
#pragma unroll 1
    for (int t0 = 0; t0 < 9; t0 += 3)
      bin_slot_group<WT, DEG, 3, false>(bwq, wbase, cv, nu, xi, part, pb, t0);
    return;
  }
  // other windows: groups of five slots, the rest in one more group, each one
  // reduce-scatter instead of ten butterflies; finer bins hold few cells, so
  // their chunks stop at the last place that holds one.  (5 x 5 windows of 64 x
  // 64 bins, 20k cells, a refinement round of eight products: 754 -> 652 us.
  // The stop cost the 3 x 3 window of 2.2M cells 4% of its round.)
  int t0 = 0;
  for (; t0 + 5 <= B.W; t0 += 5)
    bin_slot_group<WT, DEG, 5, true>(bwq, wbase, cv, nu, xi, part, pb, t0);
  switch (B.W - t0) {
    case 4: bin_slot_group<WT, DEG, 4, true>(bwq, wbase, cv, nu, xi, part, pb, t0); break;
    case 3: bin_slot_group<WT, DEG, 3, true>(bwq, wbase, cv, nu, xi, part, pb, t0); break;
    case 2: bin_slot_group<WT, DEG, 2, true>(bwq, wbase, cv, nu, xi, part, pb, t0); break;
    case 1: bin_slot_group<WT, DEG, 1, true>(bwq, wbase, cv, nu, xi, part, pb, t0); break;
  }
}

template <int WT, bool DEG, int NS>
__global__ void __launch_bounds__(kBinThreads, 8) k_bin_partials(BinGeo B, const int32_t *bchunk,
                                                              const int32_t *cown,
                                                              const int64_t *boff,
                                                              const uint32_t *blist,
                                                              const void *bwq, const float2 *x,
                                                              float4 *part) {
  const int nchunk = bchunk[B.NB];
  for (long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; c < nchunk;
       c += ((long long)gridDim.x * blockDim.x) >> 5)
    // FP32 weights: more of the longer loads in flight beside the short rows (filter
    // of 2.2M cells, eight powers: 1471 us by threes, 1454 us by five and four;
    // BF16: 1401 and 1424 us)
    bin_chunk<WT, DEG, NS, WT == 0 && !DEG>(B, bchunk, cown, boff, blist, bwq, x, part, c);
}

template <bool DEG>
inline cudaError_t launch_bin_partials(int wt, int grid, cudaStream_t s, const BinGeo &B,
                                       const int32_t *bchunk, const int32_t *cown,
                                       const int64_t *boff, const uint32_t *blist,
                                       const void *bwq, const float2 *x, float4 *part) {
  // (one slot in a kernel of its own: 56 registers and no spills beside the short
  // rows; eight powers of 320k cells on 16 x 16 bins, FP32, 271 -> 266 us)
  const int ns = B.W == 9 || B.W == 1 ? B.W : 0;
  auto k = wt == 2 ? (ns == 9 ? k_bin_partials<1, DEG, 9> : ns ? k_bin_partials<1, DEG, 1> : k_bin_partials<1, DEG, 0>)
                   : (ns == 9 ? k_bin_partials<0, DEG, 9> : ns ? k_bin_partials<0, DEG, 1> : k_bin_partials<0, DEG, 0>);
  k<<<grid, kBinThreads, 0, s>>>(B, bchunk, cown, boff, blist, bwq, x, part);
  return cudaGetLastError();
}

// Sums of bin b's row by the lanes of one warp, straight from the chunk
// partials: for every slot s whose source bucket b - offset(s) lies in the
// grid, the partials of slot s of that bucket's chunks.  The items (slot by
// slot, each bucket's chunks in order; slots in groups of 32) are dealt to
// the lanes in turn, then a fixed tree adds the lanes, so the sums are a fixed
// function of the partials.  Returns the two double-floats of the partials'
// layout.
__device__ __forceinline__ void bin_row_chunks(const BinGeo &B, int b, const int32_t *bchunk,
                                               const float4 *part, dfl *a, dfl *e) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int bx = b % B.nbx, by = b / B.nbx, wx = 2 * B.hx + 1;
  dfl sa{0.f, 0.f}, se{0.f, 0.f};
  for (int s0 = 0; s0 < B.W; s0 += 32) {
    // lane j: the chunk range of slot s0 + j's source bucket
    const int s = s0 + lane;
    int c0 = 0, n = 0;
    if (s < B.W) {
      const int sx = bx - (s % wx - B.hx), sy = by - (s / wx - B.hy);
      if (sx >= 0 && sy >= 0 && sx < B.nbx && sy < B.nby) {
        const int bb = sy * B.nbx + sx;
        c0 = bchunk[bb];
        n = bchunk[bb + 1] - c0;
      }
    }
    int inc = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(full, inc, d);
      if (lane >= d) inc += t;
    }
    const int exc = inc - n, tot = __shfl_sync(full, inc, 31);
    constexpr int kU = 4;  // items a lane loads at once
    for (int i0 = 0; i0 < tot; i0 += 32 * kU) {
      float4 q[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int i = i0 + 32 * u + lane;
        // the lane whose range holds item i: the last one starting at or before it
        int lo = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
          if (__shfl_sync(full, exc, lo + step) <= i) lo += step;
        const int cj = __shfl_sync(full, c0, lo), ej = __shfl_sync(full, exc, lo);
        q[u] = i < tot ? __ldcg(&part[(size_t)(cj + i - ej) * B.W + s0 + lo])
                       : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (i0 + 32 * u + lane < tot) {
          df_add_df(sa, dfl{q[u].x, q[u].y});
          df_add_df(se, dfl{q[u].z, q[u].w});
        }
      }
    }
  }
  *a = warp_sum_df(sa);
  *e = warp_sum_df(se);
}

// First chunk of each bin's hint bucket and the bucket of each chunk, by one
// block: a thread per bin, 1024 at a time, writes its bucket's chunks, those of a
// bin with more than kBinChunksLane the whole warp (hint build of 2.2M cells in one
// bin, 8600 chunks: 605 -> 592 us).
constexpr int kBinsOneBlock = 16384;
constexpr int kBinChunksLane = 64;
static __global__ void __launch_bounds__(1024) k_bin_chunks(int NB, const int64_t *boff,
                                                            int32_t *bchunk, int32_t *cown) {
  __shared__ int ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = 0;
  for (int b0 = 0; b0 < NB; b0 += 1024) {
    const int b = b0 + (int)threadIdx.x;
    const int n = b < NB ? (int)((boff[2 * b + 1] - boff[2 * b] + kBinChunk - 1) / kBinChunk) : 0;
    int x = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
      int t = ws[lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, t, d);
        if (lane >= d) t += y;
      }
      ws[lane] = t;
    }
    __syncthreads();
    const int c0 = carry + (w ? ws[w - 1] : 0) + x - n;
    if (b < NB) bchunk[b] = c0;
    const bool wide = n > kBinChunksLane;
    if (!wide)
      for (int c = 0; c < n; ++c) cown[c0 + c] = b;
    for (unsigned t = __ballot_sync(0xffffffffu, wide); t; t &= t - 1) {
      const int src = __ffs(t) - 1;
      const int m = __shfl_sync(0xffffffffu, n, src), at = __shfl_sync(0xffffffffu, c0, src);
      for (int c = lane; c < m; c += 32) cown[at + c] = b - lane + src;
    }
    carry += ws[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) bchunk[NB] = carry;
}

// The same for more bins: counts, to be scanned into bchunk.
static __global__ void k_bin_chunk_count(int NB, const int64_t *boff, int32_t *cnt) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < NB; b += gridDim.x * blockDim.x) {
    const long long n = boff[2 * b + 1] - boff[2 * b];
    cnt[b] = (int32_t)((n + kBinChunk - 1) / kBinChunk);
  }
}

// Bucket of each chunk: a thread per chunk finds the last bucket whose first
// chunk is at or before it (bchunk is nondecreasing).
static __global__ void k_chunk_bins(int NB, long long ncmax, const int32_t *bchunk, int32_t *cown) {
  const int nchunk = bchunk[NB];
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncmax && c < nchunk;
       c += (long long)gridDim.x * blockDim.x) {
    int lo = 0, hi = NB - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (bchunk[mid] <= c) lo = mid;
      else hi = mid - 1;
    }
    cown[c] = lo;
  }
}

}  // namespace pl
