// A2 + A3: area hints and the signed Laplacian, GPU-side (Sec. V).
//
//  * macro virtual node v_m joined to every movable cell overlapping macro m
//    by w = -exp(-maxRatio_{i,m}) * baseWeight_i;
//  * bin virtual node v_b joined to every movable cell whose centre bin lies
//    in the detection window of b by w = -exp(-maxRatio_{i,b}) phi_b
//    baseWeight_i, phi_b = 2 sigmoid(mu (D_b - C_b)) - 1;
//  * L_hint = D - A with signed D_ii; lambda_up = max_i (D_ii + sum_j |w_ij|)
//    (Gershgorin), which equals max_i 2 * (sum of positive w_ij).
// Decisions (bin of a centre, overlap) are FP32 with one stated operation
// sequence; D_b and phi_b are FP64; degree sums are double-float.  Edge
// weights are the FP64 value of the definition rounded once to the storage
// type: for BF16 storage an FP32 value (exponent argument carried in FP64)
// rounds to the same bf16 except within a few FP32 ulps of a bf16 rounding
// midpoint, where the FP64 value is computed; for FP32 storage a double-float
// value (about 2^-40) decides the rounding, except within its error bound of an
// FP32 rounding midpoint.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "pl_bins.cuh"
#include "pl_internal.h"

namespace pl {

#define TRY(x)                                       \
  do {                                               \
    cudaError_t e_ = (x);                            \
    if (e_ != cudaSuccess) return cuda_fail(e_, #x); \
  } while (0)

constexpr int kMaxWin = 31;  // detection window at most 31 x 31 bins (a window row fits a warp)

struct HintGeo {
  float xlf, ylf, sxf, syf;      // bin decision: floor((x - xl) * sx)
  float gxf, gyf, gsxf, gsyf;    // macro grid bucket of a centre
  double xl, yl, wb, hb, iwb2, ihb2;  // bin centres; 2 / w_b, 2 / h_b
  float xlh, xll, ylh, yll;          // x_l, y_l as double-floats
  float iwh, iwl, ihh, ihl;          // 2 / w_b, 2 / h_b as double-floats
  float tol;                         // relative error bound of a double-float bin weight
  int nbx, nby, hx, hy, gnx, gny;
  int32_t C, Pm, S, Mm;
  int64_t Nst, mv0, bn0, N;
};

__device__ __forceinline__ int bin_of(float x, float xl, float sc, int nb) {
  float t = __fmul_rn(__fadd_rn(x, -xl), sc);
  float f = floorf(t);
  if (!(f >= 0.f)) return 0;
  if (f > (float)(nb - 1)) return nb - 1;
  return (int)f;
}
__device__ __forceinline__ bool overlaps(float x, float y, float w, float h, float xm, float ym,
                                         float wm, float hm) {
  float dx = fabsf(__fadd_rn(x, -xm)), dy = fabsf(__fadd_rn(y, -ym));
  return dx < __fmul_rn(0.5f, __fadd_rn(w, wm)) && dy < __fmul_rn(0.5f, __fadd_rn(h, hm));
}
__device__ __forceinline__ int grid_of(float x, float x0, float sc, int n) { return bin_of(x, x0, sc, n); }

// BF16 storage rounds the FP64 weight of the definition once.  The fast FP32
// value is within a few FP32 ulps of it (FP32 exp: 2 ulps, three roundings),
// so it rounds to the same bf16 unless it lies within kNearTie FP32 ulps of a
// bf16 rounding midpoint (low 16 bits near 0x8000); only then the weight is
// recomputed in FP64 with the exact operation sequence of the definition.
constexpr int kNearTie = 8;
__device__ __forceinline__ bool near_bf16_tie(float v) {
  int d = (int)(__float_as_uint(v) & 0xffffu) - 0x8000;
  return d >= -kNearTie && d <= kNearTie;
}
// -((e^{-maxRatio} * phi) * bw) for cell centre (x, y) and bin (xx, yy), FP64.
// Kept out of line: the fast path must not carry any of its FP64 work.
__device__ __noinline__ double bin_w_exact(float x, float y, int xx, int yy, const HintGeo &G, double phi,
                              double bw) {
  double xb = __dadd_rn(G.xl, __dmul_rn((double)xx + 0.5, G.wb));
  double yb = __dadd_rn(G.yl, __dmul_rn((double)yy + 0.5, G.hb));
  double dx = fabs(__dadd_rn((double)x, -xb)), dy = fabs(__dadd_rn((double)y, -yb));
  double r = fmax(__ddiv_rn(dx, __dmul_rn(G.wb, 0.5)), __ddiv_rn(dy, __dmul_rn(G.hb, 0.5)));
  double t = __dmul_rn(__dmul_rn(exp_cw(-r), phi), bw);
  return -t;
}
// -(e^{-maxRatio} * bw) for a cell centre and a macro (centre xm, ym; size wm, hm).
__device__ __noinline__ double macro_w_exact(float x, float y, float xm, float ym, float wm, float hm,
                                double bw) {
  double dx = fabs(__dadd_rn((double)x, -(double)xm)), dy = fabs(__dadd_rn((double)y, -(double)ym));
  double r = fmax(__ddiv_rn(dx, __dmul_rn((double)wm, 0.5)), __ddiv_rn(dy, __dmul_rn((double)hm, 0.5)));
  return -__dmul_rn(exp_cw(-r), bw);
}

__device__ __forceinline__ float load_w(const void *wbuf, int wdtype, uint64_t k) {
  if (wdtype == PL_W_BF16) return bf16_to_f(reinterpret_cast<const uint16_t *>(wbuf)[k]);
  return reinterpret_cast<const float *>(wbuf)[k];
}
__device__ __forceinline__ void copy_w(void *dst, const void *src, int wdtype, uint64_t kd,
                                       uint64_t ks) {
  if (wdtype == PL_W_BF16)
    reinterpret_cast<uint16_t *>(dst)[kd] = reinterpret_cast<const uint16_t *>(src)[ks];
  else
    reinterpret_cast<float *>(dst)[kd] = reinterpret_cast<const float *>(src)[ks];
}

// Cells are taken in tiles of 2^tsh consecutive ids (hint_tile_shift) by the stable counting
// sorts (bin buckets, macro lists).
constexpr int kMaxSmemBuckets = 12288;
constexpr int kMacroSlots = 8;        // macros one cell may overlap in the tiled macro lists
constexpr int kMaxSmemMacros = 12288;  // macros of the tiled macro lists (runs and masks in smem)

// --------------------------------------------------------- H1: cells
__global__ void k_hint_cells(HintGeo G, const float2 *xy, const uint8_t *ckind,
                             const uint8_t *hflag, const float *cw, const float *ch,
                             const int64_t *gptr, const uint32_t *glist, const float4 *ggeo,
                             int32_t *cell_bin, int32_t *n_ovl, int32_t *bcnt, int32_t *mcnt,
                             int32_t *mtc, int ntile, int tsh, int32_t *cmem, int *status) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G.C; i += gridDim.x * blockDim.x) {
    // the cell's inputs in flight together, before the kind test
    const uint8_t kd = ckind[i];
    float2 p = xy[i];
    const bool hint = hflag[i] != 0;
    const float cwi = cw[i], chi = ch[i];
    if (kd != 0) {
      cell_bin[i] = -1;
      n_ovl[i] = 0;
      continue;
    }
    if (!isfinite(p.x) || !isfinite(p.y)) {
      flag(status, ST_NONFINITE);
      p = make_float2(0.f, 0.f);
    }
    int bx = bin_of(p.x, G.xlf, G.sxf, G.nbx), by = bin_of(p.y, G.ylf, G.syf, G.nby);
    int b = by * G.nbx + bx;
    cell_bin[i] = b;
    if (bcnt) atomicAdd(&bcnt[2 * b + (hint ? 0 : 1)], 1);
    int n = 0;
    if (hint) {
      int kx = grid_of(p.x, G.gxf, G.gsxf, G.gnx), ky = grid_of(p.y, G.gyf, G.gsyf, G.gny);
      long long k = (long long)ky * G.gnx + kx;
      for (long long q = gptr[k]; q < gptr[k + 1]; ++q) {
        const float4 mg = ggeo[q];
        if (overlaps(p.x, p.y, cwi, chi, mg.x, mg.y, mg.z, mg.w)) {
          const uint32_t m = glist[q];
          if (mtc) {
            atomicAdd(&mtc[(long long)m * ntile + (i >> tsh)], 1);
            if (n < kMacroSlots) cmem[(long long)i * kMacroSlots + n] = (int32_t)m;
          } else {
            atomicAdd(&mcnt[m], 1);
          }
          ++n;
        }
      }
      if (mtc && n > kMacroSlots) flag(status, ST_MANY_OVL);
    }
    n_ovl[i] = n;
  }
}

// Cells overlapping each macro (the macro virtual rows), unordered here and
// sorted by cell id afterwards.
__global__ void k_macro_scatter(HintGeo G, const float2 *xy, const uint8_t *ckind,
                                const uint8_t *hflag, const float *cw, const float *ch,
                                const int64_t *gptr, const uint32_t *glist, const float4 *ggeo,
                                int32_t *mcur, uint32_t *mlist) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G.C; i += gridDim.x * blockDim.x) {
    if (ckind[i] != 0 || !hflag[i]) continue;
    float2 p = xy[i];
    if (!isfinite(p.x) || !isfinite(p.y)) p = make_float2(0.f, 0.f);
    int kx = grid_of(p.x, G.gxf, G.gsxf, G.gnx), ky = grid_of(p.y, G.gyf, G.gsyf, G.gny);
    long long k = (long long)ky * G.gnx + kx;
    const float cwi = cw[i], chi = ch[i];
    for (long long q = gptr[k]; q < gptr[k + 1]; ++q) {
      const float4 mg = ggeo[q];
      if (overlaps(p.x, p.y, cwi, chi, mg.x, mg.y, mg.z, mg.w))
        mlist[atomicAdd(&mcur[glist[q]], 1)] = (uint32_t)i;
    }
  }
}

// Macro lists in ascending cell id without a sort: a CTA per tile of 2^tsh
// cells, counts per (macro, tile) macro-major and each cell's macros (at most
// kMacroSlots) from k_hint_cells.  In rounds of blockDim cells the warps take
// turns; inside a turn the lanes mark their macros in a per-macro lane mask,
// and a membership's place is its macro's tile start (loaded before the
// turns), the macro's run so far and the number of lower lanes marked.
__global__ void __launch_bounds__(256, 4) k_macro_tile_scatter(int32_t C, const int32_t *n_ovl,
                                                            const int32_t *cmem, int Mm,
                                                            int ntile, int tsh,
                                                            const int64_t *off,
                                                            uint32_t *mlist) {
  extern __shared__ uint32_t lmask[];  // [Mm] lane masks, then [Mm] runs (at most 4096)
  uint16_t *run = reinterpret_cast<uint16_t *>(lmask + Mm);
  for (int k = threadIdx.x; k < Mm; k += blockDim.x) {
    run[k] = 0;
    lmask[k] = 0u;
  }
  __syncthreads();
  const int t = blockIdx.x, i0 = t << tsh, i1 = min(C, i0 + (1 << tsh));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  // a round's cell memberships are loaded during the round before
  int nn = i0 + (int)threadIdx.x < i1 ? min(n_ovl[i0 + threadIdx.x], kMacroSlots) : 0;
  int32_t mn[kMacroSlots];
#pragma unroll
  for (int j = 0; j < kMacroSlots; ++j)
    mn[j] = j < nn ? cmem[(long long)(i0 + threadIdx.x) * kMacroSlots + j] : 0;
  for (int base = i0; base < i1; base += blockDim.x) {
    const int i = base + threadIdx.x;
    // n_ovl is 0 for cells other than movable hint cells
    const int n = nn;
    int32_t mk[kMacroSlots];
    long long tst[kMacroSlots];
#pragma unroll
    for (int j = 0; j < kMacroSlots; ++j) {
      mk[j] = mn[j];
      tst[j] = j < n ? off[(long long)mk[j] * ntile + t] : 0;
    }
    const int inext = i + (int)blockDim.x;
    nn = inext < i1 ? min(n_ovl[inext], kMacroSlots) : 0;
#pragma unroll
    for (int j = 0; j < kMacroSlots; ++j)
      mn[j] = j < nn ? cmem[(long long)inext * kMacroSlots + j] : 0;
    // places within the tile's runs, by turns in shared memory; the stores
    // wait for the tile starts only after the turns
    int rel[kMacroSlots];
    for (int w = 0; w < nw; ++w) {
      if (wid == w) {
#pragma unroll
        for (int j = 0; j < kMacroSlots; ++j)
          if (j < n) atomicOr(&lmask[mk[j]], 1u << lane);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kMacroSlots; ++j)
          rel[j] = j < n ? (int)run[mk[j]] + __popc(lmask[mk[j]] & lt) : 0;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < kMacroSlots; ++j) {
          if (j < n) {
            const uint32_t msk = lmask[mk[j]];
            if (msk && lane == __ffs(msk) - 1) {
              run[mk[j]] = (uint16_t)(run[mk[j]] + __popc(msk));
              lmask[mk[j]] = 0u;
            }
          }
        }
        __syncwarp();
      }
      __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kMacroSlots; ++j)
      if (j < n) mlist[tst[j] + rel[j]] = (uint32_t)i;
  }
}

// Bin buckets: key 2*bin + (baseWeight == 0).  A stable counting sort over
// tiles of 2^tsh consecutive cells writes every bucket in ascending cell id
// directly (no sort).  Counts per (bucket, tile), bucket-major.

__device__ __forceinline__ int bucket_of(const uint8_t *hflag, const int32_t *cell_bin, int i) {
  return 2 * cell_bin[i] + (hflag[i] ? 0 : 1);
}

__global__ void __launch_bounds__(256) k_bin_tile_count(int32_t C, int nbk, int ntile, int tsh,
                                                        const uint8_t *ckind,
                                                        const uint8_t *hflag,
                                                        const int32_t *cell_bin, int32_t *cnt) {
  extern __shared__ int32_t sc[];
  for (int k = threadIdx.x; k < nbk; k += blockDim.x) sc[k] = 0;
  __syncthreads();
  const int t = blockIdx.x, i0 = t << tsh, i1 = min(C, i0 + (1 << tsh));
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x)
    if (ckind[i] == 0) atomicAdd(&sc[bucket_of(hflag, cell_bin, i)], 1);
  __syncthreads();
  for (int k = threadIdx.x; k < nbk; k += blockDim.x) cnt[(long long)k * ntile + t] = sc[k];
}

// Rounds of blockDim cells; inside a round the warps take turns (so equal
// buckets keep cell order), lanes of a warp rank themselves with match_any.
__global__ void __launch_bounds__(256) k_bin_tile_scatter(int32_t C, int nbk, int ntile, int tsh,
                                                          const uint8_t *ckind,
                                                          const uint8_t *hflag,
                                                          const int32_t *cell_bin,
                                                          const int64_t *off, uint32_t *blist) {
  extern __shared__ int32_t run[];
  for (int k = threadIdx.x; k < nbk; k += blockDim.x) run[k] = 0;
  __syncthreads();
  const int t = blockIdx.x, i0 = t << tsh, i1 = min(C, i0 + (1 << tsh));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  for (int base = i0; base < i1; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const bool mv = i < i1 && ckind[i] == 0;
    const int key = mv ? bucket_of(hflag, cell_bin, i) : -1 - lane;
    const long long tst = mv ? off[(long long)key * ntile + t] : 0;  // loaded before the turns
    int rel = 0;  // place within the tile's run of the bucket (the store waits for tst after the turns)
    for (int w = 0; w < nw; ++w) {
      if (wid == w) {
        unsigned grp = __match_any_sync(0xffffffffu, key);
        int leader = __ffs(grp) - 1;
        int before = 0;
        if (mv && lane == leader) {
          before = run[key];
          run[key] = before + __popc(grp);
        }
        before = __shfl_sync(0xffffffffu, before, leader);
        rel = before + __popc(grp & lt);
      }
      __syncthreads();
    }
    if (mv) blist[tst + rel] = (uint32_t)i;
  }
}

// The same lists without turns, for grids whose per-warp counters fit shared
// memory (20 nbk bytes): in each round every warp ranks its lanes by key with
// match_any and writes its group sizes to its own row of counters; after a
// barrier a cell's place is the key's run so far, plus the same key's cells in
// the round's lower warps, plus its lower lanes of the same key, which is its
// place in cell order.  Two barriers per round instead of one per warp.
__global__ void __launch_bounds__(256) k_bin_tile_scatter_wc(int32_t C, int nbk, int ntile, int tsh,
                                                             const uint8_t *ckind,
                                                             const uint8_t *hflag,
                                                             const int32_t *cell_bin,
                                                             const int64_t *off, uint32_t *blist) {
  extern __shared__ int32_t run[];  // [nbk] runs, then uint16 [8][nbk] counts of the round
  uint16_t *wc = reinterpret_cast<uint16_t *>(run + nbk);
  for (int k = threadIdx.x; k < nbk; k += blockDim.x) run[k] = 0;
  for (int k = threadIdx.x; k < 8 * nbk; k += blockDim.x) wc[k] = 0;
  __syncthreads();
  const int t = blockIdx.x, i0 = t << tsh, i1 = min(C, i0 + (1 << tsh));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  for (int base = i0; base < i1; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const bool mv = i < i1 && ckind[i] == 0;
    const int key = mv ? bucket_of(hflag, cell_bin, i) : -1 - lane;
    const long long tst = mv ? off[(long long)key * ntile + t] : 0;
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    const bool lead = mv && lane == __ffs(grp) - 1;
    if (lead) wc[wid * nbk + key] = (uint16_t)__popc(grp);
    __syncthreads();
    int rel = 0;
    if (mv) {
      rel = run[key] + __popc(grp & lt);
      for (int w = 0; w < wid; ++w) rel += wc[w * nbk + key];
    }
    __syncthreads();  // the round's counters are read
    if (lead) {
      atomicAdd(&run[key], __popc(grp));  // warps of the round may share a key
      wc[wid * nbk + key] = 0;
    }
    __syncwarp();
    if (mv) blist[tst + rel] = (uint32_t)i;
  }
}

__global__ void k_bucket_starts(int nbk, int ntile, const int64_t *off, int64_t *boff) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= nbk; k += gridDim.x * blockDim.x)
    boff[k] = off[(long long)k * ntile];
}

// Fallback for bin grids too large for the shared-memory counters: atomic
// scatter, then the buckets are sorted.
__global__ void k_bin_scatter_atomic(int32_t C, const uint8_t *ckind, const uint8_t *hflag,
                                     const int32_t *cell_bin, int32_t *bcur, uint32_t *blist) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x)
    if (ckind[i] == 0) blist[atomicAdd(&bcur[bucket_of(hflag, cell_bin, i)], 1)] = (uint32_t)i;
}

// ------------------------------------------------ H5: bin density and phi
// D_b: FP64 sum of the cell areas w*h of bin b's sequence (its hint bucket
// then its other bucket, each ascending), in the blocked order: blocks of 64
// added left to right, block sums summed the same way, recursively.  A CTA per
// bin forms every level in parallel; level l of bin b lives at offset
// floor(start_{l-1}/64) + b of that level's region, so bins never overlap.
constexpr int kMaxLevels = 8;
struct LevelBufs {
  double *base[kMaxLevels];
};

// Cell areas w h in FP64 (exact: a product of two floats fits a double), once
// per netlist, so that the density sums take one FP64 operation per cell.
__global__ void k_cell_area(int32_t C, const float *cw, const float *ch, double *area) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x)
    area[i] = __dmul_rn((double)cw[i], (double)ch[i]);
}

// A_mov(b) as a blocked FP64 sum: the bin's cells (hint cells ascending,
// then the others ascending) in blocks of 64 added left to right, the block
// sums blocked again, until at most 64 values remain, which are added left to
// right.  Level L of bin b reads len_L(b) values starting at st_L(b) (level
// 0: cell areas through the bucket list) and writes its block sums to
// out_L(b) = st_L(b) / 64 + b onwards; these ranges are disjoint and
// increasing in b, so every block of every bin is one thread of one launch.
struct DensLevel {
  int64_t st, len, out;
};
__device__ __forceinline__ DensLevel dens_level(const int64_t *boff, int b, int L) {
  DensLevel d;
  d.st = boff[2 * b];
  d.len = boff[2 * b + 2] - d.st;
  d.out = d.st / 64 + b;
  for (int l = 0; l < L; ++l) {
    d.st = d.out;
    d.len = (d.len + 63) / 64;
    d.out = d.st / 64 + b;
  }
  return d;
}

__global__ void __launch_bounds__(256) k_dens_level(int NB, int L, const int64_t *boff,
                                                    const uint32_t *blist, const double *area,
                                                    const double *prev, double *out,
                                                    long long nidx) {
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < nidx;
       idx += (long long)gridDim.x * blockDim.x) {
    int lo = 0, hi = NB - 1;  // last bin with out_L(b) <= idx
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (dens_level(boff, mid, L).out <= idx) lo = mid; else hi = mid - 1;
    }
    const DensLevel d = dens_level(boff, lo, L);
    const int64_t j = idx - d.out;
    if (d.len <= 64 || j < 0 || j >= (d.len + 63) / 64) continue;
    const int64_t k0 = d.st + 64 * j, k1 = min(d.st + d.len, k0 + 64);
    double acc = 0.0;
    if (L == 0) {
      for (int64_t k = k0; k < k1; k += 16) {
        double a[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) a[q] = k + q < k1 ? area[blist[k + q]] : 0.0;
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (k + q < k1) acc = __dadd_rn(acc, a[q]);
      }
    } else {
      for (int64_t k = k0; k < k1; ++k) acc = __dadd_rn(acc, prev[k]);
    }
    out[idx] = acc;
  }
}

// Per bin: the last (at most 64-value) sum, D_b, C_b, phi_b and the hub row
// length (hint cells of the window bins).
__global__ void k_dens_final(HintGeo G, int nlev, const int64_t *boff, const uint32_t *blist,
                             const double *area, LevelBufs lv, const double *amac,
                             double abin, double cap, double mu, double *Db, double *Cb,
                             double *phi, float *phif, float *phil) {
  const int NB = G.nbx * G.nby;
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < NB; b += gridDim.x * blockDim.x) {
    int L = 0;
    DensLevel d = dens_level(boff, b, 0);
    while (d.len > 64 && L < nlev) {
      ++L;
      d = dens_level(boff, b, L);
    }
    const double *src = L ? lv.base[L - 1] : nullptr;
    double acc = 0.0;
    for (int64_t k = 0; k < d.len; k += 16) {
      double a[16];
#pragma unroll
      for (int q = 0; q < 16; ++q)
        a[q] = k + q < d.len ? (L == 0 ? area[blist[d.st + k + q]] : src[d.st + k + q])
                             : 0.0;
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (k + q < d.len) acc = __dadd_rn(acc, a[q]);
    }
    const double dd = __ddiv_rn(acc, abin);
    const double c = __ddiv_rn(__dmul_rn(cap, __dadd_rn(abin, -amac[b])), abin);
    const double t = __dmul_rn(mu, __dadd_rn(dd, -c));
    const double ph = __dadd_rn(__ddiv_rn(2.0, __dadd_rn(1.0, exp_cw(-t))), -1.0);
    Db[b] = dd;
    Cb[b] = c;
    phi[b] = ph;
    phif[b] = __double2float_rn(ph);
    phil[b] = __double2float_rn(ph - (double)__double2float_rn(ph));  // ph - phif
  }
}

__device__ __forceinline__ int win_count(int bx, int by, const HintGeo &G) {
  int nx = min(G.nbx - 1, bx + G.hx) - max(0, bx - G.hx) + 1;
  int ny = min(G.nby - 1, by + G.hy) - max(0, by - G.hy) + 1;
  return nx * ny;
}

// ------------------------------------------------- H6-H7: split layout
// The layout of a split matrix in three launches: every row's place follows
// from prefix sums over the rows of (short entries, hub entries, hub rows, hub
// chunks), formed together.  k_lay_sum adds them per block of kLayRows rows,
// k_lay_scan turns the block sums into offsets and totals (one block), and
// k_lay_apply recomputes its rows' lengths and writes everything that depends
// on them.  (As separate length, scan, pack and descriptor kernels this took
// 14 launches and two reads of sizes by the host.)
struct RowLen {
  uint32_t s;      // short-region length (0 for hub rows)
  uint64_t l, cl;  // hub-region length, chunked length of a hub row (st part + this matrix's part)
  bool hub;
};
struct LayIn {
  HintGeo G;
  const int32_t *cnt;  // static matrix: row lengths; nullptr: hint matrix
  const int64_t *srp;  // hint matrix: static row pointers
  const uint8_t *hflag;
  const int32_t *cell_bin, *n_ovl;
  const int64_t *moff;
  int may;  // static matrix: rows longer than this may become hub rows of the hint matrix
};
// Totals of a layout (device and host); may_*: static rows beyond LayIn::may
// that are no hub rows, and their entries; cell_*: short entries of the static
// matrix' blocks of cells' rows, in all and the most of one block.
struct LayTotals {
  unsigned long long s, l, may_entries, cell_sum;
  uint32_t f, c, may_rows, cell_max;
};

// Lengths of row v of a split matrix.  Static matrix: hub when longer than
// kLong.  Hint matrix: the stored hm part of each row (a hint cell's macro
// entries, a macro row's cells; bin rows store nothing, their sums come from
// the window blocks); a row is a hub row when it is a virtual node or its static
// entries, macro entries and window slots exceed kLong.
template <bool HINT>
__device__ __forceinline__ RowLen row_len(const LayIn &A, long long v) {
  const HintGeo &G = A.G;
  RowLen r{0u, 0ull, 0ull, false};
  if (v >= G.N) return r;
  if (!HINT) {
    const uint32_t sl = v < G.Nst ? (uint32_t)A.cnt[v] : 0u;
    r.hub = sl > (uint32_t)kLong;
    if (r.hub) r.l = r.cl = sl;
    else r.s = sl;
    return r;
  }
  // every load of the row is issued before any of them is looked at
  const bool st = v < G.Nst, cell = v < G.C, mac = v >= G.mv0 && v < G.bn0;
  const int64_t r0 = st ? A.srp[v] : 0, r1 = st ? A.srp[v + 1] : 0;
  const uint8_t hf = cell ? A.hflag[v] : 0;
  const int nov = cell ? A.n_ovl[v] : 0, b = cell ? A.cell_bin[v] : 0;
  const int64_t m0 = mac ? A.moff[v - G.mv0] : 0, m1 = mac ? A.moff[v - G.mv0 + 1] : 0;
  const long long sl = r1 - r0, hl = mac ? m1 - m0 : hf ? nov : 0;
  const bool virt = v >= G.mv0;
  // (the window slots in the grid matter, and are counted, only near the limit)
  long long ws = 0;
  if (hf && sl + hl <= kLong && sl + hl + (2 * G.hx + 1) * (2 * G.hy + 1) > kLong)
    ws = win_count(b % G.nbx, b / G.nbx, G);
  r.hub = virt || sl + hl + ws > kLong;
  if (r.hub) {
    r.l = (uint64_t)hl;
    r.cl = (uint64_t)(sl + hl);
  } else {
    r.s = (uint32_t)hl;
  }
  return r;
}
__device__ __forceinline__ uint32_t row_chunks(uint64_t cl) {
  return (uint32_t)((cl + kChunk - 1) / kChunk);  // none for a row without stored entries (bin rows)
}

constexpr int kLayPer = 8;                 // rows per lane (a warp: 256 consecutive rows)
constexpr int kLayRows = 256 * kLayPer;    // rows per block of 256 threads
struct LaySum {
  unsigned long long s, l;
  uint32_t f, c;
};

// This warp's sums over its rows (every lane gets them); sv, hubs: the lane's
// short lengths and hub bits.
template <bool HINT>
__device__ __forceinline__ LaySum warp_rows(const LayIn &A, long long v0, uint32_t *sv,
                                            uint32_t *hubs, unsigned long long *may_rows,
                                            unsigned long long *may_entries) {
  const int lane = threadIdx.x & 31;
  LaySum t{0ull, 0ull, 0u, 0u};
  *hubs = 0u;
#pragma unroll
  for (int k = 0; k < kLayPer; ++k) {
    const RowLen r = row_len<HINT>(A, v0 + 32 * k + lane);
    sv[k] = r.s;
    t.s += r.s;
    if (!HINT && v0 + 32 * k + lane < A.G.Nst && !r.hub && (int)r.s > A.may) {
      ++*may_rows;
      *may_entries += r.s;
    }
    if (r.hub) {
      *hubs |= 1u << k;
      t.l += r.l;
      t.f += 1u;
      t.c += row_chunks(r.cl);
    }
  }
  t.s = warp_sum(t.s);
  if (__any_sync(0xffffffffu, *hubs != 0u)) {
    t.l = warp_sum(t.l);
    t.f = warp_sum(t.f);
    t.c = warp_sum(t.c);
  }
  return t;
}

template <bool HINT>
__global__ void __launch_bounds__(256) k_lay_sum(LayIn A, LaySum *bsum, LayTotals *tot) {
  __shared__ LaySum w[8];
  uint32_t sv[kLayPer], hubs;
  unsigned long long mr = 0, me = 0;
  const int wid = threadIdx.x >> 5;
  const LaySum t = warp_rows<HINT>(A, (long long)blockIdx.x * kLayRows + wid * 32 * kLayPer, sv, &hubs, &mr, &me);
  if ((threadIdx.x & 31) == 0) w[wid] = t;
  if (!HINT) {
    mr = warp_sum(mr);
    if (mr) {  // the same in every lane
      me = warp_sum(me);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&tot->may_rows, (uint32_t)mr);
        atomicAdd(&tot->may_entries, me);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x) return;
  LaySum a = w[0];
  for (int k = 1; k < 8; ++k) {
    a.s += w[k].s;
    a.l += w[k].l;
    a.f += w[k].f;
    a.c += w[k].c;
  }
  bsum[blockIdx.x] = a;
  if (!HINT && (blockIdx.x + 1LL) * kLayRows <= A.G.C) {
    atomicAdd(&tot->cell_sum, a.s);
    atomicMax(&tot->cell_max, (uint32_t)a.s);
  }
}

// Exclusive scan of the block sums in place, totals to tot (one block).
__global__ void __launch_bounds__(1024) k_lay_scan(int nblk, LaySum *bsum, LayTotals *tot) {
  __shared__ LaySum w[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto add = [](LaySum &x, const LaySum &y) {
    x.s += y.s;
    x.l += y.l;
    x.f += y.f;
    x.c += y.c;
  };
  auto up = [&](LaySum x) {  // inclusive scan over the warp
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      LaySum y;
      y.s = __shfl_up_sync(0xffffffffu, x.s, d);
      y.l = __shfl_up_sync(0xffffffffu, x.l, d);
      y.f = __shfl_up_sync(0xffffffffu, x.f, d);
      y.c = __shfl_up_sync(0xffffffffu, x.c, d);
      if (lane >= d) add(x, y);
    }
    return x;
  };
  LaySum carry{0ull, 0ull, 0u, 0u};
  for (int b0 = 0; b0 < nblk; b0 += 1024) {
    const int b = b0 + (int)threadIdx.x;
    LaySum v{0ull, 0ull, 0u, 0u};
    if (b < nblk) v = bsum[b];
    const LaySum x = up(v);
    if (lane == 31) w[wid] = x;
    __syncthreads();
    if (wid == 0) w[lane] = up(w[lane]);
    __syncthreads();
    LaySum off = carry;
    if (wid) add(off, w[wid - 1]);
    if (b < nblk) {
      LaySum o = off;
      o.s += x.s - v.s;
      o.l += x.l - v.l;
      o.f += x.f - v.f;
      o.c += x.c - v.c;
      bsum[b] = o;
    }
    add(carry, w[31]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    tot->s = carry.s;
    tot->l = carry.l;
    tot->f = carry.f;
    tot->c = carry.c;
  }
}

// What the layout writes.  Short-row pointers carry the hub flag of each row in
// bit 31 and are padded with the end offset, so that aligned reads may go a few
// rows past N.  Hub rows get their node, their entries' place, their chunks and
// the places of their st and hm pieces (see SpMat): the static matrix's own hub
// region, or for the hint matrix the row's st part (short or hub region of st)
// and its hm hub part.
struct LayOut {
  uint32_t *rp;
  int64_t *srp;  // static matrix: the row pointers of all static rows
  int32_t *longidx, *lrow, *lchunk, *chunk_lr;
  uint64_t *lptr, *lsb, *lhb;
  uint32_t *lsl, *lhl;
  const uint32_t *st_rp;
  const int32_t *st_longidx;
  const uint64_t *st_lptr;
  int32_t *col;  // hint matrix: its entries, whose spare places are zeroed
  void *w;
  int wbytes;
};
// Rows alone (rp, srp, longidx): what is needed before the hub arrays' sizes
// are known.  HUBS: the hub arrays too.
template <bool HINT, bool ROWS, bool HUBS>
__global__ void __launch_bounds__(256) k_lay_apply(LayIn A, LayOut O, const LaySum *boff,
                                                   const LayTotals *tot) {
  __shared__ LaySum w[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const long long v0 = (long long)blockIdx.x * kLayRows + wid * 32 * kLayPer;
  uint32_t sv[kLayPer], hubs;
  unsigned long long mr = 0, me = 0;
  const LaySum t = warp_rows<HINT>(A, v0, sv, &hubs, &mr, &me);
  if (lane == 0) w[wid] = t;
  __syncthreads();
  LaySum o = boff[blockIdx.x];
  for (int k = 0; k < wid; ++k) {
    o.s += w[k].s;
    o.l += w[k].l;
    o.f += w[k].f;
    o.c += w[k].c;
  }
  const long long N = A.G.N;
  const unsigned long long ns = tot->s;
#pragma unroll
  for (int k = 0; k < kLayPer; ++k) {
    const long long v = v0 + 32 * k + lane;
    const bool hub = hubs >> k & 1u;
    uint32_t x = sv[k];  // inclusive scan of the short lengths (at most 128 each)
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    const unsigned long long so = o.s + x - sv[k];
    const unsigned hm = __ballot_sync(0xffffffffu, hub);
    uint64_t lo = o.l;
    uint32_t li = o.f, co = o.c;
    if (hm) {  // warp-uniform
      const RowLen r = hub ? row_len<HINT>(A, v) : RowLen{0u, 0ull, 0ull, false};
      const uint32_t nc = hub ? row_chunks(r.cl) : 0u;
      unsigned long long xl = r.l;
      uint32_t xc = nc;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long yl = __shfl_up_sync(0xffffffffu, xl, d);
        const uint32_t yc = __shfl_up_sync(0xffffffffu, xc, d);
        if (lane >= d) {
          xl += yl;
          xc += yc;
        }
      }
      lo += xl - r.l;
      li += __popc(hm & lt);
      co += xc - nc;
      if (HUBS && hub) {
        const uint64_t at = ns + lo;
        O.lrow[li] = (int32_t)v;
        O.lptr[li] = at;
        O.lchunk[li] = (int32_t)co;
        for (uint32_t c = 0; c < nc; ++c) O.chunk_lr[co + c] = (int32_t)li;
        if (!HINT) {
          O.lsb[li] = at;
          O.lsl[li] = (uint32_t)r.l;
          O.lhb[li] = 0;
          O.lhl[li] = 0;
        } else {
          const int sli = v < A.G.Nst ? O.st_longidx[v] : -1;
          O.lsb[li] = sli >= 0 ? O.st_lptr[sli] : (uint64_t)(O.st_rp[v] & kOffMask);
          O.lsl[li] = (uint32_t)(r.cl - r.l);
          O.lhb[li] = at;
          O.lhl[li] = (uint32_t)r.l;
        }
      }
      o.l += __shfl_sync(0xffffffffu, xl, 31);
      o.f += __popc(hm);
      o.c += __shfl_sync(0xffffffffu, xc, 31);
    }
    if (ROWS && v < N) {
      O.rp[v] = (uint32_t)so | (hub ? kHubFlag : 0u);
      O.longidx[v] = hub ? (int32_t)li : -1;
    }
    if (ROWS && !HINT && v <= A.G.Nst) O.srp[v] = (int64_t)(so + lo);
    o.s += __shfl_sync(0xffffffffu, x, 31);
  }
  if (blockIdx.x != gridDim.x - 1) return;
  if (HINT && threadIdx.x < kPad) {
    const unsigned long long e = ns + tot->l + threadIdx.x;
    O.col[e] = 0;
    if (O.wbytes == 2) reinterpret_cast<uint16_t *>(O.w)[e] = 0;
    else reinterpret_cast<uint32_t *>(O.w)[e] = 0u;
  }
  if (threadIdx.x > kRpPad) return;
  if (ROWS) {
    O.rp[N + threadIdx.x] = (uint32_t)ns;
  }
  if (HUBS && threadIdx.x == 0) {
    O.lptr[tot->f] = ns + tot->l;
    O.lchunk[tot->f] = (int32_t)tot->c;
  }
}

__global__ void k_u64_to_u32(const uint64_t *a, uint32_t *b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    b[i] = (uint32_t)a[i];
}

// ------------------------------------------------------- H9: row assembly
__device__ __forceinline__ void acc_deg(dfl &D, dfl &Pp, float w) {
  df_add(D, w);
  if (w > 0.f) df_add(Pp, w);
}

// |u - c| as a normalized double-float, for u = uh + ul (ul the rounding
// residue of uh) and an exactly representable c: TwoSum of uh and -c, then
// the low parts.
__device__ __forceinline__ dfl df_absdiff(float uh, float ul, float c) {
  dfl s{uh, 0.f};
  df_add(s, -c);
  s.lo = __fadd_rn(s.lo, ul);
  s = df_norm(s);
  if (s.hi < 0.f) s = dfl{-s.hi, -s.lo};
  return s;
}
__device__ __forceinline__ bool df_ge(dfl a, dfl b) {
  return a.hi > b.hi || (a.hi == b.hi && a.lo >= b.lo);
}
// e^{-r} for r = hi + lo >= 0: FP32 exp of r.hi times the first-order correction for
// r.lo.
__device__ __forceinline__ float exp_neg_df(dfl r) { return expf(-r.hi) * (1.0f - r.lo); }

// (x - o) * s for a float x, o = oh + ol and s = sh + sl (double-floats), to
// about 44 bits with FP32 operations only.
__device__ __forceinline__ dfl df_offset_scale(float x, float oh, float ol, float sh, float sl) {
  dfl d{x, 0.f};
  df_add(d, -oh);
  d.lo = __fadd_rn(d.lo, -ol);
  d = df_norm(d);
  const float ph = __fmul_rn(d.hi, sh);
  float pl = __fmaf_rn(d.hi, sh, -ph);
  pl = __fmaf_rn(d.hi, sl, pl);
  pl = __fmaf_rn(d.lo, sh, pl);
  return df_norm(dfl{ph, pl});
}
// |x - c| / h for floats x, c and h > 0 as a double-float: the difference
// is exact (TwoSum), the quotient carries its FMA remainder.
__device__ __forceinline__ dfl df_ratio(float x, float c, float h) {
  if (!(h > 0.f)) return dfl{__int_as_float(0x7f800000), 0.f};
  dfl d{x, 0.f};
  df_add(d, -c);
  d = df_norm(d);
  if (d.hi < 0.f) d = dfl{-d.hi, -d.lo};
  const float q = __fdiv_rn(d.hi, h);
  const float r = __fmaf_rn(-q, h, d.hi);
  return df_norm(dfl{q, __fdiv_rn(__fadd_rn(r, d.lo), h)});
}

// a b as a double-float.
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_norm(dfl{p, e});
}
// 2^{-j/32}, j = 0..31, as double-floats.
struct ExpTable {
  float2 t[32];
};
// e^{-r} for 0 <= r < 60 to about 2^-42, in FP32 operations (table-driven
// exponential after P. T. P. Tang, ACM TOMS 15, 1989): e^{-r} = 2^{-k/32} e^f with
// k = rint(32 r / ln 2) and |f| <= ln 2 / 64 + a few ulps; ln 2 / 32 in three
// parts, the first two of 12 bits, so that their products with k are exact; e^f
// by its Taylor series, the terms from f^3 on in one FP32 Horner form.
__device__ __forceinline__ dfl exp_neg_dd(dfl r, const float2 *tab) {
  const float kf = rintf(__fmul_rn(r.hi, 46.166241308446829f));  // 32 / ln 2
  const int k = (int)kf;
  constexpr float kL1 = 0x1.62ep-6f, kL2 = 0x1.0bep-20f, kL3 = 0x1.be8e7ap-32f;
  dfl f{__fmul_rn(kf, kL1), 0.f};
  df_add(f, -r.hi);
  df_add(f, __fmul_rn(kf, kL2));
  f.lo = __fadd_rn(f.lo, __fmaf_rn(kf, kL3, -r.lo));
  f = df_norm(f);
  const float q = __fmul_rn(f.hi, f.hi);
  const float qe = __fmaf_rn(f.hi, f.hi, -q);
  float c = __fmaf_rn(f.hi, 1.f / 120.f, 1.f / 24.f);
  c = __fmaf_rn(f.hi, c, 1.f / 6.f);
  c = __fmul_rn(__fmul_rn(q, f.hi), c);  // f^3 / 6 + f^4 / 24 + f^5 / 120
  dfl e = f;                              // e^f - 1
  df_add(e, __fmul_rn(0.5f, q));
  e.lo = __fadd_rn(e.lo, __fadd_rn(__fmaf_rn(f.hi, f.lo, __fmul_rn(0.5f, qe)), c));
  e = df_norm(e);
  const float2 tj = tab[k & 31];
  dfl t = df_mul(dfl{tj.x, tj.y}, e);
  dfl s{tj.x, 0.f};
  df_add(s, t.hi);
  s.lo = __fadd_rn(s.lo, __fadd_rn(tj.y, t.lo));
  const float sc = __uint_as_float((uint32_t)(127 - (k >> 5)) << 23);  // exact scaling
  s = df_norm(s);
  return dfl{__fmul_rn(s.hi, sc), __fmul_rn(s.lo, sc)};
}
// Whether the normalized double-float v, of relative error at most tol, may
// round to another FP32 value than the one it stands for: v lies within its
// error of a rounding midpoint, or is too small or an exact power of two (whose
// midpoints are not half an ulp away on both sides).
__device__ __forceinline__ bool near_fp32_tie(dfl v, float tol) {
  const uint32_t b = __float_as_uint(v.hi) & 0x7fffffffu;
  if ((b & 0x7fffffu) == 0u || b < (40u << 23) || b >= (250u << 23)) return true;
  const float half = __uint_as_float((b & 0x7f800000u) - (24u << 23));
  return !(fabsf(fabsf(v.lo) - half) > tol * fabsf(v.hi));
}
constexpr float kExpMax = 60.f;        // largest exponent of exp_neg_dd
constexpr float kMacroTol = 0x1p-39f;  // a macro weight's error bound at ratio 0 ...
constexpr float kMacroTolR = 0x1p-42f;  // ... and per unit of its ratio
// -e^{-r} w and -(e phi) w for FP32 storage, rounded once, from double-floats;
// *tie: the rounding is not decided and the FP64 value is needed.
__device__ __forceinline__ float df_weight(dfl e, dfl w, float tol, bool *tie) {
  const dfl v = df_mul(e, w);
  *tie = near_fp32_tie(v, tol);
  return -v.hi;
}

// Hint part of the rows of cells, macro pins and stars (thread per row): for a
// hint cell its macro entries (ascending macro), written to the row's hm
// place, and the weights of its detection-window bins as a dense block of W
// slots, slot s = (yy - by + hy) (2 hx + 1) + (xx - bx + hx) for window bin
// (xx, yy) around the cell's bin (bx, by); slots outside the bin grid hold 0.
// The column of a slot is implicit (the bin node of that window position), and
// the bin rows are the transpose of these blocks (k_bin_partials).  The degree
// sums of the whole augmented row are the static ones plus the hint entries.
// The window ratios |x - x_b| / (w_b / 2) = |u - (2 xx + 1)|, u = 2 (x - x_l) /
// w_b, come from u (double-float, once per cell) as exact double-float
// differences; macro ratios are double-float quotients.  FP64 only recomputes
// weights near a rounding midpoint of the storage type.  For FP32 storage the
// weight itself is a double-float (exponential to 2^-42, products to 2^-45): its
// FP64 form, at 1/64 of the FP32 rate, took 352 us of a 210k-cell design's refinement
// round of 970 us (order 8); with the double-float form the round takes 641 us.
// Own entries and window blocks of a warp's 32 rows are staged in shared memory
// and written as one run each: a block is W weights at a stride of W per lane,
// which as plain stores are W partial writes of several lines.  2.2M cells, BF16,
// 3 x 3 windows: 173 -> 169 us, and 146 us with the four blocks per SM that the
// smaller stage leaves room for (FP32 storage: 25 us with three, 28 with four).
constexpr int kAsmStage = 256;   // entries
constexpr int kAsmBlock = 2304;  // bytes of window blocks (wider windows are written directly)
template <bool bf>
__global__ void __launch_bounds__(256, bf ? 4 : 3) k_assemble_hints(
    HintGeo G, ExpTable xt, const uint32_t *hrp, const int32_t *longidx, const uint64_t *lptr,
    const dfl *sdsum, const dfl *spsum, const uint8_t *hflag, const int32_t *cell_bin,
    const int32_t *n_ovl, const float2 *xy, const float *cw, const float *ch,
    const int64_t *gptr, const uint32_t *glist, const float4 *ggeo, const double *base_w,
    const float *phif, const float *phil, const double *phid, int W, const int32_t *cmem, const float4 *mgeo,
    int32_t *col, void *w, void *bwin, int32_t *hbin, dfl *dsum, dfl *psum, uint64_t *mac_base,
    unsigned long long *counts) {
  __shared__ int32_t stage_col[8][kAsmStage];
  __shared__ uint32_t stage_w[8][kAsmStage];
  __shared__ float2 exp_tab[bf ? 1 : 32];
  if (!bf) {
    if (threadIdx.x < 32) exp_tab[threadIdx.x] = xt.t[threadIdx.x];
    __syncthreads();
  }
  const int lane = threadIdx.x & 31;
  int32_t *scol = stage_col[threadIdx.x >> 5];
  uint32_t *sw = stage_w[threadIdx.x >> 5];
  __shared__ __align__(16) uint8_t stage_blk[8][kAsmBlock];
  uint8_t *sblk = stage_blk[threadIdx.x >> 5];
  constexpr int wbytes = bf ? 2 : 4;
  const bool sb = 32 * W * wbytes <= kAsmBlock;
  const long long stride = (long long)gridDim.x * blockDim.x;
  unsigned long long slots = 0, hints = 0;  // this thread's window slots in the grid, hint cells
  for (long long v0 = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); v0 < G.Nst;
       v0 += stride) {
    const long long v = v0 + lane;
    // the warp's rows own a contiguous short-region range [rb, re)
    const uint64_t rb = hrp[v0] & kOffMask;
    const uint64_t re = hrp[v0 + 32 < G.Nst ? v0 + 32 : G.Nst] & kOffMask;
    const bool staged = re - rb <= (uint64_t)kAsmStage;  // warp-uniform
    if (v >= G.Nst) goto flush;
    {
    dfl Dl = sdsum[v], Pl = spsum[v];
    // a cell's inputs, loaded before its hint test so that they are in flight
    // together rather than one dependent round after another
    uint8_t hf = 0;
    int li = -1, cb = 0, nov = 0;
    uint32_t hr = 0;
    float2 p = make_float2(0.f, 0.f);
    double bw = 0.0;
    if (v < G.C) {
      hf = hflag[v];
      li = longidx[v];
      hr = hrp[v];
      p = xy[v];
      bw = base_w[v];
      cb = cell_bin[v];
      nov = n_ovl[v];
    }
    if (v < G.C) hbin[v] = hf ? cb : -1;
    if (hf) {
      ++hints;
      const uint64_t mb = li >= 0 ? lptr[li] : (uint64_t)(hr & kOffMask);
      const bool use_s = staged && li < 0;
      // an own entry: to the warp's stage (short rows) or straight to memory
      auto put = [&](uint64_t kk, int32_t c, uint32_t bits) {
        if (use_s) {
          scol[kk - rb] = c;
          sw[kk - rb] = bits;
        } else {
          col[kk] = c;
          if (bf) reinterpret_cast<uint16_t *>(w)[kk] = (uint16_t)bits;
          else reinterpret_cast<uint32_t *>(w)[kk] = bits;
        }
      };
      if (!isfinite(p.x) || !isfinite(p.y)) p = make_float2(0.f, 0.f);
      const float bwf = __double2float_rn(bw);
      const dfl bwd{bwf, bf ? 0.f : __double2float_rn(bw - (double)bwf)};
      // macro entries, ascending macro id (grid bucket lists are sorted)
      uint64_t k = mb;
      auto mac_entry = [&](int m, float4 mg) {
        uint32_t bits;
        float sv;
        if (bf) {
          const dfl rx = df_ratio(p.x, mg.x, __fmul_rn(0.5f, mg.z));
          const dfl ry = df_ratio(p.y, mg.y, __fmul_rn(0.5f, mg.w));
          const float wv = -(exp_neg_df(df_ge(rx, ry) ? rx : ry) * bwf);
          const uint16_t h = near_bf16_tie(wv)
                                 ? d2bf16(macro_w_exact(p.x, p.y, mg.x, mg.y, mg.z, mg.w, bw))
                                 : f2bf16(wv);
          bits = h;
          sv = bf16_to_f(h);
        } else {
          const dfl rx = df_ratio(p.x, mg.x, __fmul_rn(0.5f, mg.z));
          const dfl ry = df_ratio(p.y, mg.y, __fmul_rn(0.5f, mg.w));
          const dfl r = df_ge(rx, ry) ? rx : ry;
          bool tie = !(r.hi < kExpMax);
          sv = 0.f;
          if (!tie) sv = df_weight(exp_neg_dd(r, exp_tab), bwd, kMacroTol + kMacroTolR * r.hi, &tie);
          if (tie) sv = __double2float_rn(macro_w_exact(p.x, p.y, mg.x, mg.y, mg.z, mg.w, bw));
          bits = __float_as_uint(sv);
        }
        put(k, (int32_t)(G.mv0 + m), bits);
        acc_deg(Dl, Pl, sv);
        ++k;
      };
      if (cmem) {
        // the cell's macros as the cell pass found them (same geometry values)
        for (int j = 0; j < nov; ++j) {
          const int m = cmem[(long long)v * kMacroSlots + j];
          mac_entry(m, mgeo[m]);
        }
      } else {
        const int kx = grid_of(p.x, G.gxf, G.gsxf, G.gnx), ky = grid_of(p.y, G.gyf, G.gsyf, G.gny);
        const long long gk = (long long)ky * G.gnx + kx;
        const float cwv = cw[v], chv = ch[v];
        const long long qa = gptr[gk], qb = gptr[gk + 1];
        for (long long q0 = qa; q0 < qb; q0 += 4) {
          float4 mgs[4];  // four grid entries' geometry loaded at once
#pragma unroll
          for (int u = 0; u < 4; ++u) mgs[u] = q0 + u < qb ? ggeo[q0 + u] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const long long q = q0 + u;
            const float4 mg = mgs[u];
            if (q >= qb || !overlaps(p.x, p.y, cwv, chv, mg.x, mg.y, mg.z, mg.w)) continue;
            mac_entry((int)glist[q], mg);
          }
        }
      }
      // window slots, row-major over the full window
      const int b = cb, bx = b % G.nbx, by = b / G.nbx;
      const dfl ux = df_offset_scale(p.x, G.xlh, G.xll, G.iwh, G.iwl);
      const dfl uy = df_offset_scale(p.y, G.ylh, G.yll, G.ihh, G.ihl);
      uint16_t *wb16 = sb ? reinterpret_cast<uint16_t *>(sblk) + lane * W
                          : reinterpret_cast<uint16_t *>(bwin) + (size_t)v * W;
      uint32_t *wb32 = sb ? reinterpret_cast<uint32_t *>(sblk) + lane * W
                          : reinterpret_cast<uint32_t *>(bwin) + (size_t)v * W;
      int sidx = 0;
      if (bf && G.hx == 1) {
        // three window columns: their ratios and e^{-rx} once per cell, not
        // once per window row (the same values, so the same weights)
        dfl rxs[3];
        float exs[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int xx = bx - 1 + c;
          rxs[c] = df_absdiff(ux.hi, ux.lo, (float)(2 * xx + 1));
          exs[c] = (xx >= 0 && xx < G.nbx) ? exp_neg_df(rxs[c]) : 0.f;
        }
        for (int yy = by - G.hy; yy <= by + G.hy; ++yy) {
          const bool yin = yy >= 0 && yy < G.nby;
          const dfl ry = df_absdiff(uy.hi, uy.lo, (float)(2 * yy + 1));
          const float ey = yin ? exp_neg_df(ry) : 0.f;
          float ph[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const int xx = bx - 1 + c;
            ph[c] = (yin && xx >= 0 && xx < G.nbx) ? phif[yy * G.nbx + xx] : 0.f;
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const int xx = bx - 1 + c;
            uint16_t h = 0;
            if (yin && xx >= 0 && xx < G.nbx) {
              const float e = df_ge(rxs[c], ry) ? exs[c] : ey;
              const float wv = -((e * ph[c]) * bwf);
              h = near_bf16_tie(wv)
                      ? d2bf16(bin_w_exact(p.x, p.y, xx, yy, G, phid[yy * G.nbx + xx], bw))
                      : f2bf16(wv);
              acc_deg(Dl, Pl, bf16_to_f(h));
              ++slots;
            }
            wb16[sidx++] = h;
          }
        }
      } else if (bf) {
        for (int yy = by - G.hy; yy <= by + G.hy; ++yy) {
          const bool yin = yy >= 0 && yy < G.nby;
          // e^{-max(rx, ry)} is e^{-rx} or e^{-ry}
          const dfl ry = df_absdiff(uy.hi, uy.lo, (float)(2 * yy + 1));
          const float ey = yin ? exp_neg_df(ry) : 0.f;
          for (int xc = bx - G.hx; xc <= bx + G.hx; xc += 4) {
            float ph[4];  // four window bins' phi loaded at once
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int xx = xc + u;
              ph[u] = (yin && xx >= 0 && xx < G.nbx && xx <= bx + G.hx) ? phif[yy * G.nbx + xx] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int xx = xc + u;
              if (xx > bx + G.hx) break;
              uint16_t h = 0;
              if (yin && xx >= 0 && xx < G.nbx) {
                const dfl rx = df_absdiff(ux.hi, ux.lo, (float)(2 * xx + 1));
                const float e = df_ge(rx, ry) ? exp_neg_df(rx) : ey;
                const float wv = -((e * ph[u]) * bwf);
                h = near_bf16_tie(wv)
                        ? d2bf16(bin_w_exact(p.x, p.y, xx, yy, G, phid[yy * G.nbx + xx], bw))
                        : f2bf16(wv);
                acc_deg(Dl, Pl, bf16_to_f(h));
                ++slots;
              }
              wb16[sidx++] = h;
            }
          }
        }
      } else {
        // FP32 storage: double-float weights; the ratios and exponentials of
        // three window columns once per cell (wider windows: per slot)
        const bool three = G.hx == 1;
        dfl rxs[3], exs[3];
        auto column = [&](int xx, dfl *r, dfl *e) {
          *r = df_absdiff(ux.hi, ux.lo, (float)(2 * xx + 1));
          *e = r->hi < kExpMax ? exp_neg_dd(*r, exp_tab) : dfl{0.f, 0.f};
        };
        if (three) {
#pragma unroll
          for (int c = 0; c < 3; ++c) column(bx - 1 + c, &rxs[c], &exs[c]);
        }
        auto slot = [&](int xx, int yy, bool yin, dfl rx, dfl ex, dfl ry, dfl ey) {
          float sv = 0.f;
          if (yin && xx >= 0 && xx < G.nbx) {
            const int bb = yy * G.nbx + xx;
            const bool ge = df_ge(rx, ry);
            const dfl e = df_mul(ge ? ex : ey, dfl{phif[bb], phil[bb]});
            bool tie;
            sv = df_weight(e, bwd, G.tol, &tie);
            if (tie || !((ge ? rx.hi : ry.hi) < kExpMax))
              sv = __double2float_rn(bin_w_exact(p.x, p.y, xx, yy, G, phid[bb], bw));
            acc_deg(Dl, Pl, sv);
            ++slots;
          }
          wb32[sidx++] = __float_as_uint(sv);
        };
        for (int yy = by - G.hy; yy <= by + G.hy; ++yy) {
          const bool yin = yy >= 0 && yy < G.nby;
          const dfl ry = df_absdiff(uy.hi, uy.lo, (float)(2 * yy + 1));
          const dfl ey = ry.hi < kExpMax ? exp_neg_dd(ry, exp_tab) : dfl{0.f, 0.f};
          if (three) {
#pragma unroll
            for (int c = 0; c < 3; ++c) slot(bx - 1 + c, yy, yin, rxs[c], exs[c], ry, ey);
          } else {
            for (int xx = bx - G.hx; xx <= bx + G.hx; ++xx) {
              dfl rx, ex;
              column(xx, &rx, &ex);
              slot(xx, yy, yin, rx, ex, ry, ey);
            }
          }
        }
      }
      mac_base[v] = mb;
    }
    dsum[v] = df_norm(Dl);
    psum[v] = df_norm(Pl);
    }
  flush:
    // the staged blocks and entries, written with coalesced stores (the block of a
    // cell without hints is never read; whatever the stage held goes there)
    if (sb && v0 < G.C) {
      __syncwarp();
      const int nb = (int)(min((long long)32, G.C - v0) * W * wbytes);
      uint8_t *dst = reinterpret_cast<uint8_t *>(bwin) + (size_t)v0 * W * wbytes;
      for (int i = lane * 4; i + 4 <= nb; i += 128)
        *reinterpret_cast<uint32_t *>(dst + i) = *reinterpret_cast<const uint32_t *>(sblk + i);
      if ((nb & 2) && lane == 0)
        *reinterpret_cast<uint16_t *>(dst + nb - 2) = *reinterpret_cast<const uint16_t *>(sblk + nb - 2);
      __syncwarp();
    }
    if (staged) {
      __syncwarp();
      for (uint64_t i = lane; i < re - rb; i += 32) {
        col[rb + i] = scol[i];
        if (bf) reinterpret_cast<uint16_t *>(w)[rb + i] = (uint16_t)sw[i];
        else reinterpret_cast<uint32_t *>(w)[rb + i] = sw[i];
      }
      __syncwarp();
    }
  }
  slots = warp_sum(slots);
  hints = warp_sum(hints);
  if (lane == 0 && slots) atomicAdd(counts, slots);
  if (lane == 0 && hints) atomicAdd(counts + 1, hints);
}

// The window blocks of the bin rows' chunks, slot-major within a chunk: the
// weight of slot t of the i-th hint cell of chunk c (the cell at list
// position boff[2b] + (c - bchunk[b]) kBinChunk + i of its bin b) goes to
// out[(c W + t) kBinChunk + i], so the bin rows read each slot of a chunk as
// consecutive weights.  A thread per (chunk, cell) gathers the cell's block
// and writes its W weights; places past a bucket's last hint cell are not
// written (and never read).
template <typename T>
__global__ void k_blocks_to_chunks(long long nthreads, int W, const int32_t *bchunk, int NB,
                                   const int32_t *cown, const int64_t *boff,
                                   const uint32_t *blist, const T *blk, T *out) {
  const int nchunk = bchunk[NB];
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nthreads;
       q += (long long)gridDim.x * blockDim.x) {
    const long long c = q / kBinChunk;
    if (c >= nchunk) break;
    const int i = (int)(q - c * kBinChunk), b = cown[c];
    const long long k = boff[2 * b] + (long long)(c - bchunk[b]) * kBinChunk + i;
    T *dst = out + (size_t)c * W * kBinChunk + i;
    if (k < boff[2 * b + 1]) {
      const T *src = blk + (size_t)blist[k] * W;
      for (int t = 0; t < W; ++t) dst[(size_t)t * kBinChunk] = src[t];
    }
  }
}

// Macro rows, in the hub chunks of the sparse-product layout (one CTA per
// chunk of kChunk entries): a macro row lists the cells overlapping it
// (sorted by id), with the weights copied from the cells' own entries, so the
// matrix is exactly symmetric.  Degree partials per chunk.
__global__ void __launch_bounds__(256) k_hub_chunks(
    HintGeo G, int wdtype, const uint32_t *pnchunks, const int32_t *chunk_lr, const int32_t *lrow,
    const uint64_t *lptr, const int32_t *lchunk, const int64_t *moff, const uint32_t *mlist,
    const int32_t *n_ovl, const uint64_t *mac_base, int32_t *col, void *w, dfl *cpart) {
  __shared__ dfl red[2][8];
  const int nchunks = (int)*pnchunks;
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int l = chunk_lr[c];
    const int64_t v = lrow[l];
    if (v < G.mv0 || v >= G.bn0) continue;  // macro rows only
    const uint64_t base = lptr[l];
    const long long len = (long long)(lptr[l + 1] - base);
    const long long q0 = (long long)(c - lchunk[l]) * kChunk;
    const long long q1 = min(len, q0 + (long long)kChunk);
    const int m = (int)(v - G.mv0);
    dfl D{0.f, 0.f}, Pp{0.f, 0.f};
    for (long long q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
      const int i = (int)mlist[moff[m] + q];
      const uint64_t mb = mac_base[i];
      const int n = n_ovl[i];
      int j = 0;
      while (j < n - 1 && col[mb + j] != (int32_t)v) ++j;
      const uint64_t src = mb + j;
      col[base + q] = i;
      copy_w(w, w, wdtype, base + q, src);
      acc_deg(D, Pp, load_w(w, wdtype, src));
    }
    D = warp_sum_df(D);
    Pp = warp_sum_df(Pp);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
      red[0][wid] = D;
      red[1][wid] = Pp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      dfl a = red[0][0], e = red[1][0];
      for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
        df_add_df(a, red[0][k]);
        df_add_df(e, red[1][k]);
      }
      cpart[2 * (long long)c] = df_norm(a);
      cpart[2 * (long long)c + 1] = df_norm(e);
    }
    __syncthreads();
  }
}

// Degrees of virtual rows (warp per row): a macro row from its chunk
// partials, a bin row from the window blocks' degree partials per chunk.
__global__ void k_hub_finalize(HintGeo G, BinGeo B, const uint32_t *pnlong, const int32_t *lrow,
                               const int32_t *lchunk, const dfl *cpart, const int32_t *bchunk,
                               const float4 *bdeg,
                               dfl *dsum, dfl *psum) {
  const int lane = threadIdx.x & 31;
  const long long nlong = *pnlong;
  for (long long l = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; l < nlong;
       l += ((long long)gridDim.x * blockDim.x) >> 5) {
    const int64_t v = lrow[l];
    if (v < G.mv0) continue;
    dfl D{0.f, 0.f}, Pp{0.f, 0.f};
    if (v >= G.bn0) {
      bin_row_chunks(B, (int)(v - G.bn0), bchunk, bdeg, &D, &Pp);
    } else {
      for (int c = lchunk[l] + lane; c < lchunk[l + 1]; c += 32) {
        df_add_df(D, cpart[2 * (long long)c]);
        df_add_df(Pp, cpart[2 * (long long)c + 1]);
      }
      D = warp_sum_df(D);
      Pp = warp_sum_df(Pp);
    }
    if (lane == 0) {
      dsum[v] = D;
      psum[v] = Pp;
    }
  }
}

// ------------------------------------------------- H11: lambda_up, c_i
__global__ void k_lambda_max(int64_t N, const dfl *psum, unsigned long long *key) {
  unsigned long long best = 0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
       v += (long long)gridDim.x * blockDim.x) {
    dfl p = psum[v];
    dfl two = df_norm(dfl{__fmul_rn(2.f, p.hi), __fmul_rn(2.f, p.lo)});
    unsigned long long k = df_maxkey(two);
    if (k > best) best = k;
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    unsigned long long o = __shfl_xor_sync(0xffffffffu, best, m);
    best = o > best ? o : best;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(key, best);
}

// lambda_up and 1 / lambda_up from the largest key (also copied to status words
// 4..7, so that the host reads them with the status), then every row's
// coefficient a_v = 1 - D_vv / lambda_up in FP32 and the hub rows' in FP64.
__global__ void k_coef(int64_t N, const dfl *dsum, const unsigned long long *key, double *lam,
                       int *status, float *c32, const uint32_t *pnlong, const int32_t *lrow,
                       double *c64) {
  __shared__ double s_il;
  if (threadIdx.x == 0) {
    const double l = df_from_maxkey(*key);
    const bool ok = l > 0.0 && !isinf(l);
    const double il = ok ? __ddiv_rn(1.0, l) : 0.0;
    s_il = il;
    if (blockIdx.x == 0) {
      if (!ok) flag(status, ST_SPECTRUM);
      lam[0] = l;
      lam[1] = il;
      reinterpret_cast<double *>(status + 4)[0] = l;
      reinterpret_cast<double *>(status + 4)[1] = il;
    }
  }
  __syncthreads();
  const double ild = s_il;
  const float il = __double2float_rn(ild);
  const long long nlong = *pnlong, t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x,
                  nt = (long long)gridDim.x * blockDim.x;
  for (long long l = t0; l < nlong; l += nt) c64[l] = 1.0 - df_to_d(dsum[lrow[l]]) * ild;
  for (long long v = t0; v < N; v += nt) {
    dfl d = dsum[v];
    c32[v] = __fadd_rn(1.f, -__fmaf_rn(d.hi, il, __fmul_rn(d.lo, il)));
  }
}

// --------------------------------------------------------------- driver
template <typename T>
static cudaError_t d2h(T *h, const void *d, size_t n, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(h, d, n * sizeof(T), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(s);
}

static HintGeo make_geo(const pl_graph *g) {
  HintGeo G;
  G.xlf = (float)g->xl;
  G.ylf = (float)g->yl;
  G.sxf = (float)((double)g->nbx / (g->xh - g->xl));
  G.syf = (float)((double)g->nby / (g->yh - g->yl));
  G.gxf = (float)g->xl;
  G.gyf = (float)g->yl;
  G.gsxf = (float)g->gsx;
  G.gsyf = (float)g->gsy;
  G.xl = g->xl;
  G.yl = g->yl;
  G.wb = g->wb;
  G.hb = g->hb;
  G.iwb2 = 2.0 / g->wb;
  G.ihb2 = 2.0 / g->hb;
  auto split = [](double d, float *h, float *l) {
    *h = (float)d;
    *l = (float)(d - (double)*h);
  };
  split(G.xl, &G.xlh, &G.xll);
  split(G.yl, &G.ylh, &G.yll);
  split(G.iwb2, &G.iwh, &G.iwl);
  split(G.ihb2, &G.ihh, &G.ihl);
  // Error bound of a double-float bin weight against the FP64 one, relative:
  // the exponential and the products (2^-41), the ratio 2 (x - x_l) / w_b (its
  // double-float form carries about 2^-45 of the bin count and 2^-47 of the
  // region's coordinates over the bin size; the FP64 form far less).
  G.tol = (float)(std::ldexp(1.0, -39) + std::ldexp((double)g->nbx + g->nby, -43) +
                  std::ldexp(std::fmax(std::fabs(g->xl), std::fabs(g->xh)) / g->wb +
                                 std::fmax(std::fabs(g->yl), std::fabs(g->yh)) / g->hb, -44));
  G.nbx = g->nbx;
  G.nby = g->nby;
  G.hx = g->hx;
  G.hy = g->hy;
  G.gnx = g->gnx;
  G.gny = g->gny;
  G.C = g->C;
  G.Pm = g->Pm;
  G.S = g->S;
  G.Mm = g->Mm;
  G.Nst = g->Nst;
  G.mv0 = g->Nst;
  G.bn0 = g->Nst + g->Mm;
  G.N = g->N;
  return G;
}

static const ExpTable &exp_table() {
  static const ExpTable t = [] {
    ExpTable e;
    for (int j = 0; j < 32; ++j) {
      const double v = std::exp2(-(double)j / 32.0);
      e.t[j].x = (float)v;
      e.t[j].y = (float)(v - (double)e.t[j].x);
    }
    return e;
  }();
  return t;
}

static BinGeo make_bingeo(const pl_graph *g) {
  BinGeo B;
  B.nbx = g->nbx;
  B.nby = g->nby;
  B.hx = g->hx;
  B.hy = g->hy;
  B.W = (2 * g->hx + 1) * (2 * g->hy + 1);
  B.NB = g->NB;
  return B;
}

// First part of a layout: the block sums, offsets and totals (device), in
// g->lay[0] and g->lay[1].
static pl_status lay_sums(pl_graph *g, const LayIn &A, cudaStream_t s, LaySum **bsum,
                          LayTotals **tot, int *nblk) {
  *nblk = (int)((g->N + kLayRows - 1) / kLayRows);
  TRY(ensure(g->lay[0], (size_t)*nblk * sizeof(LaySum) + 256));
  TRY(ensure(g->lay[1], sizeof(LayTotals) + 256));
  *bsum = P<LaySum>(g->lay[0]);
  *tot = P<LayTotals>(g->lay[1]);
  if (A.cnt) {
    TRY(cudaMemsetAsync(*tot, 0, sizeof(LayTotals), s));
    k_lay_sum<false><<<*nblk, 256, 0, s>>>(A, *bsum, *tot);
  } else {
    k_lay_sum<true><<<*nblk, 256, 0, s>>>(A, *bsum, *tot);
  }
  note_launch();
  k_lay_scan<<<1, 1024, 0, s>>>(*nblk, *bsum, *tot);
  note_launch();
  return PL_OK;
}

static bool lay_too_large(uint64_t ns, uint64_t nl) {
  if (ns + kPad < (uint64_t)kOffMask && ns + nl < (1ull << 40)) return false;
  set_error("graph too large for the 31-bit short-row layout (%llu entries)",
            (unsigned long long)ns);
  return true;
}

// The hub arrays for nl hub rows and nc chunks.
static cudaError_t lay_hub_arrays(SpMat &m, size_t nl, size_t nc) {
  cudaError_t e = ensure(m.lrow, nl * 4 + 16);
  if (e == cudaSuccess) e = ensure(m.lptr, (nl + 1) * 8);
  if (e == cudaSuccess) e = ensure(m.lsb, nl * 8 + 16);
  if (e == cudaSuccess) e = ensure(m.lhb, nl * 8 + 16);
  if (e == cudaSuccess) e = ensure(m.lsl, nl * 4 + 16);
  if (e == cudaSuccess) e = ensure(m.lhl, nl * 4 + 16);
  if (e == cudaSuccess) e = ensure(m.lchunk, (nl + 1) * 4);
  if (e == cudaSuccess) e = ensure(m.chunk_lr, nc * 4 + 16);
  if (e == cudaSuccess) e = ensure(m.c64l, nl * 8 + 16);
  return e;
}
static size_t lay_hub_bytes(size_t nl, size_t nc) {
  return nl * 48 + nc * 4 + 9 * 256 + 256;
}

static LayOut lay_out(pl_graph *g, SpMat &m) {
  LayOut O;
  O.rp = P<uint32_t>(m.rp_s);
  O.srp = P<int64_t>(g->srp);
  O.longidx = P<int32_t>(m.longidx);
  O.lrow = P<int32_t>(m.lrow);
  O.lchunk = P<int32_t>(m.lchunk);
  O.chunk_lr = P<int32_t>(m.chunk_lr);
  O.lptr = P<uint64_t>(m.lptr);
  O.lsb = P<uint64_t>(m.lsb);
  O.lhb = P<uint64_t>(m.lhb);
  O.lsl = P<uint32_t>(m.lsl);
  O.lhl = P<uint32_t>(m.lhl);
  O.st_rp = P<uint32_t>(g->st.rp_s);
  O.st_longidx = P<int32_t>(g->st.longidx);
  O.st_lptr = P<uint64_t>(g->st.lptr);
  O.col = P<int32_t>(m.col);
  O.w = m.w.p;
  O.wbytes = m.wbytes;
  return O;
}

// The entries' arrays (nnz of them and the spare ones) and the arrays over all rows.
static pl_status lay_entries(pl_graph *g, SpMat &m, uint64_t nnz) {
  const int64_t N = g->N;
  const uint64_t cap = nnz + kPad;
  m.N = N;
  m.wbytes = g->wdtype == PL_W_BF16 ? 2 : 4;
  TRY(ensure(m.col, cap * 4));
  TRY(ensure(m.w, cap * m.wbytes));
  TRY(ensure(m.dsum, (size_t)N * 8 + 16));
  TRY(ensure(m.psum, (size_t)N * 8 + 16));
  TRY(ensure(m.c32, (size_t)N * 4 + 16));
  TRY(ensure(m.lam, 64));
  return PL_OK;
}

static void lay_totals(SpMat &m, const LayTotals &t) {
  m.nnz_s = t.s;
  m.nnz_l = t.l;
  m.nlong = (int32_t)t.f;
  m.nchunks = (int32_t)t.c;
}

// Layout of the static split matrix and the static row pointers from the row
// lengths cnt; the entries and degree sums are written by the static
// compaction.  Its totals are read with one synchronisation, after the row
// pointers were launched.
pl_status prepare_static_layout(pl_graph *g, const int32_t *cnt, cudaStream_t s) {
  const int64_t N = g->N;
  LayIn A{};
  A.G.N = N;
  A.G.Nst = g->Nst;
  A.G.C = g->C;
  A.cnt = cnt;
  A.may = kLong - g->W - kMacroSlots;
  LaySum *bsum;
  LayTotals *tot, t;
  int nblk;
  pl_status st = lay_sums(g, A, s, &bsum, &tot, &nblk);
  if (st != PL_OK) return st;
  SpMat &m = g->st;
  TRY(ensure(m.rp_s, (size_t)(N + 1 + kRpPad) * 4));
  TRY(ensure(m.longidx, (size_t)N * 4 + 16));
  TRY(ensure(g->srp, (size_t)(g->Nst + 1) * 8));
  k_lay_apply<false, true, false><<<nblk, 256, 0, s>>>(A, lay_out(g, m), bsum, tot);
  note_launch();
  {
    const D2H it[1] = {{&t, tot, sizeof(LayTotals)}};
    TRY(d2h_many(g->stage, it, 1, s));
  }
  if (lay_too_large(t.s, t.l)) return PL_ERR_UNSUPPORTED;
  lay_totals(m, t);
  g->may_rows = t.may_rows;
  g->may_entries = t.may_entries;
  g->even_rows = 2.0 * (double)t.cell_max * (g->C / kLayRows) <= 3.0 * (double)t.cell_sum;
  TRY(lay_hub_arrays(m, t.f, t.c));
  if (t.f) {
    k_lay_apply<false, false, true><<<nblk, 256, 0, s>>>(A, lay_out(g, m), bsum, tot);
    note_launch();
  } else {
    TRY(cudaMemsetAsync(m.lchunk.p, 0, 4, s));
  }
  TRY(ensure(m.part, (size_t)(t.c + 1) * 16));
  const uint64_t nnz = t.s + t.l;
  st = lay_entries(g, m, nnz);
  if (st != PL_OK) return st;
  TRY(cudaMemsetAsync(P<char>(m.col) + nnz * 4, 0, kPad * 4, s));
  TRY(cudaMemsetAsync(P<char>(m.w) + nnz * m.wbytes, 0, kPad * m.wbytes, s));
  return PL_OK;
}

// Layout of the hint matrix for nml macro-cell overlaps, without a read by the
// host where bounds on the hub rows and chunks fit the workspace: a short
// static row can only become a hub row when it is longer than kLong less the
// window slots and kMacroSlots macro entries (exact_ok: no cell has more), and
// the static layout has counted those.  later: workspace bytes that the rest of
// the build will ask for.  *nl_max, *nc_max: hub rows and chunks at most; the totals stay on the device (*tot) until the build's last read.
static pl_status layout_hints(pl_graph *g, const LayIn &A, int64_t nml, bool exact_ok,
                              size_t later, cudaStream_t s, LayTotals **tot, size_t *nl_max, size_t *nc_max) {
  const int64_t N = g->N;
  LaySum *bsum;
  int nblk;
  pl_status st = lay_sums(g, A, s, &bsum, tot, &nblk);
  if (st != PL_OK) return st;
  SpMat &m = g->hm;
  TRY(ensure(m.rp_s, (size_t)(N + 1 + kRpPad) * 4));
  TRY(ensure(m.longidx, (size_t)N * 4 + 16));
  st = lay_entries(g, m, 2 * (uint64_t)nml);
  if (st != PL_OK) return st;
  size_t nl = (size_t)g->Mm + g->NB + g->st.nlong + g->may_rows;
  size_t nc = nl + (size_t)((g->st.nnz_l + g->may_entries + 2 * (uint64_t)nml) / kChunk) + 1;
  const Arena *ar = current_arena();
  if (!exact_ok || (uint64_t)nml + kPad >= (uint64_t)kOffMask ||
      lay_hub_bytes(nl, nc) + nc * 32 + later > ar->cap - ar->used) {
    LayTotals t;
    const D2H it[1] = {{&t, *tot, sizeof(LayTotals)}};
    TRY(d2h_many(g->stage, it, 1, s));
    if (lay_too_large(t.s, t.l)) return PL_ERR_UNSUPPORTED;
    nl = t.f;
    nc = t.c;
  }
  TRY(lay_hub_arrays(m, nl, nc));
  k_lay_apply<true, true, true><<<nblk, 256, 0, s>>>(A, lay_out(g, m), bsum, *tot);
  note_launch();
  *nl_max = nl;
  *nc_max = nc;
  return PL_OK;
}

// tight: the largest tiles of the counting sorts and exact hub counts, which
// take the least memory.
static pl_status build_hints_in(pl_graph *g, const pl_params *p, const float *xy_in, bool tight,
                                cudaStream_t s) {
  const int64_t N = g->N;
  const int32_t C = g->C, NB = g->NB, Mm = g->Mm;
  const float2 *xy = reinterpret_cast<const float2 *>(xy_in);
  HintGeo G = make_geo(g);
  g->have_hints = false;
  // a hint build takes its buffers anew, above the static build's part of
  // the workspace
  for_each_buf(g, 1, [](Buf &b) { release(b); });
  g->arena.used = g->hint_mark;
  if (g->hx * 2 + 1 > kMaxWin || g->hy * 2 + 1 > kMaxWin) {
    set_error("detection window larger than 31 x 31 bins");
    return PL_ERR_UNSUPPORTED;
  }
  TRY(cudaMemsetAsync(g->status.p, 0, 32, s));
  int *status = P<int>(g->status);
  void *stmp;
  TRY(ensure(g->tmp[7], scan_tmp_bytes(N + 1) + 4096));
  stmp = g->tmp[7].p;

  // H1: bins and macro overlaps of movable cells (bucket counts by atomics
  // only when the buckets do not fit the tiled counting sort)
  const int nbk = 2 * NB;
  const bool tiled = nbk <= kMaxSmemBuckets;
  TRY(ensure(g->cell_bin, (size_t)C * 4 + 16));
  TRY(ensure(g->n_ovl, (size_t)C * 4 + 16));
  TRY(ensure(g->bcnt, (size_t)(nbk + 1) * 4));
  TRY(ensure(g->mcnt, (size_t)(Mm + 1) * 4));
  if (!tiled) TRY(cudaMemsetAsync(g->bcnt.p, 0, (size_t)(nbk + 1) * 4, s));
  int tsh = tight ? 12 : hint_tile_shift(C, NB, Mm);
  {
    // (in a workspace whose rest the counts would take a good part of: the largest
    // tiles, so that the build need not be repeated with them)
    const Arena *ar = current_arena();
    const uint64_t nt = std::max<uint64_t>(1, ((uint64_t)C + (1u << tsh) - 1) >> tsh);
    if ((nt * ((uint64_t)Mm + 2 * (uint64_t)NB)) * 12 > (ar->cap - ar->used) / 16) tsh = 12;
  }
  const int ntile = std::max(1, (int)(((int64_t)C + (1 << tsh) - 1) >> tsh));
  // macro lists by a tiled counting sort when the macros' run counters fit
  // shared memory (else: scatter by atomics, then a segmented sort)
  const bool tiledm = Mm > 0 && Mm <= kMaxSmemMacros;
  const long long nmt = (long long)Mm * ntile;
  if (tiledm) {
    TRY(ensure(g->mtc, (size_t)nmt * 4 + 16));
    TRY(ensure(g->cmem, (size_t)C * kMacroSlots * 4 + 16));
    TRY(cudaMemsetAsync(g->mtc.p, 0, (size_t)nmt * 4, s));
  } else {
    TRY(cudaMemsetAsync(g->mcnt.p, 0, (size_t)(Mm + 1) * 4, s));
  }
  k_hint_cells<<<grid_for(C, 256), 256, 0, s>>>(
      G, xy, P<uint8_t>(g->ckind), P<uint8_t>(g->hflag), P<float>(g->cw), P<float>(g->ch),
      P<int64_t>(g->gptr), P<uint32_t>(g->glist), P<float4>(g->ggeo), P<int32_t>(g->cell_bin),
      P<int32_t>(g->n_ovl), tiled ? nullptr : P<int32_t>(g->bcnt), P<int32_t>(g->mcnt),
      tiledm ? P<int32_t>(g->mtc) : nullptr, ntile, tsh, tiledm ? P<int32_t>(g->cmem) : nullptr,
      status);
  note_launch();
  // H2: bucket offsets
  TRY(ensure(g->boff, (size_t)(nbk + 1) * 8));
  TRY(ensure(g->moff, (size_t)(Mm + 1) * 8));
  if (tiledm) {
    TRY(ensure(g->mtoff, (size_t)(nmt + 1) * 8 + 256));
    TRY(ensure(g->tmp[7], scan_tmp_bytes(nmt + 1) + 4096));
    stmp = g->tmp[7].p;
    TRY((exclusive_scan<int32_t, int64_t>(P<int32_t>(g->mtc), P<int64_t>(g->mtoff), nmt, stmp, s)));
    k_bucket_starts<<<grid_for(Mm + 1, 256), 256, 0, s>>>(Mm, ntile, P<int64_t>(g->mtoff),
                                                         P<int64_t>(g->moff));
    note_launch();
  } else {
    TRY((exclusive_scan<int32_t, int64_t>(P<int32_t>(g->mcnt), P<int64_t>(g->moff), Mm, stmp, s)));
  }
  int32_t *cm = nullptr;
  int64_t *cmo = nullptr;
  if (tiled) {
    const long long ncm = (long long)nbk * ntile;
    TRY(ensure(g->tmp[5], (size_t)ncm * 4 + 256));
    TRY(ensure(g->tmp[6], (size_t)(ncm + 1) * 8 + 256));
    TRY(ensure(g->tmp[7], scan_tmp_bytes(ncm + 1) + 4096));
    stmp = g->tmp[7].p;
    cm = P<int32_t>(g->tmp[5]);
    cmo = P<int64_t>(g->tmp[6]);
    k_bin_tile_count<<<ntile, 256, (size_t)nbk * 4, s>>>(C, nbk, ntile, tsh, P<uint8_t>(g->ckind),
                                                        P<uint8_t>(g->hflag),
                                                        P<int32_t>(g->cell_bin), cm);
    note_launch();
    TRY((exclusive_scan<int32_t, int64_t>(cm, cmo, ncm, stmp, s)));
    k_bucket_starts<<<grid_for(nbk + 1, 256), 256, 0, s>>>(nbk, ntile, cmo, P<int64_t>(g->boff));
    note_launch();
  } else {
    TRY((exclusive_scan<int32_t, int64_t>(P<int32_t>(g->bcnt), P<int64_t>(g->boff), nbk, stmp, s)));
  }
  int hst[8];
  int64_t nbl, nml;
  {
    const D2H it[3] = {{hst, g->status.p, 32}, {&nbl, P<int64_t>(g->boff) + nbk, 8},
                       {&nml, P<int64_t>(g->moff) + Mm, 8}};
    TRY(d2h_many(g->stage, it, 3, s));
  }
  if (hst[0] & ST_NONFINITE) {
    set_error("non-finite movable cell coordinate");
    return PL_ERR_NONFINITE;
  }
  if (nml > (int64_t)g->nmov * kMaxCellMacros) {
    set_error("%lld macro-cell overlaps, more than %d per movable cell", (long long)nml,
              kMaxCellMacros);
    return PL_ERR_UNSUPPORTED;
  }
  // H3-H4: bin buckets (ascending cell id) and macro lists (sorted)
  TRY(ensure(g->blist, (size_t)nbl * 4 + 16));
  TRY(ensure(g->mlist, (size_t)nml * 4 + 16));
  if (tiled) {
    if ((size_t)nbk * 20 <= 48 * 1024)
      k_bin_tile_scatter_wc<<<ntile, 256, (size_t)nbk * 20, s>>>(
          C, nbk, ntile, tsh, P<uint8_t>(g->ckind), P<uint8_t>(g->hflag), P<int32_t>(g->cell_bin), cmo,
          P<uint32_t>(g->blist));
    else
      k_bin_tile_scatter<<<ntile, 256, (size_t)nbk * 4, s>>>(C, nbk, ntile, tsh, P<uint8_t>(g->ckind),
                                                            P<uint8_t>(g->hflag),
                                                            P<int32_t>(g->cell_bin), cmo,
                                                            P<uint32_t>(g->blist));
    note_launch();
  } else {
    TRY(ensure(g->bcur, (size_t)(nbk + 1) * 4));
    k_u64_to_u32<<<grid_for(nbk, 256), 256, 0, s>>>(P<uint64_t>(g->boff), P<uint32_t>(g->bcur), nbk);
    note_launch();
    k_bin_scatter_atomic<<<grid_for(C, 256), 256, 0, s>>>(C, P<uint8_t>(g->ckind), P<uint8_t>(g->hflag),
                                                          P<int32_t>(g->cell_bin),
                                                          P<int32_t>(g->bcur), P<uint32_t>(g->blist));
    note_launch();
    TRY(ensure(g->tmp[3], segsort_tmp_bytes(nbk, nbl, 4)));
    TRY((segmented_sort<uint32_t, MODE_SORT>(P<uint32_t>(g->blist), P<int64_t>(g->boff), nbk,
                                             nbl, nullptr, nullptr, nullptr, g->tmp[3].p, s)));
  }
  const bool cmem_ok = tiledm && !(hst[0] & ST_MANY_OVL);  // every hint cell's macros recorded
  if (!cmem_ok && Mm) {
    TRY(ensure(g->mcur, (size_t)(Mm + 1) * 4));
    k_u64_to_u32<<<grid_for(Mm, 256), 256, 0, s>>>(P<uint64_t>(g->moff), P<uint32_t>(g->mcur), Mm);
    note_launch();
    k_macro_scatter<<<grid_for(C, 256), 256, 0, s>>>(
        G, xy, P<uint8_t>(g->ckind), P<uint8_t>(g->hflag), P<float>(g->cw), P<float>(g->ch),
        P<int64_t>(g->gptr), P<uint32_t>(g->glist), P<float4>(g->ggeo), P<int32_t>(g->mcur),
        P<uint32_t>(g->mlist));
    note_launch();
    TRY(ensure(g->tmp[3], segsort_tmp_bytes(Mm, nml, 4)));
    TRY((segmented_sort<uint32_t, MODE_SORT>(P<uint32_t>(g->mlist), P<int64_t>(g->moff), Mm, nml,
                                             nullptr, nullptr, nullptr, g->tmp[3].p, s)));
  }
  // H5: densities and phi on the side stream, the tiled macro lists on a
  // third one, while the row lengths and the layout go on (both joined
  // before the assembly)
  TRY(ensure_side2(g));
  cudaStream_t s2 = g->side, s3 = g->side2;
  TRY(ensure(g->Db, (size_t)NB * 8 + 16));
  TRY(ensure(g->phi, (size_t)NB * 8 + 16));
  TRY(ensure(g->tmp[4], (size_t)NB * 8 + 256));
  float *phif = P<float>(g->tmp[4]), *phil = phif + NB;  // phi_b as double-floats
  SideJoin join{g, s, true};
  TRY(cudaEventRecord(g->ev_fork, s));
  TRY(cudaStreamWaitEvent(s2, g->ev_fork, 0));
  TRY(cudaStreamWaitEvent(s3, g->ev_fork, 0));
  if (cmem_ok) {
    static std::once_flag attr_once;
    std::call_once(attr_once, [] {
      cudaFuncSetAttribute(k_macro_tile_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kMaxSmemMacros * 6);
    });
    k_macro_tile_scatter<<<ntile, 256, (size_t)Mm * 6, s3>>>(C, P<int32_t>(g->n_ovl),
                                                            P<int32_t>(g->cmem), Mm, ntile, tsh,
                                                            P<int64_t>(g->mtoff),
                                                            P<uint32_t>(g->mlist));
    note_launch();
  }
  LevelBufs lv;
  int nlev = 0;  // launches: level L exists while 64^(L+1) < the longest bin
  {
    size_t sizes[kMaxLevels], tot = 0;
    size_t prev = (size_t)nbl;
    for (int k = 0; k < kMaxLevels; ++k) {
      sizes[k] = prev / 64 + (size_t)NB + 2;
      tot += sizes[k];
      prev = sizes[k];
    }
    TRY(ensure(g->hubtmp, tot * 8 + 256));
    double *q = P<double>(g->hubtmp);
    for (int k = 0; k < kMaxLevels; ++k) {
      lv.base[k] = q;
      q += sizes[k];
    }
    double span = 64.0;
    while (nlev < kMaxLevels && (double)nbl > span) {
      ++nlev;
      span *= 64.0;
    }
    for (int L = 0; L < nlev; ++L) {
      // blocks of 64 threads, so that the first level's FP64 sums spread over every SM
      k_dens_level<<<grid_for((long long)sizes[L], 64, 152 * 64), 64, 0, s2>>>(
          NB, L, P<int64_t>(g->boff), P<uint32_t>(g->blist), P<double>(g->carea),
          L ? lv.base[L - 1] : nullptr, lv.base[L], (long long)sizes[L]);
      note_launch();
    }
  }
  k_dens_final<<<grid_for(NB, 32), 32, 0, s2>>>(  // a warp per 32 bins: spread over the SMs
      G, nlev, P<int64_t>(g->boff), P<uint32_t>(g->blist), P<double>(g->carea), lv,
      P<double>(g->amac), g->abin, p->capacity, p->mu, P<double>(g->Db), P<double>(g->Cb),
      P<double>(g->phi), phif, phil);
  note_launch();
  // the bin rows' chunks, from the bucket starts
  const long long nbc_max = nbl / kBinChunk + NB + 1;  // chunks at most (the grid size)
  g->nbc_max = nbc_max;
  TRY(ensure(g->bchunk, (size_t)(NB + 1) * 4 + 256));
  TRY(ensure(g->cown, (size_t)nbc_max * 4 + 256));
  if (NB <= kBinsOneBlock) {
    k_bin_chunks<<<1, 1024, 0, s2>>>(NB, P<int64_t>(g->boff), P<int32_t>(g->bchunk), P<int32_t>(g->cown));
    note_launch();
  } else {
    TRY(ensure(g->bcur, (size_t)(NB + 1) * 4 + 256));
    TRY(ensure(g->tmp[5], scan_tmp_bytes(NB) + 4096));
    int32_t *cnt = P<int32_t>(g->bcur);
    k_bin_chunk_count<<<grid_for(NB, 256), 256, 0, s2>>>(NB, P<int64_t>(g->boff), cnt);
    note_launch();
    TRY((exclusive_scan<int32_t, int32_t>(cnt, P<int32_t>(g->bchunk), NB, g->tmp[5].p, s2)));
    k_chunk_bins<<<grid_for(nbc_max, 256), 256, 0, s2>>>(NB, nbc_max, P<int32_t>(g->bchunk),
                                                        P<int32_t>(g->cown));
    note_launch();
  }
  TRY(cudaEventRecord(g->ev_join, s2));
  // H6-H7: row lengths and layout
  LayIn LA{};
  LA.G = G;
  LA.srp = P<int64_t>(g->srp);
  LA.hflag = P<uint8_t>(g->hflag);
  LA.cell_bin = P<int32_t>(g->cell_bin);
  LA.n_ovl = P<int32_t>(g->n_ovl);
  LA.moff = P<int64_t>(g->moff);
  LayTotals *tot;
  size_t nl_max, nc_max;
  const int W = g->W;
  const size_t wb = g->wdtype == PL_W_BF16 ? 2 : 4;
  const size_t later = (size_t)C * (8 + W * wb + 4) + (size_t)(NB + 1) * 8 +
                       (size_t)nbc_max * (4 + kBinChunk * W * wb + 32 * W) + 16 * 512;
  pl_status st = layout_hints(g, LA, nml, !tight && (cmem_ok || Mm == 0), later, s, &tot, &nl_max, &nc_max);
  if (st != PL_OK) return st;
  SpMat &m = g->hm;
  // H9: hint parts of cells (macro entries, window blocks) and degrees of
  // every real node
  TRY(ensure(g->mac_base, (size_t)C * 8 + 16));
  TRY(ensure(g->hbw, (size_t)C * W * m.wbytes + 64));
  TRY(ensure(g->hbin, (size_t)C * 4 + 16));
  // the largest key (lambda_up), then the counts of window slots and hint cells
  unsigned long long *key = reinterpret_cast<unsigned long long *>(P<double>(m.lam) + 2), *counts = key + 1;
  TRY(cudaMemsetAsync(key, 0, 24, s));
  TRY(cudaStreamWaitEvent(s, g->ev_join, 0));  // phi
  (g->wdtype == PL_W_BF16 ? k_assemble_hints<true> : k_assemble_hints<false>)
      <<<grid_for(g->Nst, 256), 256, 0, s>>>(
      G, exp_table(), P<uint32_t>(m.rp_s), P<int32_t>(m.longidx), P<uint64_t>(m.lptr),
      P<dfl>(g->st.dsum), P<dfl>(g->st.psum), P<uint8_t>(g->hflag), P<int32_t>(g->cell_bin),
      P<int32_t>(g->n_ovl), xy, P<float>(g->cw), P<float>(g->ch), P<int64_t>(g->gptr),
      P<uint32_t>(g->glist), P<float4>(g->ggeo), P<double>(g->base_w), phif, phil, P<double>(g->phi),
      W, cmem_ok ? P<int32_t>(g->cmem) : nullptr, P<float4>(g->mgeo), P<int32_t>(m.col), m.w.p,
      g->hbw.p, P<int32_t>(g->hbin), P<dfl>(m.dsum), P<dfl>(m.psum), P<uint64_t>(g->mac_base),
      counts);
  note_launch();
  // macro rows (their entries and degree partials) on the third stream, behind
  // the macro lists there, beside the bin rows' blocks and degrees here
  TRY(ensure(g->tmp[5], (nc_max + 1) * 2 * sizeof(dfl) + 256));
  dfl *cpart = P<dfl>(g->tmp[5]);
  TRY(cudaEventRecord(g->ev_fork, s));
  TRY(cudaStreamWaitEvent(s3, g->ev_fork, 0));
  if (nc_max) {
    k_hub_chunks<<<(int)(nc_max < 152 * 32 ? nc_max : 152 * 32), 256, 0, s3>>>(
        G, g->wdtype, &tot->c, P<int32_t>(m.chunk_lr), P<int32_t>(m.lrow), P<uint64_t>(m.lptr),
        P<int32_t>(m.lchunk), P<int64_t>(g->moff), P<uint32_t>(g->mlist), P<int32_t>(g->n_ovl),
        P<uint64_t>(g->mac_base), P<int32_t>(m.col), m.w.p, cpart);
    note_launch();
  }
  TRY(cudaEventRecord(g->ev_join2, s3));
  // H10: bin rows (degree partials of the window blocks, chunk by chunk)
  const BinGeo B = make_bingeo(g);
  // the chunks' copy of the window blocks (read slot by slot by the bin rows)
  TRY(ensure(g->hbwq, (size_t)nbc_max * kBinChunk * W * m.wbytes + 64));
  {
    const long long nth = nbc_max * kBinChunk;
    if (g->wdtype == PL_W_BF16)
      k_blocks_to_chunks<uint16_t><<<grid_for(nth, 256), 256, 0, s>>>(
          nth, W, P<int32_t>(g->bchunk), NB, P<int32_t>(g->cown), P<int64_t>(g->boff),
          P<uint32_t>(g->blist), P<uint16_t>(g->hbw), P<uint16_t>(g->hbwq));
    else
      k_blocks_to_chunks<uint32_t><<<grid_for(nth, 256), 256, 0, s>>>(
          nth, W, P<int32_t>(g->bchunk), NB, P<int32_t>(g->cown), P<int64_t>(g->boff),
          P<uint32_t>(g->blist), P<uint32_t>(g->hbw), P<uint32_t>(g->hbwq));
    note_launch();
  }
  TRY(ensure(g->bdeg, (size_t)nbc_max * W * 16 + 256));
  TRY(ensure(g->bpart, (size_t)nbc_max * W * 16 + 256));
  const long long bwant = (nbc_max + kBinThreads / 32 - 1) / (kBinThreads / 32);
  const int bgrid = (int)(bwant < 152 * 16 ? bwant : 152 * 16);
  TRY(launch_bin_partials<true>(g->wdtype, bgrid, s, B, P<int32_t>(g->bchunk), P<int32_t>(g->cown),
                                 P<int64_t>(g->boff), P<uint32_t>(g->blist), g->hbwq.p, nullptr,
                                 P<float4>(g->bdeg)));
  note_launch();
  TRY(cudaStreamWaitEvent(s, g->ev_join2, 0));
  join.armed = false;
  if (nl_max) {
    k_hub_finalize<<<grid_for((long long)nl_max * 32, 256), 256, 0, s>>>(
        G, B, &tot->f, P<int32_t>(m.lrow), P<int32_t>(m.lchunk), cpart, P<int32_t>(g->bchunk),
        P<float4>(g->bdeg),
        P<dfl>(m.dsum), P<dfl>(m.psum));
    note_launch();
  }
  // H11: lambda_up and coefficients
  k_lambda_max<<<grid_for(N, 256, 152 * 8), 256, 0, s>>>(N, P<dfl>(m.psum), key);
  note_launch();
  // (one wave of blocks: each forms 1 / lambda_up once)
  k_coef<<<grid_for(N, 256, 152 * 8), 256, 0, s>>>(N, P<dfl>(m.dsum), key, P<double>(m.lam), status,
                                                  P<float>(m.c32), &tot->f, P<int32_t>(m.lrow),
                                                  P<double>(m.c64l));
  note_launch();
  TRY(cudaGetLastError());
  {
    unsigned long long ns[2] = {0, 0};
    LayTotals t;
    const D2H it[3] = {{hst, g->status.p, 32}, {ns, counts, 16}, {&t, tot, sizeof(LayTotals)}};
    TRY(d2h_many(g->stage, it, 3, s));
    lay_totals(m, t);
    TRY(ensure(m.part, (size_t)(t.c + 1) * 16));
    g->nslot = (int64_t)ns[0];
    g->nhint = (int64_t)ns[1];
  }
  memcpy(g->lam_h, hst + 4, sizeof(g->lam_h));
  g->have_hints = true;
  if (hst[0] & ST_SPECTRUM) {
    set_error("lambda_up <= 0 or not finite: the refinement filter is undefined");
    return PL_ERR_SPECTRUM;
  }
  return PL_OK;
}

// A workspace that does not hold the build with its quicker, larger tables is
// refused only when it does not hold the smallest one either.
pl_status build_hints(pl_graph *g, const pl_params *p, const float *xy, cudaStream_t s) {
  const pl_status st = build_hints_in(g, p, xy, false, s);
  if (st != PL_ERR_WORKSPACE) return st;
  g->arena.short_need = 0;
  return build_hints_in(g, p, xy, true, s);
}

}  // namespace pl
