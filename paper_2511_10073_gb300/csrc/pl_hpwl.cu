// A5: half-perimeter wirelength (the quality metric of Sec. VII-VIII):
// sum over nets of (max - min) pin x + (max - min) pin y, pin = cell centre +
// offset.  A warp takes 32 consecutive nets at a time and brings their pins'
// positions through shared memory in windows; a lane spans its own net there,
// the warp together the part of a net of more than kHpwlLane pins; nets of more
// than kHpwlWarpMax pins are left to the whole block.  Pin positions and
// extrema are FP32 (min/max are exact); each net's span is formed exactly and
// summed in double-float per thread, the threads' sums in FP64.  Per-block sums
// go to the caller's workspace; the last block to finish (ticket) adds them in a
// fixed order (strided over its threads, then a fixed tree), so the result does
// not depend on scheduling.  A pin whose cell index is out of range makes the
// result NaN (it is not dereferenced).
#include <cmath>
#include <mutex>

#include "pl_internal.h"

namespace pl {

constexpr int kHpwlThreads = 256;
constexpr int kHpwlBlocks = 152 * 8;
constexpr int kHpwlPerSm = 4;
constexpr int kHpwlGrid = 152 * kHpwlPerSm;     // what is launched: one wave of resident blocks
constexpr int kHpwlWin = 256;        // pins a warp stages at once
constexpr int kHpwlLane = 16;        // pins of a window that one lane spans,
constexpr int kHpwlWide = 4;         // four times as many where more nets than these have more
constexpr int kHpwlWarpMax = 1024;   // longer nets are spanned by a whole block
constexpr int kHpwlList = 31;        // such nets a warp keeps a list of

// Positions of pins k0, k0 + stride, ... (n of them, those below e): all
// cell indices and offsets are loaded, then all cells gathered.  A pin_cell
// outside [0, C) sets bad and reads cell 0 instead (the call then reports NaN):
// nothing is written or branched on between the loads, so they stay in flight
// together.
constexpr int kPins = 4;  // of a window
template <int n>
__device__ __forceinline__ void pin_pos(const float2 *xy, const int32_t *pin_cell, const float *dx,
                                        const float *dy, long long k0, int stride, long long e,
                                        int32_t C, bool &bad, float2 *p) {
  int32_t c[n];
  float ox[n], oy[n];
#pragma unroll
  for (int u = 0; u < n; ++u) {
    const long long k = k0 + (long long)u * stride;
    const bool in = k < e;
    c[u] = in ? __ldg(pin_cell + k) : 0;
    ox[u] = in && dx ? __ldg(dx + k) : 0.f;
    oy[u] = in && dy ? __ldg(dy + k) : 0.f;
  }
#pragma unroll
  for (int u = 0; u < n; ++u) {
    const bool ok = (uint32_t)c[u] < (uint32_t)C;
    const bool in = k0 + (long long)u * stride < e;
    bad |= in && !ok;
    p[u] = in && C > 0 ? xy[ok ? c[u] : 0] : make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int u = 0; u < n; ++u) {
    if (dx) p[u].x += ox[u];
    if (dy) p[u].y += oy[u];
  }
}

// A net's span (x1 - x0) + (y1 - y0) added to a double-float sum: each
// difference is exact as a TwoSum pair (FP32 arithmetic only).
__device__ __forceinline__ void span_add(dfl &acc, float x0, float x1, float y0, float y1) {
  dfl dx{x1, 0.f}, dy{y1, 0.f};
  df_add(dx, -x0);
  df_add(dy, -y0);
  df_add_df(acc, dx);
  df_add_df(acc, dy);
}

struct Extent {
  // no pin yet: an empty range (NaN coordinates leave it as it is)
  float x0 = HUGE_VALF, x1 = -HUGE_VALF, y0 = HUGE_VALF, y1 = -HUGE_VALF;
  __device__ __forceinline__ void add(float2 p) {
    x0 = fminf(x0, p.x); x1 = fmaxf(x1, p.x);
    y0 = fminf(y0, p.y); y1 = fmaxf(y1, p.y);
  }
  __device__ __forceinline__ void add(const Extent &e) {
    x0 = fminf(x0, e.x0); x1 = fmaxf(x1, e.x1);
    y0 = fminf(y0, e.y0); y1 = fmaxf(y1, e.y1);
  }
  // a net all of whose pins are NaN on an axis has no span there
  __device__ __forceinline__ void close() {
    if (x0 > x1) x0 = x1 = __int_as_float(0x7fc00000);
    if (y0 > y1) y0 = y1 = __int_as_float(0x7fc00000);
  }
  __device__ __forceinline__ void warp() {  // over the lanes
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, m));
      x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, m));
      y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, m));
      y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, m));
    }
  }
};

// This thread's share of pins [b, e) (every nt-th from t), one at a time: the
// block's warps cover one another's gathers (300 nets of 20000 pins: 4973 us; four
// pins in flight a thread, 6963 us).
__device__ __forceinline__ Extent strided_extent(const float2 *xy, const int32_t *pin_cell,
                                                 const float *dx, const float *dy, long long b,
                                                 long long e, int t, int nt, int32_t C, bool &bad) {
  Extent q;
  for (long long k = b + t; k < e; k += nt) {
    float2 p;
    pin_pos<1>(xy, pin_cell, dx, dy, k, nt, e, C, bad, &p);
    q.add(p);
  }
  return q;
}

// Bound by the latency of net_ptr -> pin_cell -> xy gathers: the next batch's
// net_ptr is loaded a batch ahead, and a window's cell indices, then its gathers,
// go out together (nothing is counted or branched on in between: the check of
// an index used to end each gather's wait before the next index was loaded).
// Windows take any batch (before, a batch above its stage of 512 pins fell back to
// a lane per net straight from memory, and every block looked through its nets
// once more for the long ones).  2.25M nets, 8.9M pins: 150 -> 77 us (five blocks
// a SM spill: 96 us; eight pins in flight a lane: 92 us).
// Long nets: spanned by the block whatever their number (those that did not fit a
// list of eight used to be left to one warp, window by window: 20 nets of 500000
// pins 71.9 ms, now 9.3 ms).  The pins are read by plain loads, so that a netlist
// that L2 holds stays there for the next score (600k cells: 33.5 us with loads
// that are evicted first, 27.9 us).
__global__ void __launch_bounds__(kHpwlThreads, kHpwlPerSm) k_hpwl(const int64_t *net_ptr,
                                                          const int32_t *pin_cell,
                                                          const float *dx, const float *dy,
                                                          const float2 *xy, int32_t M, int32_t C,
                                                          double *part, int *ticket, double *out) {
  __shared__ double red[kHpwlThreads / 32];
  __shared__ int last;
  __shared__ float2 stage_all[kHpwlThreads / 32][kHpwlWin];
  __shared__ int32_t list[kHpwlThreads / 32][kHpwlList + 1];
  __shared__ int nlongs[kHpwlThreads / 32];
  __shared__ float4 mm[kHpwlThreads / 32];
  float2 *stg = stage_all[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  dfl acc{0.f, 0.f};
  int nlong = 0;  // the same in every lane
  bool bad = false;
  const long long wg = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long step = (((long long)gridDim.x * blockDim.x) >> 5) * 32;
  auto ptr = [&](long long e) { return net_ptr[e < M ? e : M]; };
  long long na = 0, nz = 0;  // the next batch's pin range of this lane's net
  if (wg * 32 < M) {
    na = ptr(wg * 32 + lane);
    nz = ptr(wg * 32 + lane + 1);
  }
  for (long long base = wg * 32; base < M; base += step) {
    const long long a = na, z = nz;
    if (base + step < M) {
      na = ptr(base + step + lane);
      nz = ptr(base + step + lane + 1);
    }
    const long long p0 = __shfl_sync(0xffffffffu, a, 0), p1 = __shfl_sync(0xffffffffu, z, 31);
    const bool isl = z - a > kHpwlWarpMax;
    for (unsigned t = __ballot_sync(0xffffffffu, isl); t; t &= t - 1) {  // kept for later
      const int src = __ffs(t) - 1;
      if (nlong < kHpwlList) {
        if (lane == 0) list[wid][nlong] = (int32_t)(base + src);
      } else if (nlong == kHpwlList && lane == 0) {
        list[wid][kHpwlList] = (int32_t)(base + src);  // the first that the list does not hold
      }
      nlong = min(nlong + 1, kHpwlList + 1);
    }
    Extent q;
    for (long long c0 = p0; c0 < p1;) {
      // a window ends at the next long net and starts behind one
      long long e1 = p1;
      const unsigned nx = __ballot_sync(0xffffffffu, isl && z > c0);
      if (nx) {
        const long long la = __shfl_sync(0xffffffffu, a, __ffs(nx) - 1);
        if (la <= c0) {
          c0 = __shfl_sync(0xffffffffu, z, __ffs(nx) - 1);
          continue;
        }
        e1 = la;
      }
      const int n = (int)(e1 - c0 < kHpwlWin ? e1 - c0 : kHpwlWin);
      for (int k0 = 0; k0 < n; k0 += kPins * 32) {
        float2 p[kPins];
        pin_pos<kPins>(xy, pin_cell, dx, dy, c0 + k0 + lane, 32, c0 + n, C, bad, p);
#pragma unroll
        for (int u = 0; u < kPins; ++u)
          if (k0 + 32 * u + lane < n) stg[k0 + 32 * u + lane] = p[u];
      }
      __syncwarp();
      // this lane's net's part of the window
      const int lo = (int)(a > c0 ? (a - c0 < n ? a - c0 : n) : 0);
      const int hi = (int)(z > c0 ? (z - c0 < n ? z - c0 : n) : 0);
      // the warp together takes a net of more than kHpwlLane pins, about 150 clocks a net;
      // where there are many, the lanes take theirs at once up to four times that
      // (100k nets of 17 pins: 42.8 -> 33.3 us)
      bool wide = hi - lo > kHpwlLane;
      if (__popc(__ballot_sync(0xffffffffu, wide)) > kHpwlWide) wide = hi - lo > 4 * kHpwlLane;
      if (!wide)
        for (int k = lo; k < hi; ++k) q.add(stg[k]);
      for (unsigned t = __ballot_sync(0xffffffffu, wide); t; t &= t - 1) {
        const int src = __ffs(t) - 1;
        const int l = __shfl_sync(0xffffffffu, lo, src), h = __shfl_sync(0xffffffffu, hi, src);
        Extent r;
        for (int k = l + lane; k < h; k += 32) r.add(stg[k]);
        r.warp();
        if (lane == src) q.add(r);
      }
      __syncwarp();
      c0 += n;
    }
    if (!isl && z > a) {
      q.close();
      span_add(acc, q.x0, q.x1, q.y0, q.y1);
    }
  }
  // The block's long nets, warp by warp, in order.  Those that a warp's list does not
  // hold are found by looking through its batches from there once more.
  if (lane == 0) nlongs[wid] = nlong;
  auto long_nets = [&](int w, auto f) {  // the same in every thread
    for (int i = 0; i < min(nlongs[w], kHpwlList); ++i) {
      const long long e = list[w][i];
      f(net_ptr[e], net_ptr[e + 1]);
    }
    if (nlongs[w] <= kHpwlList) return;
    const long long first = list[w][kHpwlList];
    for (long long base = first & ~31LL; base < M; base += step) {
      const long long e = base + lane, a = ptr(e), z = ptr(e + 1);
      for (unsigned t = __ballot_sync(0xffffffffu, z - a > kHpwlWarpMax && e >= first); t; t &= t - 1) {
        const int src = __ffs(t) - 1;
        f(__shfl_sync(0xffffffffu, a, src), __shfl_sync(0xffffffffu, z, src));
      }
    }
  };
  __syncthreads();
  double bigacc = 0.0;  // thread 0
  for (int w = 0; w < kHpwlThreads / 32; ++w)
    long_nets(w, [&](long long a, long long z) {
      Extent r = strided_extent(xy, pin_cell, dx, dy, a, z, threadIdx.x, kHpwlThreads, C, bad);
      r.warp();
      if (lane == 0) mm[wid] = make_float4(r.x0, r.x1, r.y0, r.y1);
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int k = 1; k < kHpwlThreads / 32; ++k) {
          const float4 t = mm[k];
          r.x0 = fminf(r.x0, t.x); r.x1 = fmaxf(r.x1, t.y);
          r.y0 = fminf(r.y0, t.z); r.y1 = fmaxf(r.y1, t.w);
        }
        r.close();
        bigacc += ((double)r.x1 - (double)r.x0) + ((double)r.y1 - (double)r.y0);
      }
      __syncthreads();
    });
  if (bad) atomicAdd(ticket + 1, 1);
  const double accd = warp_sum(df_to_d(df_norm(acc)));
  if (lane == 0) red[wid] = accd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < kHpwlThreads / 32; ++k) s += red[k];
    part[blockIdx.x] = s + bigacc;
    __threadfence();
    last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  // the last block: thread t adds partials t, t + 256, ... in order, then a
  // fixed tree over the threads
  __threadfence();
  double s = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += kHpwlThreads) s += __ldcg(&part[k]);
  s = warp_sum(s);
  if (lane == 0) red[wid] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kHpwlThreads / 32; ++k) t += red[k];
    *out = __ldcg(ticket + 1) ? __longlong_as_double(0x7ff8000000000000LL) : t;
    ticket[0] = 0;
    ticket[1] = 0;
  }
}

int hpwl_blocks(int32_t M) { return grid_for((long long)M, kHpwlThreads, kHpwlBlocks); }

size_t hpwl_ws_bytes(int32_t M) { return 256 + (size_t)hpwl_blocks(M) * sizeof(double); }

cudaError_t launch_hpwl(const pl_netlist *nl, const float *xy, double *out, void *ws,
                        cudaStream_t s) {
  const int nb = grid_for((long long)nl->num_nets, kHpwlThreads, kHpwlGrid);  // at most hpwl_blocks
  int *ticket = reinterpret_cast<int *>(ws);
  double *part = reinterpret_cast<double *>(static_cast<char *>(ws) + 256);
  k_hpwl<<<nb, kHpwlThreads, 0, s>>>(nl->net_ptr, nl->pin_cell, nl->pin_dx, nl->pin_dy,
                                     reinterpret_cast<const float2 *>(xy), nl->num_nets,
                                     nl->num_cells, part, ticket, out);
  note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------- allocation-free variant
// Scratch of pl_hpwl_noalloc: the ticket words and one FP64 partial per block
// of the largest grid k_hpwl is ever launched with (kHpwlBlocks), in a
// file-scope device array of about 10 KB.  Every GPU that loads the library
// holds it until the process exits, and every call shares it.
constexpr int kNoAllocBlocks = kHpwlBlocks;
constexpr size_t kNoAllocBytes = 256 + (size_t)kNoAllocBlocks * sizeof(double);
static __device__ __align__(256) unsigned char g_hpwl_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
static std::mutex g_noalloc_mu;
static void *g_noalloc_ptr[kMaxDevices] = {};

// Device address of the scratch on the current device.  Host code cannot use
// the symbol itself (it names a host-side stand-in), so the address is looked
// up once per device, with that device current, and cached.
static cudaError_t noalloc_scratch(void **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_hpwl_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace pl

extern "C" pl_status pl_hpwl_noalloc(const pl_netlist *nl, const float *xy_cells, double *hpwl,
                                     pl_stream stream) {
  using namespace pl;
  clear_error();
  if (!nl || !xy_cells || !hpwl) {
    set_error("NULL argument");
    return PL_ERR_INVALID_ARG;
  }
  if (nl->num_nets < 0 || nl->num_cells < 0 || !nl->net_ptr || (nl->num_pins && !nl->pin_cell)) {
    set_error("bad netlist");
    return PL_ERR_INVALID_ARG;
  }
  const int nb = hpwl_blocks(nl->num_nets);
  if (nb > kNoAllocBlocks || hpwl_ws_bytes(nl->num_nets) > kNoAllocBytes) {
    set_error("pl_hpwl_noalloc: %d blocks exceed its fixed scratch of %d blocks", nb,
              kNoAllocBlocks);
    return PL_ERR_UNSUPPORTED;
  }
  void *scratch = nullptr;
  cudaError_t e = noalloc_scratch(&scratch);
  if (e != cudaSuccess) return cuda_fail(e, "pl_hpwl_noalloc scratch lookup");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  e = cudaMemsetAsync(scratch, 0, 8, s);  // ticket and error count start at zero
  if (e == cudaSuccess) e = launch_hpwl(nl, xy_cells, hpwl, scratch, s);
  if (e != cudaSuccess) return cuda_fail(e, "pl_hpwl_noalloc");
  return PL_OK;
}
