// Sec. VI: iteration-scheduled macro charge densities and their bin
// integrals, GPU-side.  For iteration t of a schedule of T iterations, each
// macro m carries a charge density rho_t over its footprint (local offsets
// dx, dy from its centre, zero outside the w x h rectangle):
//   charge redistribution:  rho = 2 eta^2 / (pi erf^2(eta / sqrt 2))
//                                 exp(-2 eta^2 (dx^2 / w^2 + dy^2 / h^2)),
//     eta(t) = eta_B(a)^(1 - s(a)) eta_A(a)^s(a), a = t / T, scheme A
//     eta_A = sqrt(-2 log r(a)) with log r log-linear from r0 to r1, scheme B
//     eta_B = sqrt(2 ln 2) / beta(a) with beta linear from beta_min to
//     beta_max, s the smoothstep between alpha0 and alpha1;
//   charge restoration, exponential-like:  rho = exp(-(tan^2(pi dx / w) +
//     tan^2(pi dy / h)) / (2 sigma^2)), sigma(t) = -sigma_factor T ln(1 - t / T);
//   linear-like:  rho = max(0, 1 - k rr);  sigmoid-like:  rho = 2 / (1 + exp(k rr)),
//     rr = sqrt(2 (dx^2 / w^2 + dy^2 / h^2)), k(t) = k_factor / tan(pi t / (2 T)).
// The density of bin b gains the integral of rho_t over the bin (area units).
// Gaussian: the separable closed form with erf; exponential-like: separable,
// a composite Gauss-Legendre rule per axis; linear- and sigmoid-like: the
// tensor rule on the bin-macro intersection.  FP64, except the radial models'
// point values and their sums within a panel (FP32, about 1e-7 relative; the
// FP64 rate of GB300 would otherwise set the kernel's time).
//
// A CTA owns a tile of bins: it lists the macros near the tile (ascending), forms
// the listed macros' integrals in shared memory, and a thread per bin adds its
// macros' terms in ascending order.
#include <cmath>

#include "pl_internal.h"

namespace pl {

constexpr int kRhoMaxNodes = 32;

struct RhoArgs {
  int panels, nodes;
  double A, c;       // Gaussian: normalization and sqrt(2) eta
  double sscale;     // exponential-like: 1 / (2 sigma^2); < 0: sigma infinite
  int szero;         // exponential-like: sigma = 0 (no charge)
  double k;          // linear- and sigmoid-like; < 0: k infinite (no charge)
  double gx[kRhoMaxNodes], gw[kRhoMaxNodes];  // Gauss-Legendre rule on [-1, 1]
  float gxf[kRhoMaxNodes], gwf[kRhoMaxNodes];  // the same in FP32 (the radial models)
  double mgx, mgy;   // margins of a macro's bin range, in bins (rounding of bin edges)
};

// Composite rule of f over [a, b] (one thread).
template <typename F>
__device__ double gl_1d(const RhoArgs &R, double a, double b, F f) {
  const double hp = (b - a) / R.panels;
  double s = 0.0;
  for (int p = 0; p < R.panels; ++p) {
    const double c = a + (p + 0.5) * hp;
    for (int i = 0; i < R.nodes; ++i) s += 0.5 * hp * R.gw[i] * f(c + 0.5 * hp * R.gx[i]);
  }
  return s;
}

// One axis' factor of a separable model over [a, b] (offsets inside a macro of
// side w), one thread.
template <int MODEL>
__device__ double rho_axis(const RhoArgs &R, double w, double a, double b) {
  if (MODEL == PL_RHO_GAUSS)
    return w * sqrt(M_PI) / (2.0 * R.c) * (erf(R.c * b / w) - erf(R.c * a / w));
  if (R.szero) return 0.0;
  if (R.sscale < 0.0) return b - a;
  auto f = [&](double d) {
    const double tv = tan(M_PI * d / w);
    return exp(-tv * tv * R.sscale);
  };
  return gl_1d(R, a, b, f);
}

// One panel's nodes x nodes points of a radial model, summed in FP32: the
// panel's centre (cu, cv) and half sides (du, dv) over the macro's sides.
template <int MODEL>
__device__ __forceinline__ float rho_panel(const RhoArgs &R, float kf, float cu, float cv,
                                           float du, float dv) {
  float ps = 0.f;
  for (int i = 0; i < R.nodes; ++i) {
    const float u = cu + du * R.gxf[i];
    float row = 0.f;
#pragma unroll 4
    for (int j = 0; j < R.nodes; ++j) {
      const float v = cv + dv * R.gxf[j];
      const float rr = sqrtf(2.0f * (u * u + v * v));
      const float val = MODEL == PL_RHO_LINEAR ? fmaxf(0.0f, 1.0f - kf * rr)
                                                 : 2.0f / (1.0f + __expf(kf * rr));
      row = fmaf(R.gwf[j], val, row);
    }
    ps = fmaf(R.gwf[i], row, ps);
  }
  return ps;
}

// A CTA of 256 threads per tile of tbx x tby bins (at most 256).
//  1. Cull: the threads test all macros against the tile in FP32 with a margin
//     that covers its rounding (a macro is dropped only when it cannot touch the
//     tile), 1024 macros in flight, and append the rest to a list in macro order.
//  2. In batches of the list, each macro's range of bins in the tile; then
//     separable models: a thread per (macro, bin column or row) forms that axis'
//     factor; radial models: half a warp per (macro, bin) pair, a lane per
//     panel.  Terms go to a table in shared memory.
//  3. A thread per bin adds the batch's terms in macro order.
// FP64 bound (2 FP64 operations per clock and SM): a factor is formed once per
// macro and bin column of a tile, not once per bin and macro, a macro far from
// the tile costs no FP64, and the radial rule converts nothing per point.
// Before, every warp tested every macro in FP64 for its 8 x 4 bins and each lane
// formed its bin's whole integral.  GB300, 8000 macros on 512 x 512 bins,
// Gaussian: 2194 -> 70 us; 550 macros on 256 x 256 bins, sigmoid-like: 1007 -> 109 us.
constexpr int kRhoThreads = 256;
constexpr int kRhoCull = 4;      // macros per thread and round of the cull
constexpr int kRhoList = 1280;   // macros listed before a flush
constexpr int kRhoBatch = 64;    // macros of a batch at most
constexpr int kRhoTable = 2048;  // table entries: terms of a batch
constexpr int kRhoAxes = 64 * 12;  // axis entries of a batch (radial models)
// a table entry of an empty interval (an integral is never negative)
__device__ __forceinline__ bool rho_none(double v) { return __double2hiint(v) == (int)0xbff00000; }

// The panels of a radial model along one axis of a (macro, bin column or row):
// panel side, half a panel and the panel centres over the macro's side.
constexpr int kRhoAxisP = 5;
struct RhoAxis {
  double hp;  // < 0: empty interval
  float d, c[kRhoAxisP];
};

struct RhoMacro {
  double cx, cy, w, h;
  int i0, j0, ni, nj;  // bins of the tile that the macro may touch: first, count
};

template <int MODEL>
__global__ void __launch_bounds__(kRhoThreads) k_macro_density(
    RhoArgs R, int32_t nm, const float *mx, const float *my, const float *mw, const float *mh,
    double xl, double yl, double wb, double hb, int nbx, int nby, int tbx, int tby, double *out) {
  __shared__ int32_t list[kRhoList];
  __shared__ int wcnt[kRhoCull][kRhoThreads / 32];
  __shared__ RhoMacro mac[kRhoBatch];
  __shared__ int pre[kRhoBatch + 1];  // tasks before each macro of the batch
  __shared__ double tab[kRhoTable];
  constexpr bool radial = MODEL == PL_RHO_LINEAR || MODEL == PL_RHO_SIGMOID;
  __shared__ RhoAxis axes[radial ? kRhoAxes : 1];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int stride = radial ? tbx * tby : tbx + tby;  // table entries of a macro
  const int batch = min(min(kRhoBatch, kRhoTable / stride), kRhoAxes / (tbx + tby));
  const int ntx = (nbx + tbx - 1) / tbx;
  const int bx0 = (int)(blockIdx.x % ntx) * tbx, by0 = (int)(blockIdx.x / ntx) * tby;
  const int nx = min(tbx, nbx - bx0), ny = min(tby, nby - by0);
  const int tx = tid % tbx, ty = tid / tbx;  // this thread's bin of the tile
  const bool mine = tx < nx && ty < ny;
  // the tile's centre and half sides for the cull
  const float tcx = (float)(xl + (bx0 + 0.5 * nx) * wb), thx = (float)(0.5 * nx * wb);
  const float tcy = (float)(yl + (by0 + 0.5 * ny) * hb), thy = (float)(0.5 * ny * hb);
  const double iwb = 1.0 / wb, ihb = 1.0 / hb;
  double acc = 0.0;

  auto flush = [&](int n) {
    for (int b0 = 0; b0 < n; b0 += batch) {
      const int nb = min(batch, n - b0);
      if (tid < nb) {
        const int m = list[b0 + tid];
        RhoMacro q;
        q.cx = mx[m];
        q.cy = my[m];
        q.w = mw[m];
        q.h = mh[m];
        // bins that [c - w/2, c + w/2] may touch, with a margin for the rounding
        // of the bin edges; the exact test follows per interval
        auto range = [](double c, double w, double o, double ib, double mg, int t0, int t, int *i0,
                        int *ni) {
          const double e = 1e-9 + mg + 1e-14 * (fabs(c) + w) * ib;
          const double lo = fmin(fmax(floor((c - 0.5 * w - o) * ib - e), (double)t0), (double)(t0 + t));
          const double hi = fmax(fmin(floor((c + 0.5 * w - o) * ib + e), (double)(t0 + t - 1)), (double)(t0 - 1));
          *i0 = (int)lo - t0;
          *ni = max(0, (int)hi - (int)lo + 1);
        };
        range(q.cx, q.w, xl, iwb, R.mgx, bx0, nx, &q.i0, &q.ni);
        range(q.cy, q.h, yl, ihb, R.mgy, by0, ny, &q.j0, &q.nj);
        mac[tid] = q;
        pre[tid + 1] = q.ni > 0 && q.nj > 0 ? (radial ? q.ni * q.nj : q.ni + q.nj) : 0;
      }
      if (tid == 0) pre[0] = 0;
      __syncthreads();
      if (wid == 0) {  // inclusive sums of the task counts, 32 macros at a time
        int carry = 0;
        for (int k0 = 0; k0 < nb; k0 += 32) {
          int v = k0 + lane < nb ? pre[k0 + lane + 1] : 0;
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, v, d);
            if (lane >= d) v += t;
          }
          if (k0 + lane < nb) pre[k0 + lane + 1] = carry + v;
          carry += __shfl_sync(0xffffffffu, v, 31);
        }
      }
      __syncthreads();
      const int tasks = pre[nb];
      auto macro_of = [&](int t) {  // the last macro whose tasks start at or before t
        int lo = 0, hi = nb - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (pre[mid] <= t) lo = mid;
          else hi = mid - 1;
        }
        return lo;
      };
      // the macro's part of bin column (row) i, as offsets from its centre
      auto span = [](double o, double b, int i, double c, double w, double *lo, double *hi) {
        *lo = fmax(o + i * b - c, -0.5 * w);
        *hi = fmin(o + (i + 1) * b - c, 0.5 * w);
      };
      if (!radial) {
        for (int t = tid; t < tasks; t += kRhoThreads) {
          const int k = macro_of(t);
          const RhoMacro &q = mac[k];
          int i = t - pre[k];
          const bool isx = i < q.ni;
          double lo, hi, w;
          int slot;
          if (isx) {
            slot = q.i0 + i;
            w = q.w;
            span(xl, wb, bx0 + slot, q.cx, w, &lo, &hi);
          } else {
            slot = q.j0 + i - q.ni;
            w = q.h;
            span(yl, hb, by0 + slot, q.cy, w, &lo, &hi);
            slot += tbx;
          }
          tab[k * stride + slot] = lo < hi ? rho_axis<MODEL>(R, w, lo, hi) : -1.0;
        }
      } else {
        // the panels of each macro's bin columns and rows (all FP64 divisions:
        // per axis, not per pair), then pair t by half a warp, lane hl taking
        // panels hl, hl + 16, ...
        const int hl = lane & 15, P = R.panels, np = P * P;
        const unsigned hmask = lane < 16 ? 0x0000ffffu : 0xffff0000u;
        const float kf = (float)R.k;
        const int np1 = P <= kRhoAxisP ? P : 1;  // a thread per panel centre
        for (int t = tid; t < nb * (tbx + tby) * np1; t += kRhoThreads) {
          const int en = t / np1, p = t - en * np1;
          const int k = en / (tbx + tby), slot = en - k * (tbx + tby);
          const RhoMacro &q = mac[k];
          const bool isx = slot < tbx;
          const int i = isx ? slot : slot - tbx;
          if ((unsigned)(i - (isx ? q.i0 : q.j0)) >= (unsigned)(isx ? q.ni : q.nj)) continue;
          const double w = isx ? q.w : q.h;
          double lo, hi;
          span(isx ? xl : yl, isx ? wb : hb, (isx ? bx0 : by0) + i, isx ? q.cx : q.cy, w, &lo, &hi);
          const double hp = (hi - lo) / P;
          RhoAxis &e = axes[en];
          if (p == 0) {
            e.hp = lo < hi ? hp : -1.0;
            e.d = (float)(0.5 * hp / w);
          }
          if (P <= kRhoAxisP) e.c[p] = (float)((lo + (p + 0.5) * hp) / w);
        }
        __syncthreads();
        for (int t = tid >> 4; t < tasks; t += kRhoThreads / 16) {
          const int k = macro_of(t);
          const RhoMacro &q = mac[k];
          const int r = t - pre[k], i = q.i0 + r % q.ni, j = q.j0 + r / q.ni;
          const RhoAxis &ex = axes[k * (tbx + tby) + i], &ey = axes[k * (tbx + tby) + tbx + j];
          const double hx = ex.hp, hy = ey.hp;
          double v = -1.0;
          if (!rho_none(hx) && !rho_none(hy)) {
            double s = 0.0;
            if (!(R.k < 0.0)) {
              if (P <= kRhoAxisP) {
                for (int e = hl; e < np; e += 16)
                  s += (double)rho_panel<MODEL>(R, kf, ex.c[e / P], ey.c[e % P], ex.d, ey.d);
              } else {
                const double ax = fmax(xl + (bx0 + i) * wb - q.cx, -0.5 * q.w);
                const double ay = fmax(yl + (by0 + j) * hb - q.cy, -0.5 * q.h);
                for (int e = hl; e < np; e += 16) {
                  const int px = e / P, py = e % P;
                  const float cu = (float)((ax + (px + 0.5) * hx) / q.w);
                  const float cv = (float)((ay + (py + 0.5) * hy) / q.h);
                  s += (double)rho_panel<MODEL>(R, kf, cu, cv, ex.d, ey.d);
                }
              }
#pragma unroll
              for (int d = 8; d > 0; d >>= 1) s += __shfl_xor_sync(hmask, s, d, 16);
              s *= 0.25 * hx * hy;
            }
            v = s;
          }
          if (hl == 0) tab[k * stride + j * tbx + i] = v;
        }
      }
      __syncthreads();
      if (mine) {
        for (int k = 0; k < nb; ++k) {
          const RhoMacro &q = mac[k];
          if ((unsigned)(tx - q.i0) >= (unsigned)q.ni || (unsigned)(ty - q.j0) >= (unsigned)q.nj) continue;
          if (radial) {
            const double v = tab[k * stride + ty * tbx + tx];
            if (!rho_none(v)) acc += v;
          } else {
            const double u = tab[k * stride + tx], v = tab[k * stride + tbx + ty];
            if (!rho_none(u) && !rho_none(v)) acc += MODEL == PL_RHO_GAUSS ? R.A * u * v : u * v;
          }
        }
      }
      __syncthreads();  // the batch's shared tables are read
    }
  };

  int nlist = 0;  // the same in every thread
  for (int m0 = 0; m0 < nm; m0 += kRhoCull * kRhoThreads) {
    if (nlist + kRhoCull * kRhoThreads > kRhoList) {
      flush(nlist);
      nlist = 0;
    }
    float x[kRhoCull], y[kRhoCull], w[kRhoCull], h[kRhoCull];
#pragma unroll
    for (int u = 0; u < kRhoCull; ++u) {
      const int m = m0 + u * kRhoThreads + tid;
      const bool in = m < nm;
      x[u] = in ? mx[m] : 0.f;
      y[u] = in ? my[m] : 0.f;
      w[u] = in ? mw[m] : 0.f;
      h[u] = in ? mh[m] : 0.f;
    }
    unsigned bal[kRhoCull];
#pragma unroll
    for (int u = 0; u < kRhoCull; ++u) {
      // dropped only when clearly apart (a comparison with a NaN keeps it)
      const float gx = 0.5f * w[u] + thx, gy = 0.5f * h[u] + thy;
      const bool apart = fabsf(x[u] - tcx) > gx + 1e-6f * (fabsf(x[u]) + fabsf(tcx) + gx) ||
                         fabsf(y[u] - tcy) > gy + 1e-6f * (fabsf(y[u]) + fabsf(tcy) + gy);
      bal[u] = __ballot_sync(0xffffffffu, w[u] > 0.f && h[u] > 0.f && !apart);
      if (lane == 0) wcnt[u][wid] = __popc(bal[u]);
    }
    __syncthreads();
    int at = nlist;
#pragma unroll
    for (int u = 0; u < kRhoCull; ++u) {
      int before = 0, all = 0;
#pragma unroll
      for (int k = 0; k < kRhoThreads / 32; ++k) {
        const int c = wcnt[u][k];
        before += k < wid ? c : 0;
        all += c;
      }
      if (bal[u] >> lane & 1u)
        list[at + before + __popc(bal[u] & ((1u << lane) - 1u))] = m0 + u * kRhoThreads + tid;
      at += all;
    }
    nlist = at;
    __syncthreads();  // the list is written, the counts are read
  }
  if (nlist) flush(nlist);
  if (mine) out[(long long)(by0 + ty) * nbx + bx0 + tx] = acc;
}

// Gauss-Legendre nodes and weights on [-1, 1] (Newton's method on P_n from
// the guesses cos(pi (i - 1/4) / (n + 1/2)); P_n' from the recurrence).
static void legendre_rule(int n, double *x, double *w) {
  for (int i = 1; i <= n; ++i) {
    double z = std::cos(M_PI * (i - 0.25) / (n + 0.5)), dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        const double pk = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = pk;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[i - 1] = -z;
    w[i - 1] = 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

}  // namespace pl

extern "C" {

void pl_rho_params_default(pl_rho_params *p) {
  if (!p) return;
  p->model = PL_RHO_GAUSS;
  p->T = 300;
  p->r0 = 0.05;
  p->r1 = 0.9;
  p->beta_min = 0.25;
  p->beta_max = 1.5;
  p->alpha0 = 0.3;
  p->alpha1 = 0.7;
  p->sigma_factor = 0.002;
  p->k_factor = 0.5;
  p->panels = 4;
  p->nodes = 8;
}

pl_status pl_macro_density(const pl_rho_params *rp, int32_t t, int32_t num_macros,
                           const float *mx, const float *my, const float *mw, const float *mh,
                           double xl, double yl, double xh, double yh, int32_t nbx, int32_t nby,
                           double *rho, pl_stream stream) {
  using namespace pl;
  clear_error();
  if (!rp || !rho || num_macros < 0 || (num_macros && (!mx || !my || !mw || !mh))) {
    set_error("NULL or negative argument");
    return PL_ERR_INVALID_ARG;
  }
  if (nbx < 1 || nby < 1 || !(xh > xl) || !(yh > yl) || !std::isfinite(xl) || !std::isfinite(xh) ||
      !std::isfinite(yl) || !std::isfinite(yh)) {
    set_error("bad bin grid or region");
    return PL_ERR_INVALID_ARG;
  }
  if (rp->model < PL_RHO_GAUSS || rp->model > PL_RHO_SIGMOID || rp->T < 1 || t < 0 || t > rp->T ||
      rp->panels < 1 || rp->panels > 64 || rp->nodes < 1 || rp->nodes > kRhoMaxNodes) {
    set_error("bad schedule parameters (model, T >= 1, 0 <= t <= T, panels 1..64, nodes 1..32)");
    return PL_ERR_INVALID_ARG;
  }
  RhoArgs R{};
  R.panels = rp->panels;
  R.nodes = rp->nodes;
  legendre_rule(rp->nodes, R.gx, R.gw);
  for (int k = 0; k < rp->nodes; ++k) {
    R.gxf[k] = (float)R.gx[k];
    R.gwf[k] = (float)R.gw[k];
  }
  R.mgx = 1e-14 * (std::fabs(xl) + std::fabs(xh)) * nbx / (xh - xl);
  R.mgy = 1e-14 * (std::fabs(yl) + std::fabs(yh)) * nby / (yh - yl);
  const double a = (double)t / (double)rp->T;
  if (rp->model == PL_RHO_GAUSS) {
    if (!(rp->r0 > 0.0 && rp->r0 < 1.0 && rp->r1 > 0.0 && rp->r1 < 1.0 && rp->beta_min > 0.0 &&
          rp->beta_max > 0.0 && rp->alpha1 > rp->alpha0)) {
      set_error("Gaussian schedule needs 0 < r0, r1 < 1, beta > 0, alpha1 > alpha0");
      return PL_ERR_INVALID_ARG;
    }
    const double ea = std::sqrt(-2.0 * ((1.0 - a) * std::log(rp->r0) + a * std::log(rp->r1)));
    const double eb = std::sqrt(2.0 * std::log(2.0)) / (rp->beta_min + (rp->beta_max - rp->beta_min) * a);
    double s = 0.0;
    if (a >= rp->alpha1) s = 1.0;
    else if (a > rp->alpha0) {
      const double z = (a - rp->alpha0) / (rp->alpha1 - rp->alpha0);
      s = 3.0 * z * z - 2.0 * z * z * z;
    }
    const double eta = std::pow(eb, 1.0 - s) * std::pow(ea, s);
    const double e = std::erf(eta / std::sqrt(2.0));
    R.A = 2.0 * eta * eta / (M_PI * e * e);
    R.c = std::sqrt(2.0) * eta;
  } else if (rp->model == PL_RHO_EXP) {
    if (!(rp->sigma_factor > 0.0)) {
      set_error("sigma_factor must be > 0");
      return PL_ERR_INVALID_ARG;
    }
    R.szero = t == 0;
    R.sscale = -1.0;
    if (t > 0 && t < rp->T) {
      const double sg = -rp->sigma_factor * rp->T * std::log(1.0 - a);
      R.sscale = 1.0 / (2.0 * sg * sg);
    }
  } else {
    if (!(rp->k_factor > 0.0)) {
      set_error("k_factor must be > 0");
      return PL_ERR_INVALID_ARG;
    }
    R.k = t == 0 ? -1.0 : (t >= rp->T ? 0.0 : rp->k_factor / std::tan(0.5 * M_PI * a));
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // Tiles: every CTA culls all macros, so larger tiles read the macros less
  // often; smaller ones balance better.  32 x 8 bins for the separable models,
  // whose work per tile is a few factors per macro; 8 x 8 for the radial ones,
  // whose work is a term per bin (550 macros on 256 x 256 bins, sigmoid-like:
  // 16 x 8 115 us, 8 x 8 109 us, 8 x 4 119 us).  8 x 4 when fewer than two tiles
  // per SM would be left.
  const bool radial = rp->model == PL_RHO_LINEAR || rp->model == PL_RHO_SIGMOID;
  int tbx = radial ? 8 : 32, tby = 8;
  auto tiles = [&] {
    return (long long)((nbx + tbx - 1) / tbx) * ((nby + tby - 1) / tby);
  };
  if (tiles() < 2 * 152) tbx = 8, tby = 4;
  auto kernel = rp->model == PL_RHO_GAUSS    ? k_macro_density<PL_RHO_GAUSS>
                : rp->model == PL_RHO_EXP    ? k_macro_density<PL_RHO_EXP>
                : rp->model == PL_RHO_LINEAR ? k_macro_density<PL_RHO_LINEAR>
                                             : k_macro_density<PL_RHO_SIGMOID>;
  kernel<<<(int)tiles(), kRhoThreads, 0, s>>>(R, num_macros, mx, my, mw, mh, xl, yl, (xh - xl) / nbx,
                                              (yh - yl) / nby, nbx, nby, tbx, tby, rho);
  note_launch();
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? PL_OK : cuda_fail(e, "pl_macro_density");
}

}  // extern "C"
