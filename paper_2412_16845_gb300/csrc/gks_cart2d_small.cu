// Several 2-D TM steps in one launch for grids too small to fill the GPU (tau = 0, mu = 1).
//
// On a 64^2 or 100^2 grid a step of the marching kernels is all latency: a launch, one dependent load
// phase and a few rows walked in turn on a few SMs (12 us FP64 at 64^2, 6 us FP32 at 100^2), with
// most of the chip idle.  Here a CTA owns a small tile, loads it with a margin of two cells per step
// and advances it `steps` steps in shared memory: the valid region shrinks by the stencil radius at
// every side and step, and the tile is what is left (cells of the margin are computed by several
// CTAs; no CTA waits for another).  The flux is the one of gks_cart2d_tau0.cu.  Per step:
//   ghosts  cells beyond a non-reflecting or PEC side (two layers) take their images anew;
//   sides   every cell's values toward its four faces;
//   faces   the left and lower face of every cell;
//   update  every cell from its four faces.
// 64^2 FP64: 4.3 us a step (general kernel 57), 100^2 FP32: 2.7 (12.4).
// Steps over a window (the adjoint's recomputed states) take this kernel on the same grids, one step a
// launch over the window's tiles, so that they repeat the bits of whole steps.
// Bound: the latency of these phases (three or four barriers a step), in FP64 the FP64 pipe.  The
// launch rule (plan) weighs the margin's work against the launches saved.
#include <cuda_runtime.h>

#include <algorithm>

#include "gks_flux2.cuh"
#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_rcp.cuh"
#include "gks_shared_limit.h"
#include "gks_tau0_2d.cuh"

namespace gks {
namespace {

template <typename T>
constexpr int NT = sizeof(T) == 4 ? 512 : 256;   // threads per CTA
constexpr int kMaxSteps = kSmallSteps;
constexpr int NF = 22;                // values a cell of the region keeps in shared memory
constexpr int PW = 32;                // the region's side at most: constant strides in shared memory
constexpr int N = PW * PW;

template <typename T>
struct SmallArgs {
  const T *V;
  T *Vout;
  const T *eps, *src;
  int sx0, sx1, sy0, sy1;
  T amp[kMaxSteps];                   // source amplitude of each step
  int nx, ny;
  int64_t pitch, cstride;
  int perx, pery, pec[4];
  AxisK<T> X, Y;
  int *flag;
  int tw, th, steps, tiles_x;         // tile, steps of this launch, tiles along x
  int wx0, wx1, wy0, wy1;             // cells to advance (a window smaller than the grid: one step only)
};

__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// Cell of index i: periodic wrap, PEC mirror image (m = true) or the clamp of the non-reflecting ghost.
__device__ __forceinline__ int image(int i, int n, int periodic, int pec_lo, int pec_hi, bool &m) {
  m = false;
  if (periodic) {
    i %= n;
    return i < 0 ? i + n : i;
  }
  if (i < 0) {
    if (!pec_lo) return 0;
    m = true;
    return min(-1 - i, n - 1);
  }
  if (i >= n) {
    if (!pec_hi) return n - 1;
    m = true;
    return max(2 * n - 1 - i, 0);
  }
  return i;
}

template <typename T, bool LIMIT>
__global__ void __launch_bounds__(NT<T>) cart2d_small_kernel(const __grid_constant__ SmallArgs<T> p) {
  extern __shared__ __align__(16) unsigned char raw[];
  grid_wait();
  grid_trigger();
  const int S = p.steps, RW = p.tw + 4 * S, RH = p.th + 4 * S;
  T *sm = reinterpret_cast<T *>(raw);
  T *fe = sm, *fa = sm + N, *fb = sm + 2 * N;         // Ez, Hx, Hy
  T *ep = sm + 3 * N, *rx = sm + 4 * N, *ry = sm + 5 * N, *ri = sm + 6 * N;   // eps; 1/(eps sums), 1/eps
  T *lx = sm + 7 * N, *hx = sm + 10 * N;              // x: sides toward the low / high face (P, QE, QH)
  T *ly = sm + 13 * N, *hy = sm + 16 * N;             // y
  T *gx = sm + 19 * N, *gy = sm + 21 * N;             // left face: GE, GH; lower face: GE (GH over ly)
  const int X0 = p.wx0 + (blockIdx.x % p.tiles_x) * p.tw - 2 * S;
  const int Y0 = p.wy0 + (blockIdx.x / p.tiles_x) * p.th - 2 * S;
  const bool nxl = !p.perx && !p.pec[0], nxh = !p.perx && !p.pec[1];
  const bool nyl = !p.pery && !p.pec[2], nyh = !p.pery && !p.pec[3];
  const int tid = threadIdx.x;
  auto cell = [&](int x, int y, bool &xm, bool &ym) {
    return (int64_t)image(y, p.ny, p.pery, p.pec[2], p.pec[3], ym) * p.pitch +
           image(x, p.nx, p.perx, p.pec[0], p.pec[1], xm);
  };
  auto outside = [&](int x, int y) {                  // beyond a side that is not periodic
    return (!p.perx && (x < 0 || x >= p.nx)) || (!p.pery && (y < 0 || y >= p.ny));
  };
  // for every cell of the region at least m cells inside it (and e more at the high sides)
  auto each = [&](int m, int e, auto &&body) {
    const unsigned w = RW - 2 * m - e, n = w * (RH - 2 * m - e);
    const unsigned M = ((1u << 20) + w - 1) / w;      // i / w as a product: exact for i w < 2^20
    for (unsigned i = tid; i < n; i += NT<T>) {
      const int r = (int)((i * M) >> 20), q = (int)(i - r * w);
      body((m + r) * PW + m + q, X0 + m + q, Y0 + m + r);
    }
  };
  each(0, 0, [&](int i, int x, int y) {
    bool xm, ym;
    const int64_t o = cell(x, y, xm, ym);
    const T e = p.V[o], a = p.V[p.cstride + o], b = p.V[2 * p.cstride + o];
    fe[i] = xm != ym ? -e : e;
    fa[i] = xm ? -a : a;
    fb[i] = ym ? -b : b;
    ep[i] = p.eps[o];
  });
  __syncthreads();
  each(1, 0, [&](int i, int, int) {
    rx[i] = rcp_normal(ep[i - 1] + ep[i]);
    ry[i] = rcp_normal(ep[i - PW] + ep[i]);
    ri[i] = rcp_normal(ep[i]);
  });
  const bool wall = outside(X0, Y0) || outside(X0 + RW - 1, Y0 + RH - 1);   // uniform over the CTA
  for (int s = 0; s < S; ++s) {
    if (wall && s > 0) {
      each(2 * s, 0, [&](int i, int x, int y) {
        if (!outside(x, y) || (!p.perx && (x < -2 || x > p.nx + 1)) ||
            (!p.pery && (y < -2 || y > p.ny + 1)))
          return;
        bool xm = false, ym = false;
        const int cx = p.perx ? x : image(x, p.nx, 0, p.pec[0], p.pec[1], xm);
        const int cy = p.pery ? y : image(y, p.ny, 0, p.pec[2], p.pec[3], ym);
        const int j = (cy - Y0) * PW + cx - X0;
        if (cx < X0 || cx >= X0 + RW || cy < Y0 || cy >= Y0 + RH) return;
        const T e = fe[j], a = fa[j], b = fb[j];
        fe[i] = xm != ym ? -e : e;
        fa[i] = xm ? -a : a;
        fb[i] = ym ? -b : b;
      });
      __syncthreads();
    }
    each(2 * s + 1, 0, [&](int i, int x, int y) {
      const T e = fe[i], a = fa[i], b = fb[i], k = ep[i];
      const T ex = raw_slope<LIMIT>(fe[i - 1], e, fe[i + 1]), ey = raw_slope<LIMIT>(fe[i - PW], e, fe[i + PW]);
      const T bx = raw_slope<LIMIT>(fb[i - 1], b, fb[i + 1]), ay = raw_slope<LIMIT>(fa[i - PW], a, fa[i + PW]);
      const T ue = k * e, ux = k * ex, uy = k * ey;
      const bool gxz = (nxl && x < 0) || (nxh && x >= p.nx), gyz = (nyl && y < 0) || (nyh && y >= p.ny);
      auto sides = [&](const AxisK<T> &K, T bb, T en, T bn, T un, T at, bool zero, T *lo, T *hi) {
        const T ev = mad(K.mq, en, bb), od = mad(K.m4, e, bn);
        const T eq = mad(K.ka, at, mad(K.c0, bn, ue)), oq = mad(K.l4, en, mad(K.m4, bb, un));
        hi[i] = zero ? T(0) : mad(T(0.25), od, ev);
        lo[i] = zero ? T(0) : mad(T(-0.25), od, ev);
        hi[i + N] = zero ? T(0) : mad(-K.ic, bn, un);
        lo[i + N] = zero ? T(0) : mad(K.ic, bn, un);
        hi[i + 2 * N] = zero ? T(0) : mad(T(0.25), oq, eq);
        lo[i + 2 * N] = zero ? T(0) : mad(T(-0.25), oq, eq);
      };
      sides(p.X, b, ex, bx, ux, ay, gxz, lx, hx);
      sides(p.Y, a, ey, ay, uy, bx, gyz, ly, hy);
    });
    __syncthreads();
    // faces left of and below a cell; GH of y goes over ly's P, which only this thread reads
    each(2 * s + 2, -1, [&](int i, int, int) {
      const T a = rx[i], b = ry[i];
      const int j = i - 1, k = i - PW;
      const T gex = mad(p.X.kE * a, hx[j + N] + lx[i + N], hx[j] + lx[i]);
      const T ghx = a * (hx[j + 2 * N] + lx[i + 2 * N]);
      const T gey = mad(p.Y.kE * b, hy[k + N] + ly[i + N], hy[k] + ly[i]);
      const T ghy = b * (hy[k + 2 * N] + ly[i + 2 * N]);
      gx[i] = gex;
      gx[i + N] = ghx;
      gy[i] = gey;
      ly[i] = ghy;
    });
    __syncthreads();
    each(2 * s + 2, 0, [&](int i, int x, int y) {
      if (outside(x, y)) return;
      T dE = mad(p.X.sE, gx[i] - gx[i + 1], p.Y.sE * (gy[i] - gy[i + PW]));
      if (p.src) {
        bool m;
        const int cx = image(x, p.nx, p.perx, 0, 0, m), cy = image(y, p.ny, p.pery, 0, 0, m);
        if (cx >= p.sx0 && cx < p.sx1 && cy >= p.sy0 && cy < p.sy1)
          dE -= p.amp[s] * p.src[(int64_t)cy * p.pitch + cx];
      }
      fe[i] = mad(dE, ri[i], fe[i]);
      fa[i] = mad(p.Y.sH, ly[i] - ly[i + PW], fa[i]);
      fb[i] = mad(p.X.sH, gx[i + N] - gx[i + 1 + N], fb[i]);
    });
    __syncthreads();
  }
  bool bad = false;
  each(2 * S, 0, [&](int i, int x, int y) {
    if (x >= p.wx1 || y >= p.wy1) return;
    const int64_t o = (int64_t)y * p.pitch + x;
    p.Vout[o] = fe[i];
    p.Vout[p.cstride + o] = fa[i];
    p.Vout[2 * p.cstride + o] = fb[i];
    bad |= !(isfinite(fe[i]) && isfinite(fa[i]) && isfinite(fb[i]));
  });
  if (__any_sync(0xffffffffu, bad) && (tid & 31) == 0) atomicOr(p.flag, 1);
}

int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 1;
  }
  return sms;
}

// Tile and steps per launch with the least estimated time per step: a launch with its loads, the
// phases' latency per step, and the work of the shrinking region on one SM; at most per_sm CTAs an SM.
SmallPlan plan(int nx, int ny, bool fp64, int most, int per_sm = 1) {
  const double launch = 2.2, phase = fp64 ? 1.2 : 1.0, cell = fp64 ? 0.0120 : 0.0020;   // us
  const int sms = sm_count();
  SmallPlan best;
  static const int sizes[] = {4, 6, 8, 10, 12, 16, 20, 24};
  for (int tw : sizes)
    for (int th : sizes) {
      if (th > tw || tw > 3 * th) continue;
      const int64_t ctas = (int64_t)((nx + tw - 1) / tw) * ((ny + th - 1) / th);
      if (ctas > (int64_t)sms * per_sm) continue;
      double work = 0.0;
      for (int S = 1; S <= std::min(most, kMaxSteps); ++S) {
        if (tw + 4 * S > PW || th + 4 * S > PW) break;
        work += (double)(tw + 4 * S - 2) * (th + 4 * S - 2) * cell;
        const double us = (launch + S * phase + work) / S;
        if (us < best.us) {
          best.tw = tw; best.th = th; best.steps = S; best.us = us;
        }
      }
    }
  return best;
}

template <typename T>
cudaError_t launch_t(const CartGeom &g, const CartStepArgs &a, const SmallPlan &pl, const double *amp,
                     cudaStream_t st) {
  SmallArgs<T> p;
  p.V = static_cast<const T *>(a.V);
  p.Vout = static_cast<T *>(a.Vout);
  p.eps = static_cast<const T *>(a.eps);
  p.src = static_cast<const T *>(a.src);
  p.sx0 = a.src_box[0]; p.sx1 = a.src_box[1];
  p.sy0 = a.src_box[2]; p.sy1 = a.src_box[3];
  for (int s = 0; s < pl.steps; ++s) p.amp[s] = T(amp[s]);
  p.nx = g.nx; p.ny = g.ny;
  p.pitch = g.pitch; p.cstride = g.cstride;
  p.perx = g.periodic[0]; p.pery = g.periodic[1];
  for (int k = 0; k < 4; ++k) p.pec[k] = g.pec[k];
  p.X = make_axis<T>(a.C, a.c, g.h[0], g.h[1], 1.0);
  p.Y = make_axis<T>(a.C, a.c, g.h[1], g.h[0], -1.0);
  p.flag = a.flag;
  p.tw = pl.tw; p.th = pl.th; p.steps = pl.steps;
  p.wx0 = a.window[0]; p.wx1 = a.window[1]; p.wy0 = a.window[2]; p.wy1 = a.window[3];
  p.tiles_x = (p.wx1 - p.wx0 + pl.tw - 1) / pl.tw;
  const int grid = p.tiles_x * ((p.wy1 - p.wy0 + pl.th - 1) / pl.th);
  constexpr int smem = N * NF * (int)sizeof(T);
  auto kern = a.limiter ? cart2d_small_kernel<T, true> : cart2d_small_kernel<T, false>;
  static SharedLimit limit;
  const cudaError_t e = limit.raise(smem, cart2d_small_kernel<T, true>, cart2d_small_kernel<T, false>);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, grid, NT<T>, smem, st, p);
}

}  // namespace

SmallPlan cart2d_small_plan(const CartGeom &g, bool fp64, int most) {
  SmallPlan pl = plan(g.nx, g.ny, fp64, most);
  const double march = fp64 ? 12.0 : 6.0;             // the marching kernels' step on such a grid
  if (!(pl.us < march)) pl.steps = 0;
  return pl;
}

SmallPlan cart2d_small_step_plan(const int win[4], bool fp64) {
  const int nx = win[1] - win[0], ny = win[3] - win[2];
  const SmallPlan pl = plan(nx, ny, fp64, 1);
  // FP32 tiles whose region takes the threads more than one pass: two smaller ones an SM are faster (shared
  // memory has room for both; 250^2 4.4 us against 5.2, 169^2, one pass, 4.0 against 3.7)
  return !fp64 && (pl.tw + 4) * (pl.th + 4) > NT<float> ? plan(nx, ny, fp64, 1, 2) : pl;
}

cudaError_t launch_cart2d_small(const CartGeom &g, const CartStepArgs &a, const SmallPlan &pl,
                                const double *amp, bool fp64, cudaStream_t st) {
  return fp64 ? launch_t<double>(g, a, pl, amp, st) : launch_t<float>(g, a, pl, amp, st);
}

}  // namespace gks
