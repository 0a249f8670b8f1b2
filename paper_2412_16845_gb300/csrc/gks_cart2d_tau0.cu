// Fused 2-D TM GKS step in the non-viscous limit (tau = 0, Sec. 4.1) with mu = 1.
//
// For tau -> 0 the coefficients C2, C4 and C5 vanish and the time-integrated flux keeps two terms,
// F = C1 <u g0> + C3 <u g_t>.  With mu = 1 it is a sum over the two sides of the face, and the
// flux of the normal H vanishes.  For a face of normal x (b = Hy, ic = 1/c, r = 1/(eps_l + eps_r)):
//     GE = (P_l + P_r) + kE r (QE_l + QE_r),     GH = r (QH_l + QH_r),
//     F_Ez = sE GE,   F_Hy = sH GH,
// where each side's three values depend on that cell alone: its Ez, Hy, eps, the raw central
// differences ex, bx along the normal and ay (of the normal H) along the tangent.  With the
// reconstructions V +- (difference)/4 a cell forms, for its right (l, upper signs) and left face,
//     P  = (Hy - ic ex/4) +- (bx - 4 ic Ez)/4          QE = eps ex -+ ic bx
//     QH = (eps Ez + (k3 - ic/4) bx + ka ay) +- (eps ex - 4 ic Hy - 4 k3 ic ex)/4
// : 13 operations an axis and cell.  The y axis is the same form with Hx for Hy and ic, k3, ka
// negated.  Non-reflecting ghosts have zero sides and the inner cell's eps; PEC ghosts are mirror
// images (Sec. 5.5).
//
// A row is processed once: its sides along both axes, its x-faces, and the y-face to the row
// below, which completes the row below.  What bounds the two kernels:
//  * FP32 (cart2d_tau0_kernel): instruction issue and HBM.  About 54 paired FP32 instructions per
//    two cells; the general flux takes 132.  4096 x 4096: 105.7 us a step where the staged general
//    kernel (gks_cart2d.cu) takes 170.7; 1801 x 1203 with the limiter 23.1 against 36.4.
//  * FP64 (cart2d_tau0_f64_kernel): the FP64 pipe.  A GB300 issues one FP64 warp instruction per
//    64 cycles and scheduler (measured), so the count of FP64 operations, 51 and three reciprocals a
//    cell, and an even spread of rows over the 608 schedulers are the whole time.
//    1531 x 1022: 234 us a step, general kernel 579; the arithmetic alone 174.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "gks_flux2.cuh"
#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_rcp.cuh"
#include "gks_tau0_2d.cuh"
#include "gks_tma.cuh"

namespace gks {
namespace {

using f2 = float2;
constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------------------ values: pairs and doubles
__device__ __forceinline__ f2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 vadd(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 vsub(f2 a, f2 b) { return __ffma2_rn(b, pk(-1.f, -1.f), a); }
__device__ __forceinline__ f2 vmul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 vmul(float k, f2 b) { return __fmul2_rn(pk(k, k), b); }
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 vfma(float k, f2 b, f2 c) { return __ffma2_rn(pk(k, k), b, c); }
__device__ __forceinline__ f2 vrcp(f2 s) { return pk(rcp_normal(s.x), rcp_normal(s.y)); }

// The columns of one lane in FP64: 32 apart.
template <int NC>
struct DV {
  double v[NC];
};
#define GKS_DV(expr)                                  \
  DV<NC> o;                                           \
  _Pragma("unroll") for (int i = 0; i < NC; ++i) o.v[i] = expr; \
  return o
template <int NC> __device__ __forceinline__ DV<NC> vadd(const DV<NC> &a, const DV<NC> &b) { GKS_DV(a.v[i] + b.v[i]); }
template <int NC> __device__ __forceinline__ DV<NC> vsub(const DV<NC> &a, const DV<NC> &b) { GKS_DV(a.v[i] - b.v[i]); }
template <int NC> __device__ __forceinline__ DV<NC> vmul(const DV<NC> &a, const DV<NC> &b) { GKS_DV(a.v[i] * b.v[i]); }
template <int NC> __device__ __forceinline__ DV<NC> vmul(double k, const DV<NC> &b) { GKS_DV(k * b.v[i]); }
template <int NC> __device__ __forceinline__ DV<NC> vfma(const DV<NC> &a, const DV<NC> &b, const DV<NC> &c) { GKS_DV(fma(a.v[i], b.v[i], c.v[i])); }
template <int NC> __device__ __forceinline__ DV<NC> vfma(double k, const DV<NC> &b, const DV<NC> &c) { GKS_DV(fma(k, b.v[i], c.v[i])); }
template <int NC> __device__ __forceinline__ DV<NC> vrcp(const DV<NC> &a) { GKS_DV(rcp_normal(a.v[i])); }
#undef GKS_DV

template <bool LIMIT>
__device__ __forceinline__ f2 vslope(f2 m, f2 c, f2 p) {
  if (!LIMIT) return vsub(p, m);
  return pk(raw_slope<LIMIT>(m.x, c.x, p.x), raw_slope<LIMIT>(m.y, c.y, p.y));
}
template <bool LIMIT, int NC>
__device__ __forceinline__ DV<NC> vslope(const DV<NC> &m, const DV<NC> &c, const DV<NC> &p) {
  DV<NC> o;
#pragma unroll
  for (int i = 0; i < NC; ++i) o.v[i] = raw_slope<LIMIT>(m.v[i], c.v[i], p.v[i]);
  return o;
}
__device__ __forceinline__ void vzero(f2 &a) { a = pk(0.f, 0.f); }
template <int NC>
__device__ __forceinline__ void vzero(DV<NC> &a) {
#pragma unroll
  for (int i = 0; i < NC; ++i) a.v[i] = 0.0;
}

// ------------------------------------------------------------------ the flux
// A cell's three values for one of its faces.
template <typename V>
struct Side {
  V P, QE, QH;
};
template <typename V>
__device__ __forceinline__ void zero_side(Side<V> &s) {
  vzero(s.P);
  vzero(s.QE);
  vzero(s.QH);
}

// The sides of a cell toward its high (l) and its low face (r) along one axis: e = Ez, b the
// tangential H, ue = eps e, en, bn their raw differences along the normal, uen = eps en, at the raw
// tangential difference of the normal H.  P and QH as even and odd parts, P_l,r = Ev +- Od/4.
template <typename V, typename T>
__device__ __forceinline__ void cell_sides(const V &e, const V &b, const V &ue, const V &en,
                                           const V &bn, const V &uen, const V &at,
                                           const AxisK<T> &k, Side<V> &l, Side<V> &r) {
  const V ev = vfma(k.mq, en, b), od = vfma(k.m4, e, bn);
  l.P = vfma(T(0.25), od, ev);
  r.P = vfma(T(-0.25), od, ev);
  l.QE = vfma(k.mic, bn, uen);
  r.QE = vfma(k.ic, bn, uen);
  const V eq = vfma(k.ka, at, vfma(k.c0, bn, ue)), oq = vfma(k.l4, en, vfma(k.m4, b, uen));
  l.QH = vfma(T(0.25), oq, eq);
  r.QH = vfma(T(-0.25), oq, eq);
}

// Face between the sides l and r with r = 1/(eps_l + eps_r).
template <typename V, typename T>
__device__ __forceinline__ void face(const Side<V> &l, const Side<V> &r, const V &inv,
                                     const AxisK<T> &k, V &GE, V &GH) {
  GE = vfma(vmul(k.kE, inv), vadd(l.QE, r.QE), vadd(l.P, r.P));
  GH = vmul(inv, vadd(l.QH, r.QH));
}

// Arguments shared by both kernels.
// (not __restrict__: an early-started kernel must not use the read-only path, gks_pdl.cuh)
template <typename T>
struct Args {
  const T *V;
  T *Vout;
  const T *eps;
  const T *src;
  int sx0, sx1, sy0, sy1;
  T src_amp;
  int nx, ny;
  int64_t pitch, cstride;
  int perx, pery;
  int pec[4];
  AxisK<T> X, Y;
  int *flag;
  int wx0, wx1, wy0, wy1;     // columns and rows to advance
  int ntiles, rows;           // tiles of columns, rows per chunk
};

// Cell of index i on an axis of n cells: periodic wrap, PEC mirror image (m = true; clamped beyond
// the two-cell stencil) or the clamp of the non-reflecting Green-Gauss ghost.
__device__ __forceinline__ int axis_cell(int i, int n, int periodic, int pec_lo, int pec_hi,
                                         bool &m) {
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

// ------------------------------------------------------------------ FP32
// A CTA owns up to four strips of W columns and a chunk of rows; each warp marches one strip.  Lane
// l holds the columns A = x0-1+l and B = x0+31+l as the halves of a float2, so that no pair is
// assembled from two lanes: the column left of A is the previous lane's A, that of B the previous
// lane's B (lane 0's B: lane 31's A).  Each lane evaluates the left faces of A and B with the left
// cell's side taken by shuffle, and takes the right faces from the next lane; lane 0's A and lane
// 31's B are halo columns.
// Rows are staged in shared memory by TMA, one box of 256 columns x (Ez, Hx, Hy) and one of eps for
// the whole CTA (one thread's two copies a row: issued per warp they were a fifth of all
// instructions), into a ring of NSLOT rows with a full and an empty mbarrier each; waits are
// bounded.  Every read is the lane's column plus a constant, so a row needs two addresses.  The
// columns beyond the grid's sides are written into the staged row (fix_row) by the warp that reads
// them.  EDGE: PEC walls or a periodic axis (compiled in only then).
constexpr int WARPS = 4;                // warps per CTA at most
constexpr int W = 62;
constexpr int TW = 256;                 // staged columns: x0-2 rounded down to a multiple of 4, ...
constexpr int NSLOT = 8;
constexpr int LAG = 2;                  // rows the copies wait behind the issuing warp
static_assert((NSLOT & (NSLOT - 1)) == 0, "the ring index masks with NSLOT - 1");
struct alignas(128) StagedRow { float a[4][TW]; };     // Ez, Hx, Hy; eps
struct Stage {
  StagedRow row[NSLOT];
  unsigned long long full[NSLOT], empty[NSLOT];
};
constexpr unsigned kRowBytes = 4 * TW * 4;

__device__ __forceinline__ void mbar_arrive(unsigned long long *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(b)) : "memory");
}

template <bool EDGE, bool LIMIT>
__global__ void __launch_bounds__(WARPS * 32, 6)
    cart2d_tau0_kernel(const __grid_constant__ CUtensorMap tmV,
                       const __grid_constant__ CUtensorMap tmE,
                       const __grid_constant__ Args<float> p) {
  extern __shared__ __align__(128) unsigned char smem_s[];
  grid_wait();
  grid_trigger();
  Stage &s = *reinterpret_cast<Stage *>(smem_s);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int tile = blockIdx.x % p.ntiles, chunk = blockIdx.x / p.ntiles;
  const int y0 = p.wy0 + chunk * p.rows;
  const int y1 = min(y0 + p.rows, p.wy1);
  const int xt = p.wx0 + tile * nw * W;               // the tile's first column
  const int xs = (xt - 2) & ~3;                       // first staged column (16-byte aligned)
  const int x0 = xt + warp * W;
  const int xend = min(x0 + W, p.wx1);
  const int A = x0 - 1 + lane, B = A + 32;
  const bool perx = EDGE && p.perx, pery = EDGE && p.pery;
  const bool pxl = EDGE && p.pec[0], pxh = EDGE && p.pec[1];
  const bool pyl = EDGE && p.pec[2], pyh = EDGE && p.pec[3];
  const bool xlo_nr = !perx && !pxl, xhi_nr = !perx && !pxh;
  const bool ylo_nr = !pery && !pyl, yhi_nr = !pery && !pyh;
  const bool stA = lane > 0 && A < xend, stB = lane < 31 && B < xend;
  // cells beyond a non-reflecting x side carry no distributions
  const bool gA = (xlo_nr && A < 0) || (xhi_nr && A >= p.nx);
  const bool gB = (xlo_nr && B < 0) || (xhi_nr && B >= p.nx);

  // Columns beyond the grid, written into every staged row by the warps that read them: lane
  // 4 q + f holds array f of ghost column q = (-2, -1, nx, nx+1).  A non-reflecting side copies the
  // edge cell, a PEC wall its mirror image (Ez and Hx negated), both from the staged row; a
  // periodic axis the wrapped cell, loaded a row ahead.
  const int gq = (lane >> 2) & 3, gf = lane & 3;
  const int gcol = gq == 0 ? -2 : gq == 1 ? -1 : gq == 2 ? p.nx : p.nx + 1;
  const bool gon = lane < 16 && gcol >= x0 - 2 && gcol <= x0 + W + 1;
  const bool xfix = __any_sync(FULL, gon);
  const bool gmirror = gq < 2 ? pxl : pxh;
  const int gsrc = gmirror ? (gq < 2 ? min(-1 - gcol, p.nx - 1) : max(2 * p.nx - 1 - gcol, 0))
                           : (gq < 2 ? 0 : p.nx - 1);
  const float gsign = gmirror && gf < 2 ? -1.f : 1.f;
  const float *gptr = nullptr;
  if (EDGE && perx && gon) {
    int c = gcol % p.nx;
    c = c < 0 ? c + p.nx : c;
    gptr = (gf < 3 ? p.V + gf * p.cstride : p.eps) + c;
  }

  const int first = y0 - 2, last = y1 + 1;            // staged rows
  auto slot = [first](int r) { return (r - first) & (NSLOT - 1); };
  auto parity = [first](int r) { return (unsigned)(((r - first) / NSLOT) & 1); };
  auto grid_row = [&](int r) {
    if (pery) return r < 0 ? r + p.ny : (r >= p.ny ? r - p.ny : r);
    if (r < 0) return pyl ? min(-1 - r, p.ny - 1) : 0;
    if (r >= p.ny) return pyh ? max(2 * p.ny - 1 - r, 0) : p.ny - 1;
    return r;
  };
  bool ok = true;                                     // false: a bounded wait ran out
  int issued = first - 1;                             // the last row whose copy is issued
  auto issue = [&](int r) {
    const int i = slot(r), gr = grid_row(r);
    fence_proxy_async();
    mbar_expect_tx(&s.full[i], kRowBytes);
    tma_load_3d(&s.row[i].a[0][0], &tmV, xs, gr, 0, &s.full[i]);
    tma_load_2d(&s.row[i].a[3][0], &tmE, xs, gr, &s.full[i]);
    issued = r;
  };
  if (threadIdx.x == 0) {
    for (int i = 0; i < NSLOT; ++i) {
      mbar_init(&s.full[i], 1);
      mbar_init(&s.empty[i], nw);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    for (int r = first; r <= min(last, first + NSLOT - 1); ++r) issue(r);
  }
  __syncthreads();                                    // the barriers are set up
  float gval = 0.f;
  if (EDGE && gptr) gval = __ldcg(gptr + (int64_t)grid_row(first) * p.pitch);

  auto wait_row = [&](int r) {                        // after a failure nothing is waited for
    if (ok) ok = mbar_wait(&s.full[slot(r)], parity(r));
  };
  auto fix_row = [&](int r) {                         // the whole warp, rows in order
    const bool yg = EDGE && ((r < 0 && pyl) || (r >= p.ny && pyh));
    if (!xfix && !yg) return;
    float(&R)[4][TW] = s.row[slot(r)].a;
    // the image of a row past a PEC y wall (-Ez, -Hy) is formed as the warp reads it
    if (gon) {
      float v;
      if (EDGE && gptr) {
        v = gval;
        if (r < last) gval = __ldcg(gptr + (int64_t)grid_row(r + 1) * p.pitch);
      } else {
        v = gsign * R[gf][gsrc - xs];
      }
      R[gf][gcol - xs] = v;
    }
    __syncwarp();
  };
  // row r has been read by this warp; the first warp's lane 0 refills the slot of row r - LAG
  auto release = [&](int r) {
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&s.empty[slot(r)]);
      const int q = r - LAG;
      if (warp == 0 && ok && q >= first && q + NSLOT <= last) {
        ok = mbar_wait(&s.empty[slot(q)], parity(q));
        if (ok) issue(q + NSLOT);
      }
    }
  };

  const int lprev = (lane + 31) & 31, lnext = (lane + 1) & 31;
  // of the left (right) neighbours of A and B; the ends are halo columns and are not used
  auto from_left = [&](f2 v) {
    const float a = __shfl_sync(FULL, v.x, lprev), b = __shfl_sync(FULL, v.y, lprev);
    return pk(a, lane == 0 ? a : b);
  };
  auto from_right = [&](f2 v) {
    const float a = __shfl_sync(FULL, v.x, lnext), b = __shfl_sync(FULL, v.y, lnext);
    return pk(lane == 31 ? b : a, b);
  };
  const int t0 = A - xs;                              // staged column of A; B's is t0 + 32
  // array f of the columns A + d and B + d of a staged row; sy: -1 for the images in a mirror row
  auto get = [&](const StagedRow &R, int f, int d) { return pk(R.a[f][t0 + d], R.a[f][t0 + 32 + d]); };
  auto getE = [&](const StagedRow &R, int f, int d, int r) {
    f2 v = get(R, f, d);
    if constexpr (EDGE) {
      const float sy = (r < 0 && pyl) || (r >= p.ny && pyh) ? -1.f : 1.f;
      v = vmul(sy, v);
    }
    return v;
  };

  f2 em, e0, hm, h0;                                  // Ez, Hx of rows k-1 and k
  f2 epsm, pE, pH;                                    // row k-1: eps, pending dE and new Hx
  Side<f2> yl;                                        // row k-1's side toward row k
  f2 acc = pk(0.f, 0.f);                              // 0 * (updated values): NaN iff one is not finite
  float *oE = p.Vout + (int64_t)y0 * p.pitch + A, *oX = oE + p.cstride, *oY = oX + p.cstride;

  wait_row(first);
  fix_row(first);
  wait_row(y0 - 1);
  fix_row(y0 - 1);
  em = getE(s.row[slot(first)], 0, 0, first);
  hm = get(s.row[slot(first)], 1, 0);
  e0 = getE(s.row[slot(y0 - 1)], 0, 0, y0 - 1);
  h0 = get(s.row[slot(y0 - 1)], 1, 0);
  release(first);

  // row k: PART 0 the row below the chunk (its high y side only), 1 the chunk's first row, 2 its
  // other rows, 3 the row above it (its low y side; completes the last row)
  auto pass = [&](auto part, int k) {
    constexpr int PART = decltype(part)::value;
    wait_row(k + 1);
    fix_row(k + 1);
    const StagedRow &R0 = s.row[slot(k)], &R1 = s.row[slot(k + 1)];
    const f2 ep = getE(R1, 0, 0, k + 1), hp = get(R1, 1, 0);
    const f2 eps = get(R0, 3, 0);
    f2 b0 = pk(0.f, 0.f);
    if (LIMIT || PART == 1 || PART == 2) b0 = getE(R0, 2, 0, k);
    const f2 bx = vslope<LIMIT>(getE(R0, 2, -1, k), b0, getE(R0, 2, 1, k));
    const f2 ey = vslope<LIMIT>(em, e0, ep), ay = vslope<LIMIT>(hm, h0, hp);
    const f2 ue = vmul(eps, e0), uey = vmul(eps, ey);
    f2 aE = pk(0.f, 0.f), nhy = pk(0.f, 0.f);
    if constexpr (PART == 1 || PART == 2) {           // x-faces of the row
      const f2 ex = vslope<LIMIT>(getE(R0, 0, -1, k), e0, getE(R0, 0, 1, k));
      const f2 epsl = get(R0, 3, -1);
      const f2 uex = vmul(eps, ex);
      Side<f2> l, r;
      cell_sides(e0, b0, ue, ex, bx, uex, ay, p.X, l, r);
      if (xfix) {
        __syncwarp();                                 // a branch, not selects in every warp
        if (gA) l.P.x = l.QE.x = l.QH.x = r.P.x = r.QE.x = r.QH.x = 0.f;
        if (gB) l.P.y = l.QE.y = l.QH.y = r.P.y = r.QE.y = r.QH.y = 0.f;
      }
      l.P = from_left(l.P);
      l.QE = from_left(l.QE);
      l.QH = from_left(l.QH);
      f2 GE, GH;
      face(l, r, vrcp(vadd(epsl, eps)), p.X, GE, GH);
      aE = vmul(p.X.sE, vsub(GE, from_right(GE)));
      nhy = vfma(p.X.sH, vsub(GH, from_right(GH)), b0);
      if (p.src && k >= p.sy0 && k < p.sy1) {
        const float *q = p.src + (int64_t)k * p.pitch;
        if (A >= p.sx0 && A < p.sx1) aE.x -= p.src_amp * q[A];
        if (B >= p.sx0 && B < p.sx1) aE.y -= p.src_amp * q[B];
      }
      if (stA) oY[0] = nhy.x;
      if (stB) oY[32] = nhy.y;
      oY += p.pitch;
    }
    Side<f2> yh, r;                                   // toward the rows above and below
    cell_sides(e0, h0, ue, ey, ay, uey, bx, p.Y, yh, r);
    if constexpr (PART > 0) {                         // y-face between rows k-1 and k
      if (PART == 3 && k >= p.ny && yhi_nr) zero_side(r);
      f2 GE, GH;
      face(yl, r, vrcp(vadd(epsm, eps)), p.Y, GE, GH);
      if constexpr (PART > 1) {                       // completes row k-1
        const f2 ne = vfma(vfma(-p.Y.sE, GE, pE), vrcp(epsm), em);
        const f2 nhx = vfma(-p.Y.sH, GH, pH);
        if (stA) {
          oE[0] = ne.x;
          oX[0] = nhx.x;
        }
        if (stB) {
          oE[32] = ne.y;
          oX[32] = nhx.y;
        }
        oE += p.pitch;
        oX += p.pitch;
        acc = vfma(0.f, vadd(vadd(ne, nhx), nhy), acc);
      } else {
        acc = vfma(0.f, nhy, acc);
      }
      pE = vfma(p.Y.sE, GE, aE);
      pH = vfma(p.Y.sH, GH, h0);
    }
    if constexpr (PART < 3) {
      yl = yh;
      if (PART == 0 && k < 0 && ylo_nr) zero_side(yl);
      epsm = eps;
      em = e0; e0 = ep;
      hm = h0; h0 = hp;
    }
    release(k);
  };
  pass(std::integral_constant<int, 0>{}, y0 - 1);
  pass(std::integral_constant<int, 1>{}, y0);
#pragma unroll 2
  for (int k = y0 + 1; k < y1; ++k) pass(std::integral_constant<int, 2>{}, k);
  pass(std::integral_constant<int, 3>{}, y1);
  if (!__all_sync(FULL, ok)) {
    if (lane == 0) atomicOr(p.flag, 2);
    if (threadIdx.x == 0)                             // copies in flight, each awaited (bounded)
      for (int r = max(first, issued - NSLOT + 1); r <= issued; ++r)
        mbar_wait(&s.full[slot(r)], parity(r));
  }
  // columns past the grid hold no finite values: only what was stored counts
  const bool bad = (stA && !isfinite(acc.x)) || (stB && !isfinite(acc.y));
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.flag, 1);
}

// ------------------------------------------------------------------ FP64
// The same march with NC columns per lane (32 apart) and rows loaded straight into registers, two
// ahead of use.  Everything but FP64 arithmetic is free here (64 issue slots pass per FP64
// instruction), so signs of mirror images and the test for non-finite values are integer
// operations, and halo columns and rows are kept few: 2 of 32 NC columns, half a row per chunk.
template <int NC>
struct Row64 {
  DV<NC> e, a, b, ep;
  double ee, be;              // Ez, Hy of the column beyond the warp's (lanes 0 and 31)
};

__device__ __forceinline__ double flip(double v, bool neg) {
  return neg ? __longlong_as_double(__double_as_longlong(v) ^ (1ll << 63)) : v;
}
__device__ __forceinline__ bool not_finite(double v) {
  return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

template <int NC, bool LIMIT>
__global__ void __launch_bounds__(WARPS * 32, 2)
    cart2d_tau0_f64_kernel(const __grid_constant__ Args<double> p) {
  constexpr int WD = 32 * NC - 2;
  grid_wait();
  grid_trigger();
  const int lane = threadIdx.x & 31;
  const int wid = blockIdx.x * WARPS + (threadIdx.x >> 5);
  const int strip = wid % p.ntiles, chunk = wid / p.ntiles;
  const int y0 = p.wy0 + chunk * p.rows;
  if (y0 >= p.wy1) return;                            // whole warp leaves together
  const int y1 = min(y0 + p.rows, p.wy1);
  const int x0 = p.wx0 + strip * WD;
  const int xend = min(x0 + WD, p.wx1);
  const bool xlo_nr = !p.perx && !p.pec[0], xhi_nr = !p.perx && !p.pec[1];
  const bool ylo_nr = !p.pery && !p.pec[2], yhi_nr = !p.pery && !p.pec[3];
  int X[NC], ci[NC], ce;                              // columns, the cells they read, the edge's
  bool xm[NC], em_, ghost[NC], st[NC];
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    X[i] = x0 - 1 + 32 * i + lane;
    ci[i] = axis_cell(X[i], p.nx, p.perx, p.pec[0], p.pec[1], xm[i]);
    ghost[i] = (xlo_nr && X[i] < 0) || (xhi_nr && X[i] >= p.nx);
    st[i] = X[i] >= x0 && X[i] < xend;
  }
  ce = axis_cell(lane == 0 ? x0 - 2 : x0 + WD + 1, p.nx, p.perx, p.pec[0], p.pec[1], em_);
  const bool rim = lane == 0 || lane == 31;

  auto load = [&](int r) {
    Row64<NC> o;
    bool ym;
    const int64_t ro = (int64_t)axis_cell(r, p.ny, p.pery, p.pec[2], p.pec[3], ym) * p.pitch;
    const double *q = p.V + ro, *qe = p.eps + ro;
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      o.e.v[i] = flip(__ldcg(q + ci[i]), xm[i] != ym);
      o.a.v[i] = flip(__ldcg(q + p.cstride + ci[i]), xm[i]);
      o.b.v[i] = flip(__ldcg(q + 2 * p.cstride + ci[i]), ym);
      o.ep.v[i] = __ldcg(qe + ci[i]);
    }
    o.ee = o.be = 0.0;
    if (rim) {
      o.ee = flip(__ldcg(q + ce), em_ != ym);
      o.be = flip(__ldcg(q + 2 * p.cstride + ce), ym);
    }
    return o;
  };
  const int lprev = (lane + 31) & 31, lnext = (lane + 1) & 31;
  // the value of the column to the left (right); `rimv` at the warp's ends
  auto from_left = [&](const DV<NC> &v, double rimv) {
    DV<NC> o;
#pragma unroll
    for (int i = 0; i < NC; ++i) o.v[i] = __shfl_sync(FULL, v.v[i], lprev);
    if (lane == 0) {
#pragma unroll
      for (int i = NC - 1; i > 0; --i) o.v[i] = o.v[i - 1];
      o.v[0] = rimv;
    }
    return o;
  };
  auto from_right = [&](const DV<NC> &v, double rimv) {
    DV<NC> o;
#pragma unroll
    for (int i = 0; i < NC; ++i) o.v[i] = __shfl_sync(FULL, v.v[i], lnext);
    if (lane == 31) {
#pragma unroll
      for (int i = 0; i + 1 < NC; ++i) o.v[i] = o.v[i + 1];
      o.v[NC - 1] = rimv;
    }
    return o;
  };

  DV<NC> em, hm, epsm, pE, pH;
  Row64<NC> c, u, v1, v2;                             // rows k, k+1, and two in flight
  {
    const Row64<NC> d = load(y0 - 2);
    em = d.e;
    hm = d.a;
  }
  c = load(y0 - 1);
  u = load(y0);
  v1 = load(y0 + 1);
  Side<DV<NC>> yl;
  bool bad = false;

  auto pass = [&](auto part, int k) {
    constexpr int PART = decltype(part)::value;
    if constexpr (PART < 2) v2 = load(min(k + 3, y1 + 1));
    const DV<NC> bx = vslope<LIMIT>(from_left(c.b, c.be), c.b, from_right(c.b, c.be));
    const DV<NC> ey = vslope<LIMIT>(em, c.e, u.e), ay = vslope<LIMIT>(hm, c.a, u.a);
    const DV<NC> ue = vmul(c.ep, c.e), uey = vmul(c.ep, ey);
    DV<NC> aE;
    vzero(aE);
    if constexpr (PART == 1) {
      const DV<NC> ex = vslope<LIMIT>(from_left(c.e, c.ee), c.e, from_right(c.e, c.ee));
      const DV<NC> uex = vmul(c.ep, ex);
      Side<DV<NC>> l, r;
      cell_sides(c.e, c.b, ue, ex, bx, uex, ay, p.X, l, r);
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (ghost[i]) l.P.v[i] = l.QE.v[i] = l.QH.v[i] = r.P.v[i] = r.QE.v[i] = r.QH.v[i] = 0.0;
      l.P = from_left(l.P, 0.0);
      l.QE = from_left(l.QE, 0.0);
      l.QH = from_left(l.QH, 0.0);
      DV<NC> GE, GH;
      face(l, r, vrcp(vadd(from_left(c.ep, 1.0), c.ep)), p.X, GE, GH);
      aE = vmul(p.X.sE, vsub(GE, from_right(GE, 0.0)));
      const DV<NC> nb = vfma(p.X.sH, vsub(GH, from_right(GH, 0.0)), c.b);
      const int64_t ro = (int64_t)k * p.pitch;
      if (p.src && k >= p.sy0 && k < p.sy1) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
          if (X[i] >= p.sx0 && X[i] < p.sx1) aE.v[i] -= p.src_amp * p.src[ro + X[i]];
      }
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (st[i]) {
          p.Vout[2 * p.cstride + ro + X[i]] = nb.v[i];
          bad |= not_finite(nb.v[i]);
        }
    }
    Side<DV<NC>> yh, r;
    cell_sides(c.e, c.a, ue, ey, ay, uey, bx, p.Y, yh, r);
    if constexpr (PART > 0) {
      if (k >= p.ny && yhi_nr) zero_side(r);
      DV<NC> GE, GH;
      face(yl, r, vrcp(vadd(epsm, c.ep)), p.Y, GE, GH);
      if (k > y0) {
        const DV<NC> ne = vfma(vfma(-p.Y.sE, GE, pE), vrcp(epsm), em);
        const DV<NC> nh = vfma(-p.Y.sH, GH, pH);
        double *o = p.Vout + (int64_t)(k - 1) * p.pitch;
#pragma unroll
        for (int i = 0; i < NC; ++i)
          if (st[i]) {
            o[X[i]] = ne.v[i];
            o[p.cstride + X[i]] = nh.v[i];
            bad |= not_finite(ne.v[i]) | not_finite(nh.v[i]);
          }
      }
      if constexpr (PART == 1) {
        pE = vfma(p.Y.sE, GE, aE);
        pH = vfma(p.Y.sH, GH, c.a);
      }
    }
    if constexpr (PART < 2) {
      yl = yh;
      if (k < 0 && ylo_nr) zero_side(yl);
      epsm = c.ep;
      em = c.e;
      hm = c.a;
      c = u;
      u = v1;
      v1 = v2;
    }
  };
  pass(std::integral_constant<int, 0>{}, y0 - 1);
#pragma unroll 1
  for (int k = y0; k < y1; ++k) pass(std::integral_constant<int, 1>{}, k);
  pass(std::integral_constant<int, 2>{}, y1);
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.flag, 1);
}

// ------------------------------------------------------------------ launches
template <typename T>
Args<T> make_args(const CartGeom &g, const CartStepArgs &a) {
  Args<T> p;
  p.V = static_cast<const T *>(a.V);
  p.Vout = static_cast<T *>(a.Vout);
  p.eps = static_cast<const T *>(a.eps);
  p.src = static_cast<const T *>(a.src);
  p.sx0 = a.src_box[0]; p.sx1 = a.src_box[1];
  p.sy0 = a.src_box[2]; p.sy1 = a.src_box[3];
  p.src_amp = T(a.src_amp);
  p.nx = g.nx; p.ny = g.ny;
  p.pitch = g.pitch; p.cstride = g.cstride;
  p.perx = g.periodic[0]; p.pery = g.periodic[1];
  for (int k = 0; k < 4; ++k) p.pec[k] = g.pec[k];
  p.X = make_axis<T>(a.C, a.c, g.h[0], g.h[1], 1.0);
  p.Y = make_axis<T>(a.C, a.c, g.h[1], g.h[0], -1.0);
  p.flag = a.flag;
  p.wx0 = a.window[0]; p.wx1 = a.window[1]; p.wy0 = a.window[2]; p.wy1 = a.window[3];
  return p;
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

cudaError_t launch_f32(const CartGeom &g, const CartStepArgs &a, cudaStream_t st) {
  Args<float> p = make_args<float>(g, a);
  using K = void (*)(const CUtensorMap, const CUtensorMap, const Args<float>);
  static const K kern[2][2] = {{cart2d_tau0_kernel<false, false>, cart2d_tau0_kernel<false, true>},
                               {cart2d_tau0_kernel<true, false>, cart2d_tau0_kernel<true, true>}};
  constexpr int smem = (int)sizeof(Stage);
  static_assert(smem <= 48 * 1024, "more needs the kernels' limit raised");
  const int sms = sm_count();
  const int wrows = p.wy1 - p.wy0, strips = (p.wx1 - p.wx0 + W - 1) / W;
  const int nw = std::min(WARPS, strips);
  p.ntiles = (strips + nw - 1) / nw;
  // Rows a chunk: one wave of six CTAs per SM while that takes 24 rows or fewer; past that about eight
  // waves, chunks of 16 rows or more (a chunk's prologue costs about a row and a half).  us a step (open sides,
  // a line source): 1448 x 1448 one wave (10 rows) 16.0, 8: 18.0, 12: 18.4, 16: 23.3; 2048 x 2048 one wave (21)
  // 35.3, 8 to 14 rows 33.0 to 35.4, 16 (1.3 waves) 37.4, 24: 38.7; 2900 x 2900 16 rows 56.4, 10: 55.4, 24:
  // 58.0, 48: 67.8; 4096 x 4096 16 rows 99.5, 12 and 14: 99.1, 8: 102.6, 24: 103.8.
  const int64_t resident = (int64_t)sms * 6;
  const int64_t fit = std::max<int64_t>(1, resident / p.ntiles);
  int rows = std::max(2, (int)((wrows + fit - 1) / fit));
  if (rows > 24) {
    const int64_t chunks = std::max<int64_t>(1, 8 * resident / p.ntiles);
    rows = std::max(16, (int)((wrows + chunks - 1) / chunks));
  }
  p.rows = rows;
  const int64_t grid = (int64_t)p.ntiles * ((wrows + rows - 1) / rows);
  CUtensorMap tmV, tmE;
  const cuuint64_t dim[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, 3};
  const cuuint64_t stride[2] = {(cuuint64_t)g.pitch * 4, (cuuint64_t)g.cstride * 4};
  const cuuint32_t box[3] = {TW, 1, 3};
  if (!encode_f32_map(&tmV, p.V, 3, dim, stride, box) ||
      !encode_f32_map(&tmE, p.eps, 2, dim, stride, box))
    return cudaErrorInvalidValue;
  const bool edge = p.perx || p.pery || p.pec[0] || p.pec[1] || p.pec[2] || p.pec[3];
  return launch_pdl(kern[edge ? 1 : 0][a.limiter ? 1 : 0], (unsigned)grid, nw * 32, smem, st, tmV, tmE, p);
}

cudaError_t launch_f64(const CartGeom &g, const CartStepArgs &a, cudaStream_t st) {
  Args<double> p = make_args<double>(g, a);
  const int wrows = p.wy1 - p.wy0, wcols = p.wx1 - p.wx0;
  // Columns per lane and rows per warp: the least FP64 work on the busiest scheduler, for one to
  // eight warps on each (a CTA puts one warp on each of an SM's four); a chunk of rows costs half a
  // row more, and a single warp per scheduler cannot hide its loads (an eighth).
  const int64_t sched = (int64_t)sm_count() * WARPS;
  double best = 1e300;
  int cols = 1;
  for (int nc = 1; nc <= 2; ++nc) {
    const int strips = (wcols + 32 * nc - 3) / (32 * nc - 2);
    for (int m = 1; m <= 8; ++m) {
      const int64_t chunks = std::max<int64_t>(1, m * sched / strips);
      const int rows = (int)((wrows + chunks - 1) / chunks);
      const int64_t nw = (int64_t)strips * ((wrows + rows - 1) / rows);
      const double cost = (double)((nw + sched - 1) / sched) * nc * (rows + 0.5) *
                          (nw > sched ? 1.0 : 1.125);
      if (cost < best * 0.999) {
        best = cost;
        cols = nc;
        p.ntiles = strips;
        p.rows = rows;
      }
    }
  }
  const int64_t nwarps = (int64_t)p.ntiles * ((wrows + p.rows - 1) / p.rows);
  const int grid = (int)((nwarps + WARPS - 1) / WARPS);
  using K = void (*)(const Args<double>);
  static const K kern[2][2] = {{cart2d_tau0_f64_kernel<1, false>, cart2d_tau0_f64_kernel<1, true>},
                               {cart2d_tau0_f64_kernel<2, false>, cart2d_tau0_f64_kernel<2, true>}};
  return launch_pdl(kern[cols - 1][a.limiter ? 1 : 0], grid, WARPS * 32, 0, st, p);
}

}  // namespace

bool cart2d_tau0_supported(const CartGeom &g, const CartStepArgs &a, bool fp64) {
  // (the reciprocals of eps are those of gks_rcp.cuh)
  if (a.mu || a.C[1] != 0.0 || a.C[3] != 0.0 || a.C[4] != 0.0 || !(a.C[0] > 0.0) || !a.eps_normal)
    return false;
  if (fp64) return true;
  if (g.periodic[1] && g.ny < 2) return false;        // FP32: the staged rows wrap by one period
  return aligned(a.V, 16) && tensor_map_encoder() != nullptr;
}

cudaError_t launch_cart2d_tau0(const CartGeom &g, const CartStepArgs &a, bool fp64,
                               cudaStream_t st) {
  return fp64 ? launch_f64(g, a, st) : launch_f32(g, a, st);
}

}  // namespace gks
