// Adjoint of the 2-D TM step for tau = 0 and mu = 1 (periodic and non-reflecting sides): the transpose of
// the two-term flux of gks_cart2d_tau0.cu, and the eps-gradient of a step.
//
// Transpose.  With q = lambda_E / eps, a face with cells L and R receives GE = sE (q_R - q_L) and
// GH = sH (lambda_H,R - lambda_H,L); each of its two sides receives (P, Q, H) = (GE, kE r GE, r GH),
// r = 1/(eps_L + eps_R).  With the values of a cell's high (h) and low (l) face along an axis, and
// sums S and differences D = h - l of them, the transposed sides add (b the tangential H, d_* the
// adjoints of the raw differences)
//     Ez += eps SH - ic DP       b += SP - ic DH
//     d_e = -ic/4 SP + l4/4 DH + eps (SQ + DH/4)
//     d_b = DP/4 - ic DQ + c0 SH       d_at = ka SH
// and the difference of a cell is transposed last: +d to the cell above, -d to the cell below.  The
// normal H has no other difference, so four difference adjoints a cell remain of the general six.
// Off the grid lambda is zero and eps the edge cell's: the face formula then is the boundary one.
//
// adjoint_tau0_kernel (FP32) marches rows like cart2d_tau0_kernel: a CTA's rows of 256 columns staged by
// TMA, a warp per strip of 61 columns (64 lanes' columns x0-1 .. x0+62, whose left faces they
// evaluate), row j completed when row j+2 has been read.  Bound by instruction issue, as the step:
// 2048 x 2048 34 us, the general kernel (adjoint_lambda_kernel) 49.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_rcp.cuh"
#include "gks_tau0_2d.cuh"
#include "gks_tma.cuh"

namespace gks {
namespace {

using f2 = float2;
constexpr unsigned FULL = 0xffffffffu;
constexpr int WARPS = 4;
constexpr int W = 61;                   // columns written per warp
constexpr int TW = 256;                 // staged columns
constexpr int NSLOT = 8;
constexpr int LAG = 2;                  // rows the copies wait behind the issuing warp
struct alignas(128) StagedRow { float a[4][TW]; };     // lambda_E, lambda_Hx, lambda_Hy; eps
struct Stage {
  StagedRow row[NSLOT];
  unsigned long long full[NSLOT], empty[NSLOT];
};
constexpr unsigned kRowBytes = 4 * TW * 4;

__device__ __forceinline__ f2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 vadd(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 vsub(f2 a, f2 b) { return __ffma2_rn(b, pk(-1.f, -1.f), a); }
__device__ __forceinline__ f2 vmul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 vmul(float k, f2 b) { return __fmul2_rn(pk(k, k), b); }
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 vfma(float k, f2 b, f2 c) { return __ffma2_rn(pk(k, k), b, c); }
__device__ __forceinline__ f2 vrcp(f2 s) { return pk(rcp_normal(s.x), rcp_normal(s.y)); }

__device__ __forceinline__ void mbar_arrive(unsigned long long *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(b)) : "memory");
}

struct Axis {                           // AxisK with the quarters of the transpose folded in
  float mic, mq, l4q, c0, ka, kE, sE, sH;
};

struct Args {
  float *out;                           // (not __restrict__: gks_pdl.cuh)
  const float *lam;
  const float *eps;
  int nx, ny;
  int64_t pitch, cstride;
  int perx, pery;
  Axis X, Y;
  int *flag;
  int wx0, wx1, wy0, wy1;               // columns and rows to compute
  int ntiles, rows;
};

struct Trip { f2 P, Q, H; };            // what a face gives each of its sides

__device__ __forceinline__ Trip face_bar(f2 dq, f2 dh, f2 esum, const Axis &k) {
  Trip t;
  const f2 inv = vrcp(esum);
  t.P = vmul(k.sE, dq);
  t.Q = vmul(vmul(k.kE, inv), t.P);
  t.H = vmul(inv, vmul(k.sH, dh));
  return t;
}

// Adjoints one axis gives a cell: of Ez (eps SH left to the caller), b, and the differences; SH.
struct CellBar { f2 e, b, de, db, SH; };
__device__ __forceinline__ CellBar cell_bar(const Trip &h, const Trip &l, f2 eps, const Axis &k) {
  const f2 SP = vadd(h.P, l.P), DP = vsub(h.P, l.P), SQ = vadd(h.Q, l.Q), DQ = vsub(h.Q, l.Q);
  const f2 DH = vsub(h.H, l.H);
  CellBar c;
  c.SH = vadd(h.H, l.H);
  c.e = vmul(k.mic, DP);
  c.b = vfma(k.mic, DH, SP);
  c.de = vfma(eps, vfma(0.25f, DH, SQ), vfma(k.l4q, DH, vmul(k.mq, SP)));
  c.db = vfma(k.c0, c.SH, vfma(k.mic, DQ, vmul(0.25f, DP)));
  return c;
}

__global__ void __launch_bounds__(WARPS * 32, 5)
    adjoint_tau0_kernel(const __grid_constant__ CUtensorMap tmL, const __grid_constant__ CUtensorMap tmE,
                        const __grid_constant__ Args p) {
  extern __shared__ __align__(128) unsigned char smem_a[];
  grid_wait();
  grid_trigger();
  Stage &s = *reinterpret_cast<Stage *>(smem_a);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int tile = blockIdx.x % p.ntiles, chunk = blockIdx.x / p.ntiles;
  const int y0 = p.wy0 + chunk * p.rows;
  const int y1 = min(y0 + p.rows, p.wy1);
  const int xt = p.wx0 + tile * nw * W;
  const int xs = (xt - 2) & ~3;
  const int x0 = xt + warp * W;
  const int xend = min(x0 + W, p.wx1);
  const int A = x0 - 1 + lane, B = A + 32;
  const bool stA = lane > 0 && A < xend, stB = lane < 30 && B < xend;

  // ghost columns -2, -1, nx, nx+1 of a staged row: the edge's eps (lambda stays zero there), or the
  // wrapped cell; lane 4 q + f holds array f of ghost column q
  const int gq = (lane >> 2) & 3, gf = lane & 3;
  const int gcol = gq == 0 ? -2 : gq == 1 ? -1 : gq == 2 ? p.nx : p.nx + 1;
  const bool gon = lane < 16 && gcol >= x0 - 2 && gcol <= x0 + 63 && (p.perx || gf == 3);
  const bool xfix = __any_sync(FULL, gon);
  const int gsrc = gq < 2 ? 0 : p.nx - 1;
  const float *gptr = nullptr;
  if (p.perx && gon) {
    int c = gcol % p.nx;
    c = c < 0 ? c + p.nx : c;
    gptr = (gf < 3 ? p.lam + gf * p.cstride : p.eps) + c;
  }
  const int first = y0 - 2, last = y1 + 1;
  auto slot = [first](int r) { return (r - first) & (NSLOT - 1); };
  auto parity = [first](int r) { return (unsigned)(((r - first) / NSLOT) & 1); };
  auto wrap = [&](int r) { return r < 0 ? r + p.ny : (r >= p.ny ? r - p.ny : r); };
  auto eps_row = [&](int r) { return p.pery ? wrap(r) : min(max(r, 0), p.ny - 1); };
  bool ok = true;                                     // false: a bounded wait ran out
  int issued = first - 1;
  auto issue = [&](int r) {
    const int i = slot(r);
    fence_proxy_async();
    mbar_expect_tx(&s.full[i], kRowBytes);
    // rows past a non-reflecting side lie outside the tensor and read as zero
    tma_load_3d(&s.row[i].a[0][0], &tmL, xs, p.pery ? wrap(r) : r, 0, &s.full[i]);
    tma_load_2d(&s.row[i].a[3][0], &tmE, xs, eps_row(r), &s.full[i]);
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
  if (gptr) gval = __ldcg(gptr + (int64_t)eps_row(first) * p.pitch);
  auto wait_row = [&](int r) {                        // after a failure nothing is waited for
    if (ok) ok = mbar_wait(&s.full[slot(r)], parity(r));
  };
  // (a periodic x with a non-reflecting y: rows past the side keep lambda = 0)
  auto fix_row = [&](int r) {
    if (!xfix) return;
    float(&R)[4][TW] = s.row[slot(r)].a;
    if (gon) {
      float v;
      if (gptr) {
        v = gf < 3 && !p.pery && (r < 0 || r >= p.ny) ? 0.f : gval;
        if (r < last) gval = __ldcg(gptr + (int64_t)eps_row(r + 1) * p.pitch);
      } else {
        v = R[3][gsrc - xs];
      }
      R[gf][gcol - xs] = v;
    }
    __syncwarp();
  };
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
  auto from_left = [&](f2 v) {
    const float a = __shfl_sync(FULL, v.x, lprev), b = __shfl_sync(FULL, v.y, lprev);
    return pk(a, lane == 0 ? a : b);
  };
  auto from_right = [&](f2 v) {
    const float a = __shfl_sync(FULL, v.x, lnext), b = __shfl_sync(FULL, v.y, lnext);
    return pk(lane == 31 ? b : a, b);
  };
  const int t0 = A - xs;
  auto get = [&](const StagedRow &R, int f, int d) { return pk(R.a[f][t0 + d], R.a[f][t0 + 32 + d]); };
  // columns whose neighbour lies off a non-reflecting side, and the edge columns (clamped ends)
  const bool edge = !p.perx && __any_sync(FULL, A <= 0 || A + 1 >= p.nx || B + 1 >= p.nx);
  auto dxT = [&](f2 d) {                              // transposed central difference along x
    f2 l = from_left(d), r = from_right(d);
    if (edge) {
      __syncwarp();
      const f2 own = d;
      if (A - 1 < 0) l.x = 0.f;
      if (A + 1 >= p.nx) r.x = 0.f;
      if (B + 1 >= p.nx) r.y = 0.f;
      if (A == 0) l.x -= own.x;                       // (B > 0 always)
      if (A == p.nx - 1) r.x -= own.x;
      if (B == p.nx - 1) r.y -= own.y;
    }
    return vsub(l, r);
  };

  f2 qm, am, epsm;                                    // row r-1: q, lambda_Hx, eps
  Trip yb;                                            // its lower face
  f2 pE = pk(0.f, 0.f), pA = pE, cE = pE, cA = pE;    // row j-1's output so far; its y-differences
  {
    wait_row(first);
    fix_row(first);
    const StagedRow &R = s.row[slot(first)];
    epsm = get(R, 3, 0);
    qm = vmul(get(R, 0, 0), vrcp(epsm));
    am = get(R, 1, 0);
    release(first);
    wait_row(first + 1);
    fix_row(first + 1);
    const StagedRow &R1 = s.row[slot(first + 1)];
    const f2 e1 = get(R1, 3, 0), q1 = vmul(get(R1, 0, 0), vrcp(e1)), a1 = get(R1, 1, 0);
    yb = face_bar(vsub(q1, qm), vsub(a1, am), vadd(epsm, e1), p.Y);
    qm = q1;
    am = a1;
    epsm = e1;
  }
  float *oE = p.out + (int64_t)y0 * p.pitch + A, *oA = oE + p.cstride, *oB = oA + p.cstride;
#pragma unroll 2
  for (int r = y0; r <= y1 + 1; ++r) {                // completes row j = r - 1
    const int j = r - 1;
    wait_row(r);
    fix_row(r);
    const StagedRow &R0 = s.row[slot(j)], &R1 = s.row[slot(r)];
    const f2 e1 = get(R1, 3, 0), q1 = vmul(get(R1, 0, 0), vrcp(e1)), a1 = get(R1, 1, 0);
    const Trip yt = face_bar(vsub(q1, qm), vsub(a1, am), vadd(epsm, e1), p.Y);
    const f2 b0 = get(R0, 2, 0), el = get(R0, 3, -1);
    const f2 ql = vmul(get(R0, 0, -1), vrcp(el));
    const Trip xl = face_bar(vsub(qm, ql), vsub(b0, get(R0, 2, -1)), vadd(el, epsm), p.X);
    Trip xr;
    xr.P = from_right(xl.P);
    xr.Q = from_right(xl.Q);
    xr.H = from_right(xl.H);
    const CellBar x = cell_bar(xr, xl, epsm, p.X), y = cell_bar(yt, yb, epsm, p.Y);
    const f2 dBx = vfma(p.Y.ka, y.SH, x.db), dAy = vfma(p.X.ka, x.SH, y.db);
    const bool in = p.pery || (j >= 0 && j < p.ny);
    const f2 dE = in ? y.de : pk(0.f, 0.f), dA = in ? dAy : pk(0.f, 0.f);
    f2 oe = vadd(vadd(get(R0, 0, 0), vfma(epsm, vadd(x.SH, y.SH), vadd(x.e, y.e))),
                 vadd(dxT(x.de), cE));
    f2 oa = vadd(vadd(am, y.b), cA);
    const f2 ob = vadd(vadd(b0, x.b), dxT(dBx));
    if (!p.pery) {                                    // clamped ends
      if (j == p.ny - 1) { oe = vadd(oe, dE); oa = vadd(oa, dA); }
      if (j == 0) { oe = vsub(oe, dE); oa = vsub(oa, dA); }
    }
    if (j > y0) {                                     // row j-1 is complete
      const f2 fe = vsub(pE, dE), fa = vsub(pA, dA);
      if (stA) { oE[0] = fe.x; oA[0] = fa.x; }
      if (stB) { oE[32] = fe.y; oA[32] = fa.y; }
      oE += p.pitch;
      oA += p.pitch;
    }
    if (j >= y0 && j < y1) {
      if (stA) oB[0] = ob.x;
      if (stB) oB[32] = ob.y;
      oB += p.pitch;
    }
    pE = oe;
    pA = oa;
    cE = dE;
    cA = dA;
    yb = yt;
    qm = q1;
    am = a1;
    epsm = e1;
    release(j);
  }
  if (!__all_sync(FULL, ok)) {
    if (lane == 0) atomicOr(p.flag, 2);
    if (threadIdx.x == 0)                             // copies in flight, each awaited (bounded)
      for (int r = max(first, issued - NSLOT + 1); r <= issued; ++r)
        mbar_wait(&s.full[slot(r)], parity(r));
  }
}

// ------------------------------------------------------------------ probe term and eps-gradient
// Over the box of probe and design cells, after the march (32 x 8 tiles, one thread per cell):
//  * lambda^n += dq/dV^n = 2 dt |Omega| Ez^n on the probe;
//  * dJ/deps_d += -lambda_E (E^{n+1} - E^n)/eps_d + sum over the cell's faces of
//    GE_bar dGE/deps_d + GH_bar dGH/deps_d (lambda = lambda^{n+1}, V = V^n), where eps_d enters a face
//    through r = 1/(eps_l + eps_r) and through the cell's own QE (d = d_n E) and QH (d = E +- d_n E/4).
// lambda^{n+1}, eps and V^n are staged with a two-cell halo.  130 operations a cell; the general flux's
// derivative takes 500.
constexpr int GX = 32, GY = 8, GSX = GX + 4, GSY = GY + 4;

template <typename T>
struct PostArgs {
  const T *lam, *eps, *Vn, *Vn1;
  T *out;
  const int32_t *dslot;
  double *grad;
  const double *pw;
  int px0, px1, py0, py1, dx0, dx1, dy0, dy1, bx0, bx1, by0, by1;
  double dt2;
  int nx, ny, perx, pery;
  int64_t pitch, cstride;
  AxisK<T> X, Y;
};

template <typename T>
struct PostSmem {
  T lam[3][GSY][GSX], eps[GSY][GSX], vn[3][GSY][GSX];
};

// QE and QH of a cell toward its high (S = 1) or low (S = -1) face along x (AX = 0) or y.
template <int AX, int S, typename T>
__device__ __forceinline__ void post_side(const PostSmem<T> &s, int sx, int sy, const AxisK<T> &k,
                                          T &QE, T &QH) {
  constexpr int B = AX == 0 ? 2 : 1, N = AX == 0 ? 1 : 2;   // tangential and normal H
  constexpr int dx = AX == 0, dy = AX == 1;
  const T e = s.vn[0][sy][sx], b = s.vn[B][sy][sx], ep = s.eps[sy][sx];
  const T en = s.vn[0][sy + dy][sx + dx] - s.vn[0][sy - dy][sx - dx];
  const T bn = s.vn[B][sy + dy][sx + dx] - s.vn[B][sy - dy][sx - dx];
  const T at = s.vn[N][sy + dx][sx + dy] - s.vn[N][sy - dx][sx - dy];
  const T un = ep * en;
  QE = un - T(S) * k.ic * bn;
  QH = ep * e + k.c0 * bn + k.ka * at + T(0.25 * S) * (un + k.m4 * b + k.l4 * en);
}

template <typename T>
__global__ void __launch_bounds__(GX * GY) adjoint_post_tau0_kernel(const __grid_constant__ PostArgs<T> p) {
  __shared__ PostSmem<T> s;
  grid_wait();
  grid_trigger();
  const int tid = threadIdx.x, tx = tid % GX, ty = tid / GX;
  const int x0 = p.bx0 + blockIdx.x * GX, y0 = p.by0 + blockIdx.y * GY;
  const int gx = x0 + tx, gy = y0 + ty;
  const bool in = gx < p.bx1 && gy < p.by1;
  const int64_t o = (int64_t)gy * p.pitch + gx;
  if (p.pw && in && gx >= p.px0 && gx < p.px1 && gy >= p.py0 && gy < p.py1) {
    const double w = p.pw[(int64_t)(gy - p.py0) * (p.px1 - p.px0) + (gx - p.px0)];
    p.out[o] += T(p.dt2 * w) * p.Vn[o];
  }
  if (!p.grad) return;                                  // uniform over the launch
  const int slot = in && gx >= p.dx0 && gx < p.dx1 && gy >= p.dy0 && gy < p.dy1 ? p.dslot[o] : -1;
  const T en1 = slot >= 0 ? p.Vn1[o] : T(0);
  const double g_old = slot >= 0 ? p.grad[slot] : 0.0;
  auto idx = [](int i, int n, int per) {
    if (per) {
      i %= n;
      return i < 0 ? i + n : i;
    }
    return min(max(i, 0), n - 1);
  };
#pragma unroll
  for (int i = tid; i < GSX * GSY; i += GX * GY) {
    const int sy = i / GSX, sx = i - sy * GSX;
    const int64_t q = (int64_t)idx(y0 - 2 + sy, p.ny, p.pery) * p.pitch + idx(x0 - 2 + sx, p.nx, p.perx);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      s.lam[c][sy][sx] = p.lam[c * p.cstride + q];
      s.vn[c][sy][sx] = p.Vn[c * p.cstride + q];
    }
    s.eps[sy][sx] = p.eps[q];
  }
  __syncthreads();
  if (slot < 0) return;
  const int sx = tx + 2, sy = ty + 2;
  const T ed = s.eps[sy][sx], e = s.vn[0][sy][sx], ie = rcp_normal(ed), q0 = s.lam[0][sy][sx] * ie;
  T gs = -q0 * (en1 - e);
  // one face: HI the cell's high face (its neighbour's low side); off: the neighbour is off the grid
  auto face = [&](auto axis, auto high, bool off) {
    constexpr int AX = decltype(axis)::value, S = decltype(high)::value ? 1 : -1;
    constexpr int B = AX == 0 ? 2 : 1, dx = AX == 0, dy = AX == 1;
    const AxisK<T> &k = AX == 0 ? p.X : p.Y;
    const int nx_ = sx + S * dx, ny_ = sy + S * dy;
    const T en = s.vn[0][sy + dy][sx + dx] - s.vn[0][sy - dy][sx - dx];
    T QE, QH, nE = T(0), nH = T(0), qn = T(0), bn = T(0);
    post_side<AX, S>(s, sx, sy, k, QE, QH);
    const T epn = off ? ed : s.eps[ny_][nx_];
    if (!off) {
      post_side<AX, -S>(s, nx_, ny_, k, nE, nH);
      qn = s.lam[0][ny_][nx_] * rcp_normal(epn);
      bn = s.lam[B][ny_][nx_];
    }
    const T inv = rcp_normal(ed + epn), di = (off ? T(-2) : T(-1)) * inv * inv;
    // adjoints of GE, GH: scale times (high cell - low cell)
    const T gE = k.sE * (T(S) * (qn - q0)), gH = k.sH * (T(S) * (bn - s.lam[B][sy][sx]));
    gs += gE * k.kE * (di * (QE + nE) + inv * en) +
          gH * (di * (QH + nH) + inv * (e + T(0.25 * S) * en));
  };
  using std::integral_constant;
  face(integral_constant<int, 0>{}, integral_constant<bool, false>{}, !p.perx && gx == 0);
  face(integral_constant<int, 0>{}, integral_constant<bool, true>{}, !p.perx && gx == p.nx - 1);
  face(integral_constant<int, 1>{}, integral_constant<bool, false>{}, !p.pery && gy == 0);
  face(integral_constant<int, 1>{}, integral_constant<bool, true>{}, !p.pery && gy == p.ny - 1);
  p.grad[slot] = g_old + double(gs);
}

template <typename T>
cudaError_t post_t(const CartGeom &g, const AdjointArgs &a, const int b[4], cudaStream_t st) {
  PostArgs<T> p;
  p.lam = static_cast<const T *>(a.lam_in);
  p.out = static_cast<T *>(a.lam_out);
  p.eps = static_cast<const T *>(a.eps);
  p.Vn = static_cast<const T *>(a.Vn);
  p.Vn1 = static_cast<const T *>(a.Vn1);
  p.dslot = a.dslot;
  p.grad = a.grad && a.dbox[1] > a.dbox[0] && a.dbox[3] > a.dbox[2] ? a.grad : nullptr;
  p.pw = a.probe_w;
  p.px0 = a.pbox[0]; p.px1 = a.pbox[1]; p.py0 = a.pbox[2]; p.py1 = a.pbox[3];
  p.dx0 = a.dbox[0]; p.dx1 = a.dbox[1]; p.dy0 = a.dbox[2]; p.dy1 = a.dbox[3];
  p.bx0 = b[0]; p.bx1 = b[1]; p.by0 = b[2]; p.by1 = b[3];
  p.dt2 = 2.0 * a.dt;
  p.nx = g.nx; p.ny = g.ny; p.perx = g.periodic[0]; p.pery = g.periodic[1];
  p.pitch = g.pitch; p.cstride = g.cstride;
  p.X = make_axis<T>(a.C, a.c, g.h[0], g.h[1], 1.0);
  p.Y = make_axis<T>(a.C, a.c, g.h[1], g.h[0], -1.0);
  const dim3 grid((b[1] - b[0] + GX - 1) / GX, (b[3] - b[2] + GY - 1) / GY);
  return launch_pdl(adjoint_post_tau0_kernel<T>, grid, GX * GY, 0, st, p);
}

Axis make_adj_axis(const double C[5], double c, double hn, double ht, double sign) {
  const AxisK<double> k = make_axis<double>(C, c, hn, ht, sign);
  Axis a;
  a.mic = float(k.mic); a.mq = float(k.mq); a.l4q = float(0.25 * k.l4); a.c0 = float(k.c0);
  a.ka = float(k.ka); a.kE = float(k.kE); a.sE = float(k.sE); a.sH = float(k.sH);
  return a;
}

}  // namespace

bool adjoint_tau0_supported(const CartGeom &g, const AdjointArgs &a) {
  if (a.C[1] != 0.0 || a.C[3] != 0.0 || a.C[4] != 0.0 || !(a.C[0] > 0.0) || !a.eps_normal) return false;
  if (g.periodic[1] && g.ny < 2) return false;        // the staged rows wrap by one period
  return aligned(a.lam_in, 16) && tensor_map_encoder() != nullptr;
}

cudaError_t launch_adjoint_post_tau0(const CartGeom &g, const AdjointArgs &a, const int box[4],
                                     bool fp64, cudaStream_t st) {
  return fp64 ? post_t<double>(g, a, box, st) : post_t<float>(g, a, box, st);
}

cudaError_t launch_adjoint_tau0(const CartGeom &g, const AdjointArgs &a, cudaStream_t st) {
  Args p;
  p.lam = static_cast<const float *>(a.lam_in);
  p.out = static_cast<float *>(a.lam_out);
  p.eps = static_cast<const float *>(a.eps);
  p.nx = g.nx; p.ny = g.ny;
  p.pitch = g.pitch; p.cstride = g.cstride;
  p.perx = g.periodic[0]; p.pery = g.periodic[1];
  p.X = make_adj_axis(a.C, a.c, g.h[0], g.h[1], 1.0);
  p.Y = make_adj_axis(a.C, a.c, g.h[1], g.h[0], -1.0);
  p.flag = a.flag;
  p.wx0 = a.window[0]; p.wx1 = a.window[1]; p.wy0 = a.window[2]; p.wy1 = a.window[3];
  constexpr int smem = (int)sizeof(Stage);
  static_assert(smem <= 48 * 1024, "more needs the kernel's limit raised");
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 1;
  }
  // Rows a chunk (which computes two rows more): one wave of five CTAs per SM while that takes 40 rows or
  // fewer, past that about four waves, 24 rows or more.  us a step: 1448 x 1448 one wave (12 rows) 18.8, 8:
  // 21.5, 14: 21.1; 2048 x 2048 one wave (25) 33.9, 24 (1.02 waves) 43.7, 28: 37.7, 14: 35.8; 2900 x 2900 24
  // rows 61.5, 16: 62.8, 48: 61.0, 32: 67.6; 4096 x 4096 24 rows 111.0, 16: 113.8, 32: 112.7.
  const int wrows = p.wy1 - p.wy0, strips = (p.wx1 - p.wx0 + W - 1) / W;
  const int nw = std::min(WARPS, strips);
  p.ntiles = (strips + nw - 1) / nw;
  const int64_t resident = (int64_t)sms * 5;
  const int64_t fit = std::max<int64_t>(1, resident / p.ntiles);
  int rows = std::max(4, (int)((wrows + fit - 1) / fit));
  if (rows > 40) {
    const int64_t chunks = std::max<int64_t>(1, 4 * resident / p.ntiles);
    rows = std::max(24, (int)((wrows + chunks - 1) / chunks));
  }
  p.rows = rows;
  const int64_t grid = (int64_t)p.ntiles * ((wrows + rows - 1) / rows);
  CUtensorMap tmL, tmE;
  const cuuint64_t dim[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, 3};
  const cuuint64_t stride[2] = {(cuuint64_t)g.pitch * 4, (cuuint64_t)g.cstride * 4};
  const cuuint32_t box[3] = {TW, 1, 3};
  if (!encode_f32_map(&tmL, p.lam, 3, dim, stride, box) ||
      !encode_f32_map(&tmE, p.eps, 2, dim, stride, box))
    return cudaErrorInvalidValue;
  return launch_pdl(adjoint_tau0_kernel, (unsigned)grid, nw * 32, smem, st, tmL, tmE, p);
}

}  // namespace gks
