// 3-D divergence-cleaning step (Sec. 2.1, V = (E, H, phi, psi), mu = 1) for tau = 0: the two-term flux by
// sides, any boundary kind, van Leer slopes optional, FP32 and FP64.
//
// With C2 = C4 = C5 = 0 a cell sends 12 values through each of its faces (Maxwell: 6, gks_pair3.cuh): per
// pair (E_e, H_h), S = +-1, the P, QE, QH of the Maxwell form with the cleaning terms added, and for the
// potentials and the normal components (chi_n, gamma_n: chi/c, gamma/c; lam = C3/(2 h_n C1); primes mark
// derivatives scaled to the normal's raw differences; upper signs the high face)
//   F_En  = C1 chi/(2 h) [(phi + chi_c En'/4) +- (phi' + 4 chi_c En)/4
//           + 2 lam chi r (eps div E' +- (chi phi' + curl_n H')/c)]
//   F_phi = C1 chi/h r [(eps En + (chi_c/4 - lam chi) phi' + lam curl_n H')
//           +- (eps En' + 4 chi_c phi - 4 lam/c (chi^2 En' - div_t E'))/4]
//   F_Hn  = C1 gam/(2 h) [(psi + gam_c Hn'/4 - lam gam div H') +- (psi' + 4 gam_c Hn
//           - 4 lam/c (gam^2 psi' - gam curl_n E'))/4]
//   F_psi = C1 gam/(2 h) [(Hn + (gam_c/4 - lam gam) psi') +- (Hn' (1 - 4 lam gam^2/c) + 4 gam_c psi)/4
//           + 2 lam r (-eps curl_n E' +- div_t H'/c)]
// as sums over the face's two sides (checked against the oracle's faces to 5e-16 in numpy).
//
// The march is 2.5-D, a thread per column of a 32 x BY tile (its outer ring computes sides only).  A
// plane: differences from the staged plane (x, y) and registers (z); sides; the z-face below completes the
// plane below; x by shuffles; y-sides and y-fluxes through shared memory, two barriers a plane.  Planes
// arrive by asynchronous copies one plane ahead (loaded through registers they stalled the march: 227 us a
// step).  About 850 warp instructions a plane, 444 of them arithmetic, where the general kernel, which
// exchanges gradients and rebuilds both sides of every face, issues 1865 a cell.
// 150 x 139 x 128 FP32: 126 us a step (general kernel: 277).  Bound: instruction issue, 72% busy with 12
// warps an SM (41% before the copies); BY = 14 and 16 spill below 150 registers (190, 198 us), BY = 10
// carries a larger ring (147 us).  FP64 takes BY = 8 for its 255 registers, and spills 304 bytes all the same.
#include <cuda_runtime.h>

#include <type_traits>

#include "gks_flux2.cuh"
#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_rcp.cuh"
#include "gks_shared_limit.h"

namespace gks {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int BX = 32, PX = BX + 2;
template <typename T>
constexpr int kBY = sizeof(T) == 4 ? 12 : 8;
enum { PH = 6, PS = 7 };

template <typename T>
struct AxK {                            // one axis: [0] direction n+1, [1] direction n+2
  T lam, l4, kap[2], lk[2], c1[2], c2[2], c3[2], c4[2], c5[2], c6[2];
  T sE, sH, kE;                         // C1/(2h), C1/h, 2 lam
  T f1, f2, h1, h2, h3, s1, s2;         // phi, Hn, psi (see sides8)
  T sEn, kEn, sPhi, sHn, kPs;           // their scales
};

template <typename T>
struct Args {
  const T *V;
  T *Vout;
  const T *eps, *src;
  int sb[6];
  T amp;
  int n[3], per[3], pec[6];
  int64_t pitch, plane, cstride;
  T ic, ic4, qic, chi, chic4, chiq, gam, gamc4, gamq;   // 1/c and its multiples with chi, gamma
  AxK<T> k[3];
  int zchunk;
  int *flag;
};

template <typename T>
struct Smem {
  T V[3][9][kBY<T> + 2][PX];            // staged planes (state, eps) with a ring around the threads
  T Y[13][kBY<T>][BX];                  // sides toward the next row, and eps
  T F[8][kBY<T>][BX];                   // flux through the face below each row (written after the
                                        // first barrier of a plane, read after the second)
};

__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// Sides of a cell along axis A toward its high (l) and low (r) face: per pair P, Q, H; En: P, Q; phi; Hn;
// psi: P, Q.
template <int A, typename T>
__device__ __forceinline__ void sides8(const T v[8], const T ue[3], const T d[3][8], const T ed[3][3],
                                       const Args<T> &a, T l[12], T r[12]) {
  constexpr int D[2] = {(A + 1) % 3, (A + 2) % 3};
  const AxK<T> &k = a.k[A];
  const T q4 = T(0.25);
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    constexpr T one = T(1);
    const T S = p == 0 ? one : -one;
    const int e = D[p], h = D[1 - p];   // E_e and H_h; kap[p] belongs to e, kap[1-p] to h
    const T H = v[3 + h], E = v[e], ne = d[A][e], nH = d[A][3 + h], une = ed[A][e];
    const T hs = d[h][PS], hn = d[h][3 + A], ef = d[e][PH], en = d[e][A];
    const T ev = mad(-k.c1[1 - p], hs, mad(S * a.qic, ne, H));
    const T od = mad(-k.c2[1 - p], hn, mad(S * a.ic4, E, nH));
    l[3 * p] = mad(q4, od, ev);
    r[3 * p] = mad(-q4, od, ev);
    const T x = mad(-k.kap[p], ed[e][A], une), y = mad(-k.c3[p], ef, S * nH);
    l[3 * p + 1] = mad(a.ic, y, x);
    r[3 * p + 1] = mad(-a.ic, y, x);
    const T eq = mad(-k.c4[p], ef, mad(S * k.lk[1 - p], hn, mad(S * (a.qic - k.lam), nH, ue[e])));
    const T oq = mad(S * k.c6[1 - p], hs,
                     mad(-k.c5[p], en, mad(-k.l4, ne, mad(S * a.ic4, H, une))));
    l[3 * p + 2] = mad(q4, oq, eq);
    r[3 * p + 2] = mad(-q4, oq, eq);
  }
  constexpr int P = D[0], Q = D[1];
  const T nE = d[A][A], nF = d[A][PH], nH = d[A][3 + A], nS = d[A][PS];
  const T curlH = mad(k.kap[0], d[P][3 + Q], -(k.kap[1] * d[Q][3 + P]));
  const T curlE = mad(k.kap[0], d[P][Q], -(k.kap[1] * d[Q][P]));
  const T ucurlE = mad(k.kap[0], ed[P][Q], -(k.kap[1] * ed[Q][P]));
  const T tE = mad(k.kap[0], d[P][P], k.kap[1] * d[Q][Q]);
  const T tH = mad(k.kap[0], d[P][3 + P], k.kap[1] * d[Q][3 + Q]);
  const T udiv = mad(k.kap[0], ed[P][P], mad(k.kap[1], ed[Q][Q], ed[A][A]));
  {
    const T ev = mad(a.chiq, nE, v[PH]), od = mad(a.chic4, v[A], nF), y = a.ic * mad(a.chi, nF, curlH);
    l[6] = mad(q4, od, ev);
    r[6] = mad(-q4, od, ev);
    l[7] = udiv + y;
    r[7] = udiv - y;
  }
  {
    const T ev = mad(k.lam, curlH, mad(k.f1, nF, ue[A]));
    const T od = mad(k.l4, tE, mad(-k.f2, nE, mad(a.chic4, v[PH], ed[A][A])));
    l[8] = mad(q4, od, ev);
    r[8] = mad(-q4, od, ev);
  }
  {
    const T ev = mad(-k.h1, nH + tH, mad(a.gamq, nH, v[PS]));
    const T od = mad(k.h3, curlE, mad(-k.h2, nS, mad(a.gamc4, v[3 + A], nS)));
    l[9] = mad(q4, od, ev);
    r[9] = mad(-q4, od, ev);
  }
  {
    const T ev = mad(k.s1, nS, v[3 + A]), od = mad(a.gamc4, v[PS], mad(-k.s2, nH, nH));
    l[10] = mad(q4, od, ev);
    r[10] = mad(-q4, od, ev);
    const T y = a.ic * tH;
    l[11] = y - ucurlE;
    r[11] = -y - ucurlE;
  }
}

// Flux of a face of axis A (components E, H, phi, psi), inv = 1/(eps_l + eps_r).
template <int A, typename T>
__device__ __forceinline__ void face8(const T l[12], const T r[12], T inv, const AxK<T> &k, T F[8]) {
  constexpr int P = (A + 1) % 3, Q = (A + 2) % 3;
  const T t = k.kE * inv, u = k.sH * inv;
  F[P] = k.sE * mad(-t, l[1] + r[1], l[0] + r[0]);
  F[3 + Q] = u * (l[2] + r[2]);
  F[Q] = -k.sE * mad(t, l[4] + r[4], l[3] + r[3]);
  F[3 + P] = -u * (l[5] + r[5]);
  F[A] = mad(k.kEn * inv, l[7] + r[7], k.sEn * (l[6] + r[6]));
  F[PH] = k.sPhi * inv * (l[8] + r[8]);
  F[3 + A] = k.sHn * (l[9] + r[9]);
  F[PS] = mad(k.kPs * inv, l[11] + r[11], k.sHn * (l[10] + r[10]));
}

// Cell of index i: periodic wrap, PEC mirror image (m = true; clamped beyond the stencil) or the clamp of
// the non-reflecting ghost.
__device__ __forceinline__ int image8(int i, int n, int periodic, int pec_lo, int pec_hi, bool &m) {
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

// One value from global to shared memory, asynchronously; and the wait for all of the thread's copies.
template <typename T>
__device__ __forceinline__ void copy_async(T *dst, const T *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(
                   (unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"(sizeof(T))
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <typename T, bool LIMIT>
__global__ void __launch_bounds__(BX *kBY<T>, 1)
    cart3d_phm_tau0_kernel(const __grid_constant__ Args<T> p) {
  constexpr int BY = kBY<T>, NRING = 2 * PX + 2 * BY;
  extern __shared__ __align__(16) unsigned char raw[];
  Smem<T> &s = *reinterpret_cast<Smem<T> *>(raw);
  grid_wait();
  grid_trigger();
  const int tid = threadIdx.x, tx = tid % BX, ty = tid / BX;
  const int x0 = blockIdx.x * (BX - 2), y0 = blockIdx.y * (BY - 2);
  const int z0 = blockIdx.z * p.zchunk, z1 = min(z0 + p.zchunk, p.n[2]);
  const int x = x0 - 1 + tx, y = y0 - 1 + ty;
  const bool inner = tx >= 1 && tx <= BX - 2 && ty >= 1 && ty <= BY - 2 && x < p.n[0] && y < p.n[1];
  auto beyond = [&](int a, int i) {                   // past a non-reflecting side: no distributions
    return !p.per[a] && ((i < 0 && !p.pec[2 * a]) || (i >= p.n[a] && !p.pec[2 * a + 1]));
  };
  const bool gx = beyond(0, x), gy = beyond(1, y);
  // In-plane offset and mirror flags of the thread's column, and of the ring entry it stages.  No cell of the
  // grid reads columns past the two ghost layers; they are wrapped so that a warp's lanes copy from different
  // addresses.  (Clamped past an open side, or to the far side's cell past a wall, they were one cell, and a
  // warp's copies from one address go one after the other: 32^3 open 18.8 us a step, 100 x 90 x 80 70, where
  // periodic sides took 8.4 and 42.)
  bool mx, my, rmx, rmy;
  auto column = [&](int cx, int cy, bool &ax, bool &ay) {
    return (int64_t)image8(cy, p.n[1], p.per[1], p.pec[2], p.pec[3], ay) * p.pitch +
           image8(cx, p.n[0], p.per[0] | ((unsigned)(cx - p.n[0] - 2) < 64u), p.pec[0], p.pec[1], ax);
  };
  const int64_t own = column(x, y, mx, my);
  const bool ringer = tid < NRING;
  int rpx = 0, rpy = 0;
  if (tid < PX) rpx = tid;
  else if (tid < 2 * PX) { rpy = BY + 1; rpx = tid - PX; }
  else if (ringer) { rpy = 1 + ((tid - 2 * PX) >> 1); rpx = ((tid - 2 * PX) & 1) ? PX - 1 : 0; }
  const int64_t rown = column(x0 - 2 + rpx, y0 - 2 + rpy, rmx, rmy);
  // Plane z into slot q by asynchronous copies: each thread its own entry and, the first NRING, one of the
  // ring; they land while the plane before is worked on.
  auto fetch = [&](int z, int q) {
    bool az;
    const int64_t o = (int64_t)image8(z, p.n[2], p.per[2], p.pec[4], p.pec[5], az) * p.plane;
    const T *g = p.V + (o + own);
#pragma unroll
    for (int c = 0; c < 8; ++c, g += p.cstride) copy_async(&s.V[q][c][ty + 1][tx + 1], g);
    copy_async(&s.V[q][8][ty + 1][tx + 1], p.eps + (o + own));
    if (ringer) {
      g = p.V + (o + rown);
#pragma unroll
      for (int c = 0; c < 8; ++c, g += p.cstride) copy_async(&s.V[q][c][rpy][rpx], g);
    }
  };
  // The mirror image beyond a PEC wall flips E unless normal to the wall, H if normal, phi, not psi.
  const bool any_x = mx | my | rmx | rmy;
  auto mirror = [&](int py, int px, int q, bool ax, bool ay, bool az) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const bool neg = c == PS ? false
                       : c == PH ? (ax != (ay != az))
                                 : (ax && ((c < 3) != (c % 3 == 0))) !=
                                       ((ay && ((c < 3) != (c % 3 == 1))) !=
                                        (az && ((c < 3) != (c % 3 == 2))));
      if (neg) s.V[q][c][py][px] = -s.V[q][c][py][px];
    }
  };
  auto land = [&](int z, int q) {                     // this thread's copies of plane z are in place
    copy_wait();
    const bool az = !p.per[2] && ((z < 0 && p.pec[4]) || (z >= p.n[2] && p.pec[5]));
    if (any_x | az) {
      mirror(ty + 1, tx + 1, q, mx, my, az);
      if (ringer) mirror(rpy, rpx, q, rmx, rmy, az);
    }
  };
  T vm[8], v0[8], vp[8], em, e0, ep;                  // planes z-1, z, z+1
  T zl[12], pend[8];
  bool bad = false;
  int q = 0, q1 = 1, q2 = 2;                          // slots of planes z, z+1, z+2
  auto take = [&](int slot, T v[8]) {
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = s.V[slot][c][ty + 1][tx + 1];
    return s.V[slot][8][ty + 1][tx + 1];
  };
  fetch(z0 - 2, q2);
  fetch(z0 - 1, q);
  land(z0 - 2, q2);
  land(z0 - 1, q);
  em = take(q2, vm);
  e0 = take(q, v0);
  em = e0;
  fetch(z0, q1);
#pragma unroll
  for (int c = 0; c < 8; ++c) pend[c] = T(0);
  __syncthreads();
  // plane z0-1 gives only its sides toward z0; plane z1 only the face below it
#pragma unroll 1
  for (int z = z0 - 1; z <= z1; ++z) {
    const bool full = z >= z0 && z < z1;
    land(z + 1, q1);
    ep = take(q1, vp);
    if (z < z1) fetch(z + 2, q2);
    T d[3][8], ue[3], ed[3][3];
    {
      const int py = ty + 1, px = tx + 1;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        d[0][c] = raw_slope<LIMIT>(s.V[q][c][py][px - 1], v0[c], s.V[q][c][py][px + 1]);
        d[1][c] = raw_slope<LIMIT>(s.V[q][c][py - 1][px], v0[c], s.V[q][c][py + 1][px]);
        d[2][c] = raw_slope<LIMIT>(vm[c], v0[c], vp[c]);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        ue[c] = e0 * v0[c];
#pragma unroll
        for (int a = 0; a < 3; ++a) ed[a][c] = e0 * d[a][c];
      }
    }
    T l[12], r[12], F[8], acc[8];
    // z
    sides8<2>(v0, ue, d, ed, p, l, r);
    if (beyond(2, z)) {
#pragma unroll
      for (int i = 0; i < 12; ++i) l[i] = r[i] = T(0);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = T(0);
    if (z >= z0) {
      face8<2>(zl, r, rcp_normal(em + e0), p.k[2], F);
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] = F[c];
      if (z > z0 && inner) {                          // completes plane z-1 (vm)
        const int64_t o = (int64_t)(z - 1) * p.plane + (int64_t)y * p.pitch + x;
        const T ie = rcp_normal(em);
        T sum = T(0);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const T u = pend[c] - F[c];
          const T w = c < 3 ? mad(u, ie, vm[c]) : vm[c] + u;
          p.Vout[c * p.cstride + o] = w;
          sum += w;
        }
        bad |= !isfinite(sum);
      }
    }
    if (z == z1) break;
#pragma unroll
    for (int i = 0; i < 12; ++i) zl[i] = l[i];
    if (full) {
      // x: the face left of the cell; its right face is the next lane's
      sides8<0>(v0, ue, d, ed, p, l, r);
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        if (gx) l[i] = r[i] = T(0);
        l[i] = __shfl_up_sync(FULL, l[i], 1);
      }
      face8<0>(l, r, rcp_normal(__shfl_up_sync(FULL, e0, 1) + e0), p.k[0], F);
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] += F[c] - __shfl_down_sync(FULL, F[c], 1);
      sides8<1>(v0, ue, d, ed, p, l, r);
      if (gy) {
#pragma unroll
        for (int i = 0; i < 12; ++i) l[i] = r[i] = T(0);
      }
#pragma unroll
      for (int i = 0; i < 12; ++i) s.Y[i][ty][tx] = l[i];
      s.Y[12][ty][tx] = e0;
    }
    __syncthreads();
    if (full) {
      T below[12];
      const int b = ty > 0 ? ty - 1 : 0;
#pragma unroll
      for (int i = 0; i < 12; ++i) below[i] = s.Y[i][b][tx];
      face8<1>(below, r, rcp_normal(s.Y[12][b][tx] + e0), p.k[1], F);
#pragma unroll
      for (int c = 0; c < 8; ++c) s.F[c][ty][tx] = F[c];
    }
    __syncthreads();
    if (full) {
      const int u = ty < BY - 1 ? ty + 1 : ty;
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] += F[c] - s.F[c][u][tx];
      if (p.src && inner && x >= p.sb[0] && x < p.sb[1] && y >= p.sb[2] && y < p.sb[3] && z >= p.sb[4] &&
          z < p.sb[5])
        acc[2] -= p.amp * p.src[(int64_t)z * p.plane + (int64_t)y * p.pitch + x];
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      pend[c] = acc[c];
      vm[c] = v0[c];
      v0[c] = vp[c];
    }
    em = e0;
    e0 = ep;
    const int free = q;
    q = q1;
    q1 = q2;
    q2 = free;
  }
  if (__any_sync(FULL, bad) && (tid & 31) == 0) atomicOr(p.flag, 1);
}

template <typename T>
cudaError_t launch_t(const CartGeom &g, const CartStepArgs &a, double chi, double gam, cudaStream_t st) {
  constexpr int BY = kBY<T>, NTH = BX * BY;
  Args<T> p;
  p.V = static_cast<const T *>(a.V);
  p.Vout = static_cast<T *>(a.Vout);
  p.eps = static_cast<const T *>(a.eps);
  p.src = static_cast<const T *>(a.src);
  p.amp = T(a.src_amp);
  const int n[3] = {g.nx, g.ny, g.nz};
  const double ic = 1.0 / a.c;
  p.ic = T(ic); p.ic4 = T(4 * ic); p.qic = T(0.25 * ic);
  p.chi = T(chi); p.chic4 = T(4 * chi * ic); p.chiq = T(0.25 * chi * ic);
  p.gam = T(gam); p.gamc4 = T(4 * gam * ic); p.gamq = T(0.25 * gam * ic);
  for (int A = 0; A < 3; ++A) {
    p.n[A] = n[A]; p.per[A] = g.periodic[A];
    for (int q = 0; q < 2; ++q) {
      p.pec[2 * A + q] = g.pec[2 * A + q];
      p.sb[2 * A + q] = a.src_box[2 * A + q];
    }
    const double K1 = a.C[0] / g.h[A], lam = a.C[2] / (2.0 * g.h[A] * a.C[0]);
    AxK<T> &k = p.k[A];
    k.lam = T(lam); k.l4 = T(4 * lam * ic);
    for (int q = 0; q < 2; ++q) {
      const double kap = g.h[A] / g.h[(A + 1 + q) % 3];
      k.kap[q] = T(kap); k.lk[q] = T(lam * kap);
      k.c1[q] = T(lam * gam * kap); k.c2[q] = T(4 * lam * gam * gam * ic * kap);
      k.c3[q] = T(chi * kap); k.c4[q] = T(lam * chi * kap);
      k.c5[q] = T(4 * lam * chi * chi * ic * kap); k.c6[q] = T(4 * lam * gam * ic * kap);
    }
    k.sE = T(0.5 * K1); k.sH = T(K1); k.kE = T(2 * lam);
    k.f1 = T(0.25 * chi * ic - lam * chi); k.f2 = T(4 * lam * ic * chi * chi);
    k.h1 = T(lam * gam); k.h2 = T(4 * lam * ic * gam * gam); k.h3 = T(4 * lam * ic * gam);
    k.s1 = T(0.25 * gam * ic - lam * gam); k.s2 = T(4 * lam * gam * gam * ic);
    k.sEn = T(0.5 * K1 * chi); k.kEn = T(-K1 * lam * chi * chi);
    k.sPhi = T(K1 * chi); k.sHn = T(0.5 * K1 * gam); k.kPs = T(K1 * lam * gam);
  }
  p.pitch = g.pitch; p.plane = g.plane; p.cstride = g.cstride;
  p.flag = a.flag;
  constexpr int smem = (int)sizeof(Smem<T>);
  static SharedLimit limit;
  const cudaError_t e = limit.raise(smem, cart3d_phm_tau0_kernel<T, true>, cart3d_phm_tau0_kernel<T, false>);
  if (e != cudaSuccess) return e;
  static int res[2] = {0, 0};
  auto kern = a.limiter ? cart3d_phm_tau0_kernel<T, true> : cart3d_phm_tau0_kernel<T, false>;
  int &resident = res[a.limiter ? 1 : 0];
  if (!resident) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, NTH, smem);
    resident = sms * (per > 0 ? per : 1);
  }
  // z chunks that fill whole waves of resident CTAs best, the two extra planes counted as one and a half
  const int gx = (g.nx + BX - 3) / (BX - 2), gy = (g.ny + BY - 3) / (BY - 2);
  int zchunks = 1;
  double best = -1.0;
  for (int zc = 1; zc <= 64 && zc <= g.nz; ++zc) {
    const int len = (g.nz + zc - 1) / zc, nzc = (g.nz + len - 1) / len;
    const int64_t ctas = (int64_t)gx * gy * nzc;
    const double waves = (double)((ctas + resident - 1) / resident);
    const double eff = (double)ctas / (waves * resident) * (double)g.nz / (double)(nzc * (len + 1.5));
    if (eff > best + 1e-9) { best = eff; zchunks = nzc; }
  }
  p.zchunk = (g.nz + zchunks - 1) / zchunks;
  zchunks = (g.nz + p.zchunk - 1) / p.zchunk;
  return launch_pdl(kern, dim3(gx, gy, zchunks), NTH, smem, st, p);
}

}  // namespace

cudaError_t launch_cart3d_phm_tau0(const CartGeom &g, const CartStepArgs &a, double chi, double gamma,
                                   bool fp64, cudaStream_t st) {
  return fp64 ? launch_t<double>(g, a, chi, gamma, st) : launch_t<float>(g, a, chi, gamma, st);
}

}  // namespace gks
