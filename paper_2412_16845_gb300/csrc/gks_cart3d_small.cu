// One 3-D step of a grid too small to fill the GPU (tau = 0, mu = 1; any sides, van Leer slopes optional).
//
// A step of the marching kernels on a 45 x 34 x 27 grid is latency: 108 CTAs each stage four planes and
// then walk a few planes behind two barriers each (8.6 us FP32, 76 FP64; here 7.0 and 35).  Here a CTA takes one small tile: it loads
// the tile and a margin of two cells, computes the sides of its cells along all axes (gks_pair3.cuh), then
// the faces, then adds them to its cells: three barriers in all (with the axes one after the other, six
// phases, a step took 6 us at 16^3).  Margin cells' sides are computed by two CTAs; with one tile per
// SM that work is otherwise idle lanes.  Bound: the latency of the phases.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "gks_flux2.cuh"
#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_pair3.cuh"
#include "gks_rcp.cuh"
#include "gks_shared_limit.h"

namespace gks {
namespace {

// Tiles (constant strides in shared memory: with tile sizes as arguments the address arithmetic was four
// fifths of the instructions) and the layout of one: the region with its margin, and per axis the sides
// of the tile's cells and one more at each end, and their faces.
constexpr int kTiles[][3] = {{8, 8, 8}, {8, 8, 4}, {8, 4, 4}, {4, 4, 4}};
constexpr int kNumTiles = 4;
template <int I>
struct Tile {
  static constexpr int B0 = kTiles[I][0], B1 = kTiles[I][1], B2 = kTiles[I][2];
  static constexpr int R0 = B0 + 4, R1 = B1 + 4, N = R0 * R1 * (B2 + 4);
  static constexpr int S0 = (B0 + 2) * B1 * B2, S1 = B0 * (B1 + 2) * B2, S2 = B0 * B1 * (B2 + 2);
  static constexpr int NS = S0 + S1 + S2;
  static constexpr int G0 = (B0 + 1) * B1 * B2, G1 = B0 * (B1 + 1) * B2, G2 = B0 * B1 * (B2 + 1);
  static constexpr int NG = G0 + G1 + G2;
  static constexpr int words = 7 * N + 12 * NS + 4 * NG;
  // threads: one pass over the sides of small tiles, two or four over the large ones'
  static constexpr int NT = I < 2 ? 512 : (NS + 31) / 32 * 32;
};

template <typename T>
struct OpX {
  static __device__ __forceinline__ float fma(float k, float x, float a) { return fmaf(k, x, a); }
  static __device__ __forceinline__ double fma(double k, double x, double a) { return ::fma(k, x, a); }
  static __device__ __forceinline__ float fmav(float k, float x, float a) { return fmaf(k, x, a); }
  static __device__ __forceinline__ double fmav(double k, double x, double a) { return ::fma(k, x, a); }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ T mulk(T a, T b) { return a * b; }
};

template <typename T>
struct SmallArgs3 {
  const T *V;
  T *Vout;
  const T *eps, *src;
  int sb[6];
  T amp;
  int n[3], per[3], pec[6];
  int64_t pitch, plane, cstride;
  PairK<T> k[3][2];
  int *flag;
  int tiles[2];                       // tiles along x and y
};

// Cell of index i: periodic wrap, PEC mirror image (m = true) or the clamp of the non-reflecting ghost.
__device__ __forceinline__ int image3(int i, int n, int periodic, int pec_lo, int pec_hi, bool &m) {
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

template <typename T, int I, bool LIMIT>
__global__ void __launch_bounds__(Tile<I>::NT)
    cart3d_small_kernel(const __grid_constant__ SmallArgs3<T> p) {
  using L = Tile<I>;
  constexpr int B0 = L::B0, B1 = L::B1, B2 = L::B2, R0 = L::R0, R1 = L::R1, N = L::N;
  constexpr int st[3] = {1, R0, R0 * R1};
  extern __shared__ __align__(16) unsigned char raw[];
  grid_wait();
  grid_trigger();
  T *sm = reinterpret_cast<T *>(raw);
  T *f = sm, *ep = f + 6 * N, *hi = ep + N, *lo = hi + 6 * L::NS, *g = lo + 6 * L::NS;
  const int bx = blockIdx.x % p.tiles[0], by = blockIdx.x / p.tiles[0] % p.tiles[1],
            bz = blockIdx.x / (p.tiles[0] * p.tiles[1]);
  const int O[3] = {bx * B0 - 2, by * B1 - 2, bz * B2 - 2};
  const int tid = threadIdx.x;
  for (int i = tid; i < N; i += L::NT) {
    const int x = i % R0, y = i / R0 % R1, z = i / (R0 * R1);
    bool m[3];
    const int64_t o =
        (int64_t)image3(O[2] + z, p.n[2], p.per[2], p.pec[4], p.pec[5], m[2]) * p.plane +
        (int64_t)image3(O[1] + y, p.n[1], p.per[1], p.pec[2], p.pec[3], m[1]) * p.pitch +
        image3(O[0] + x, p.n[0], p.per[0], p.pec[0], p.pec[1], m[0]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const T v = p.V[c * p.cstride + o];
      const bool e = c < 3;                           // E flips unless normal to the wall, H if normal
      const bool neg = (m[0] && (e != (c % 3 == 0))) != ((m[1] && (e != (c % 3 == 1))) !=
                                                         (m[2] && (e != (c % 3 == 2))));
      f[c * N + i] = neg ? -v : v;
    }
    ep[i] = p.eps[o];
  }
  __syncthreads();
  // side j of axis A: cells of the tile and one more at each end of the axis, x fastest
  auto side = [&](auto which, int j) {
    constexpr int A = decltype(which)::value, P = (A + 1) % 3, Q = (A + 2) % 3;
    constexpr int s = st[A], sp = st[P], sq = st[Q], off = A == 0 ? 0 : A == 1 ? L::S0 : L::S0 + L::S1;
    constexpr int w = B0 + 2 * (A == 0), h = B1 + 2 * (A == 1);
    const int c3[3] = {j % w + 2 - (A == 0), j / w % h + 2 - (A == 1), j / (w * h) + 2 - (A == 2)};
    const int i = (c3[2] * R1 + c3[1]) * R0 + c3[0];
    auto at = [&](int c, int o) { return f[c * N + i + o]; };
    auto diff = [&](int c, int o) { return raw_slope<LIMIT>(at(c, -o), at(c, 0), at(c, o)); };
    const T e = ep[i];
    Sides3<T> l, r;
    const T nP = diff(P, s), nQ = diff(Q, s);
    pair_sides<OpX<T>>(at(P, 0), at(3 + Q, 0), e * at(P, 0), nP, diff(3 + Q, s), e * nP,
                       e * diff(A, sp), diff(3 + A, sq), p.k[A][0], l.v, r.v);
    pair_sides<OpX<T>>(at(Q, 0), at(3 + P, 0), e * at(Q, 0), nQ, diff(3 + P, s), e * nQ,
                       e * diff(A, sq), diff(3 + A, sp), p.k[A][1], l.v + 3, r.v + 3);
    const int c = O[A] + c3[A];
    const bool zero = (c < 0 && !p.per[A] && !p.pec[2 * A]) ||
                      (c >= p.n[A] && !p.per[A] && !p.pec[2 * A + 1]);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      hi[q * L::NS + off + j] = zero ? T(0) : l.v[q];
      lo[q * L::NS + off + j] = zero ? T(0) : r.v[q];
    }
  };
  // face j of axis A, below cell (x, y, z) of the tile (one more at the high end)
  auto face = [&](auto which, int j) {
    constexpr int A = decltype(which)::value;
    constexpr int soff = A == 0 ? 0 : A == 1 ? L::S0 : L::S0 + L::S1;
    constexpr int goff = A == 0 ? 0 : A == 1 ? L::G0 : L::G0 + L::G1;
    constexpr int w = B0 + (A == 0), h = B1 + (A == 1);
    constexpr int sw = B0 + 2 * (A == 0), sh = B1 + 2 * (A == 1);
    constexpr int step = A == 0 ? 1 : A == 1 ? sw : sw * sh;
    const int x = j % w, y = j / w % h, z = j / (w * h);
    const int b = soff + (z * sh + y) * sw + x;       // the side below the face; above: b + step
    const int i = ((z + 2) * R1 + y + 2) * R0 + x + 2;
    Sides3<T> l, r;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      l.v[q] = hi[q * L::NS + b];
      r.v[q] = lo[q * L::NS + b + step];
    }
    T G[4];
    face3<OpX<T>>(l, r, rcp_normal(ep[i - st[A]] + ep[i]), p.k[A], G);
#pragma unroll
    for (int q = 0; q < 4; ++q) g[q * L::NG + goff + j] = G[q];
  };
  using C0 = std::integral_constant<int, 0>;
  using C1 = std::integral_constant<int, 1>;
  using C2 = std::integral_constant<int, 2>;
  for (int j = tid; j < L::NS; j += L::NT) {
    if (j < L::S0) side(C0{}, j);
    else if (j < L::S0 + L::S1) side(C1{}, j - L::S0);
    else side(C2{}, j - L::S0 - L::S1);
  }
  __syncthreads();
  for (int j = tid; j < L::NG; j += L::NT) {
    if (j < L::G0) face(C0{}, j);
    else if (j < L::G0 + L::G1) face(C1{}, j - L::G0);
    else face(C2{}, j - L::G0 - L::G1);
  }
  __syncthreads();
  // the thread's own cell
  const int cx = tid % B0, cy = tid / B0 % B1, cz = tid / (B0 * B1);
  const int gx = O[0] + 2 + cx, gy = O[1] + 2 + cy, gz = O[2] + 2 + cz;
  const bool own = cz < B2 && gx < p.n[0] && gy < p.n[1] && gz < p.n[2];
  const int me = ((cz + 2) * R1 + cy + 2) * R0 + cx + 2;
  T acc[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
  auto gather = [&](auto which) {
    constexpr int A = decltype(which)::value;
    constexpr int goff = A == 0 ? 0 : A == 1 ? L::G0 : L::G0 + L::G1;
    constexpr int w = B0 + (A == 0), h = B1 + (A == 1), step = A == 0 ? 1 : A == 1 ? w : w * h;
    const T *q = g + goff + (cz * h + cy) * w + cx;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      acc[face_comp<A>(k)] += ((k & 1) ? p.k[A][k / 2].sH : p.k[A][k / 2].sE) *
                              (q[k * L::NG] - q[k * L::NG + step]);
  };
  if (own) {
    gather(C0{});
    gather(C1{});
    gather(C2{});
  }
  bool bad = false;
  if (own) {
    const int64_t o = (int64_t)gz * p.plane + (int64_t)gy * p.pitch + gx;
    if (p.src && gx >= p.sb[0] && gx < p.sb[1] && gy >= p.sb[2] && gy < p.sb[3] && gz >= p.sb[4] &&
        gz < p.sb[5])
      acc[2] -= p.amp * p.src[o];
    const T inv = rcp_normal(ep[me]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const T v = c < 3 ? OpX<T>::fma(acc[c], inv, f[c * N + me]) : f[c * N + me] + acc[c];
      p.Vout[c * p.cstride + o] = v;
      bad |= !isfinite(v);
    }
  }
  if (__any_sync(0xffffffffu, bad) && (tid & 31) == 0) atomicOr(p.flag, 1);
}

template <typename T, int I>
cudaError_t launch_t(const CartGeom &g, const CartStepArgs &a, cudaStream_t st) {
  using L = Tile<I>;
  constexpr int smem = L::words * (int)sizeof(T);
  SmallArgs3<T> p;
  p.V = static_cast<const T *>(a.V);
  p.Vout = static_cast<T *>(a.Vout);
  p.eps = static_cast<const T *>(a.eps);
  p.src = static_cast<const T *>(a.src);
  p.amp = T(a.src_amp);
  const int n[3] = {g.nx, g.ny, g.nz};
  for (int d = 0; d < 3; ++d) {
    p.n[d] = n[d]; p.per[d] = g.periodic[d];
    for (int q = 0; q < 2; ++q) {
      p.pec[2 * d + q] = g.pec[2 * d + q];
      p.sb[2 * d + q] = a.src_box[2 * d + q];
      p.k[d][q] = make_pair_k<T>(a.C, g.h, a.c, d, q);
    }
  }
  p.pitch = g.pitch; p.plane = g.plane; p.cstride = g.cstride;
  p.flag = a.flag;
  p.tiles[0] = (g.nx + L::B0 - 1) / L::B0;
  p.tiles[1] = (g.ny + L::B1 - 1) / L::B1;
  const int grid = p.tiles[0] * p.tiles[1] * ((g.nz + L::B2 - 1) / L::B2);
  static SharedLimit limit;
  const cudaError_t e =
      limit.raise(smem, cart3d_small_kernel<T, I, true>, cart3d_small_kernel<T, I, false>);
  if (e != cudaSuccess) return e;
  auto kern = a.limiter ? cart3d_small_kernel<T, I, true> : cart3d_small_kernel<T, I, false>;
  return launch_pdl(kern, grid, L::NT, smem, st, p);
}

}  // namespace

// The tile with the least estimated time, against the kernel that the step would take otherwise: fits to
// steps of 24 grids of 8^3 to 120^3 cells with every tile, open sides, with and without the limiter.  A tile
// costs its sides' work; a second FP32 tile on an SM hides the first one's latency unless shared memory holds
// only one (8 x 8 x 8).  us a step with one, two, four and eight tiles on the busiest SM: FP32 8 x 4 x 4 4.4,
// 6.9, 8.9, 14.9; 8 x 8 x 8 7.6, 13.9, 26.0, 49.8; FP64 8 x 8 x 4 24.5, 46.3, 93.4, 181.  The estimates of the
// tiles taken are within 11%.  Otherwise: FP32 with open or periodic sides the march (8.1 at 32^3, 10.2 at
// 48^3: crossing near 100,000 cells); with the limiter or walls the general kernel (18.8 and 22.9; limited small
// tiles 5.8 and 11.7; crossing near 500,000); FP64 the march (48^3 107, small tiles 70; 130 x 118 x 97 929,
// small tiles 985).
SmallPlan3 cart3d_small_plan(const CartGeom &g, const CartStepArgs &a, bool fp64) {
  SmallPlan3 best;
  const bool lim = a.limiter != 0;
  static int sms = 0;
  if (!sms) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    sms = n > 0 ? n : 1;
  }
  const int words[kNumTiles] = {Tile<0>::words, Tile<1>::words, Tile<2>::words, Tile<3>::words};
  const int sides[kNumTiles] = {Tile<0>::NS, Tile<1>::NS, Tile<2>::NS, Tile<3>::NS};
  for (int i = 0; i < kNumTiles; ++i) {
    if ((int64_t)words[i] * (fp64 ? 8 : 4) > 227 * 1024) continue;
    const int *b = kTiles[i];
    const int64_t ctas = (int64_t)((g.nx + b[0] - 1) / b[0]) * ((g.ny + b[1] - 1) / b[1]) *
                         ((g.nz + b[2] - 1) / b[2]);
    const double per = (double)((ctas + sms - 1) / sms);
    const double us = fp64 ? 3.5 + per * sides[i] * (lim ? 0.0495 : 0.0228)
                           : 2.5 + per * (0.3 + sides[i] * (lim ? 0.0029 : 0.0026)) +
                                 (i == 0 ? 0.9 * (per - 1.0) : 0.0);
    if (us < best.us) {
      best.us = us;
      best.tile = i;
    }
  }
  const double kcells = 1e-3 * g.nx * g.ny * g.nz;
  const double other = fp64                               ? cart3d_tau0_f64_us(g, lim)
                       : cart3d_side_supported(g, a, fp64) ? 8.5 + 0.015 * kcells
                                                           : 15.0 + (lim ? 0.075 : 0.06) * kcells;
  if (!(best.us < other)) best.tile = -1;
  return best;
}

cudaError_t launch_cart3d_small(const CartGeom &g, const CartStepArgs &a, const SmallPlan3 &pl,
                                bool fp64, cudaStream_t st) {
  if (fp64)
    return pl.tile == 1   ? launch_t<double, 1>(g, a, st)
           : pl.tile == 2 ? launch_t<double, 2>(g, a, st)
                          : launch_t<double, 3>(g, a, st);
  return pl.tile == 0   ? launch_t<float, 0>(g, a, st)
         : pl.tile == 1 ? launch_t<float, 1>(g, a, st)
         : pl.tile == 2 ? launch_t<float, 2>(g, a, st)
                        : launch_t<float, 3>(g, a, st);
}

}  // namespace gks
