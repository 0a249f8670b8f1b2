// 3-D GKS step in FP64 for tau = 0 and mu = 1 (the pair flux of gks_pair3.cuh), van Leer slopes
// optional; any boundary kind.
//
// Bound: the FP64 pipe, then latency.  A GB300 issues one FP64 warp instruction per 64 cycles and
// scheduler (measured; one warp with independent instructions fills it), so the least time is the number of
// FP64 operations (162 and four reciprocals a cell; the general kernel runs 763) times how unevenly they are
// spread over the 608 schedulers.  The pipe is 79% busy at 120^3 (the 2-D FP64 march, which loads two rows
// ahead, 83%): a pass uses its loads and shuffles where it issues them, and two warps a scheduler do not hide
// all of it (stalls per issue: wait 7.2, short scoreboard 6.7, long scoreboard 3.9).  Issue slots themselves
// -- index arithmetic, uncoalesced access -- are plenty, 64 per FP64 instruction.
//
// Layout.  Warps are independent.  One warp takes a strip of 30 cells along the lane axis, up to 8
// rows of the row axis and a chunk of planes of the march axis.  It walks the rows of a plane in
// order: the sides toward the next row stay in registers; the sides toward the next plane and the
// pending update of each row wait in shared memory (12 values a cell) for the next plane.  Faces
// along the lane axis come from shuffles.  Work computed twice: 2 of 32 lanes, and about a third of
// a row (plane) per chunk of rows (planes).  The three roles may be any cyclic renaming of x, y, z
// (the flux is the same under it), so the lane axis is the one whose length fills strips best.
// 130 x 118 x 97: 0.93 ms a step, the general kernel 2.59; the arithmetic alone 0.46, with the halo cells
// and the uneven last wave of this split 0.67.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "gks_flux2.cuh"
#include "gks_internal.h"
#include "gks_pair3.cuh"
#include "gks_rcp.cuh"
#include "gks_shared_limit.h"

namespace gks {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int WARPS = 4;              // one per scheduler
constexpr int WL = 30;                // cells advanced along the lane axis
constexpr int MAXR = 8;               // rows per warp
constexpr int NST = 12;               // doubles a cell keeps between planes

struct OpD {
  static __device__ __forceinline__ double fma(double k, double x, double a) { return ::fma(k, x, a); }
  static __device__ __forceinline__ double fmav(double k, double x, double a) { return ::fma(k, x, a); }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double mulk(double a, double b) { return a * b; }
};

// Arguments in role order (0 lane, 1 row, 2 march axis); F[0..2] = E, F[3..5] = H along the roles.
struct Args {
  const double *F[6];
  double *out[6];
  const double *eps, *src;
  int srcc;                           // component the source drives (role index of E_z)
  int sb[6];                          // source box per role
  double src_amp;
  int n[3], per[3], pec[6];
  int64_t s[3];                       // strides of the roles
  PairK<double> k[3][2];
  int strips, nrow, nmarch;           // strips, row chunks, march chunks
  int R, Z;                           // rows per warp, planes per chunk
  int *flag;
};

__device__ __forceinline__ double flip(double v, bool neg) {
  return neg ? __longlong_as_double(__double_as_longlong(v) ^ (1ll << 63)) : v;
}
__device__ __forceinline__ bool not_finite(double v) {
  return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

// Cell of index i on an axis of n cells: periodic wrap, PEC mirror image (m = true; clamped beyond
// the stencil) or the clamp of the non-reflecting Green-Gauss ghost.
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

// A coordinate along one role: its element offset and whether it is a mirror image.
struct At {
  int64_t o;
  bool m;
};

enum { FULLP, ROWLO, ROWHI, MARLO, MARHI };   // what a pass over one row of one plane computes

template <bool LIMIT>
__global__ void __launch_bounds__(WARPS * 32, 2) cart3d_tau0_f64_kernel(const __grid_constant__ Args p) {
  extern __shared__ double sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wid = blockIdx.x * WARPS + warp;
  const int mc = wid / (p.strips * p.nrow), rest = wid - mc * (p.strips * p.nrow);
  const int strip = rest / p.nrow, rc = rest - strip * p.nrow;
  if (mc >= p.nmarch) return;                         // whole warp leaves together
  double *st = sm + (size_t)warp * p.R * NST * 32 + lane;   // st[(row * NST + value) * 32]
  const int x0 = strip * WL, xend = min(x0 + WL, p.n[0]);
  const int j0 = rc * p.R, j1 = min(j0 + p.R, p.n[1]);
  const int k0 = mc * p.Z, k1 = min(k0 + p.Z, p.n[2]);
  const int X = x0 - 1 + lane;
  auto at = [&](int role, int i) {
    At a;
    a.o = axis_cell(i, p.n[role], p.per[role], p.pec[2 * role], p.pec[2 * role + 1], a.m) * p.s[role];
    return a;
  };
  auto ghost = [&](int role, int i) {                 // beyond a non-reflecting side
    return !p.per[role] && ((i < 0 && !p.pec[2 * role]) || (i >= p.n[role] && !p.pec[2 * role + 1]));
  };
  // field c at three coordinates, with the sign of its mirror image (E flips across a wall unless
  // normal to it, H only if normal)
  auto get = [&](int c, const At &a, const At &b, const At &d) {
    const bool e = c < 3;
    const int w = e ? c : c - 3;
    const bool neg = (a.m && (e != (w == 0))) != ((b.m && (e != (w == 1))) != (d.m && (e != (w == 2))));
    return flip(__ldg(p.F[c] + a.o + b.o + d.o), neg);
  };
  const At ax = at(0, X), axe = at(0, lane == 0 ? x0 - 2 : x0 + WL + 1);
  const bool rim = lane == 0 || lane == 31, gx = ghost(0, X), store = X >= x0 && X < xend;
  const int lprev = (lane + 31) & 31, lnext = (lane + 1) & 31;
  bool bad = false;

  // carried from row to row: the previous row's sides toward this one, its eps and pending update
  Sides3<double> yl;
  double epsr = 1.0, accp[6];

  auto pass = [&](auto what, int j, int k) {
    constexpr int WHAT = decltype(what)::value;
    constexpr bool ROW = WHAT == FULLP || WHAT == ROWLO || WHAT == ROWHI;
    constexpr bool MAR = WHAT == FULLP || WHAT == MARLO || WHAT == MARHI;
    const At bj = at(1, j), ck = at(2, k);
    const At bm = at(1, j - 1), bp = at(1, j + 1), cm = at(2, k - 1), cp = at(2, k + 1);
    double v[6], d[3][6], ue[3], ed[3][3];
    const double eps = __ldg(p.eps + ax.o + bj.o + ck.o);
#pragma unroll
    for (int c = 0; c < 6; ++c) v[c] = get(c, ax, bj, ck);
    // raw differences d[a][c], c not along a
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      if (c % 3 != 0) {
        const double e = rim ? get(c, axe, bj, ck) : 0.0;
        const double lo = __shfl_sync(FULL, v[c], lprev), hi = __shfl_sync(FULL, v[c], lnext);
        d[0][c] = raw_slope<LIMIT>(lane == 0 ? e : lo, v[c], lane == 31 ? e : hi);
      }
      if (c % 3 != 1) d[1][c] = raw_slope<LIMIT>(get(c, ax, bm, ck), v[c], get(c, ax, bp, ck));
      if (c % 3 != 2) d[2][c] = raw_slope<LIMIT>(get(c, ax, bj, cm), v[c], get(c, ax, bj, cp));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ue[c] = eps * v[c];
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a != c) ed[a][c] = eps * d[a][c];
    }
    double acc[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) acc[c] = c < 3 ? 0.0 : v[c];
    double G[4];
    if constexpr (WHAT == FULLP) {                    // lane faces
      Sides3<double> l, r;
      cell_sides3<0, OpD>(v, ue, d, ed, p.k[0], l, r);
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        if (gx) l.v[i] = r.v[i] = 0.0;
        l.v[i] = __shfl_sync(FULL, l.v[i], lprev);
      }
      const double inv = rcp_normal(__shfl_sync(FULL, eps, lprev) + eps);
      face3<OpD>(l, r, inv, p.k[0], G);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double df = G[i] - __shfl_sync(FULL, G[i], lnext);
        acc[face_comp<0>(i)] = fma((i & 1) ? p.k[0][i / 2].sH : p.k[0][i / 2].sE, df,
                                   acc[face_comp<0>(i)]);
      }
      if (p.src && store && X >= p.sb[0] && X < p.sb[1] && j >= p.sb[2] && j < p.sb[3] &&
          k >= p.sb[4] && k < p.sb[5]) {
        const double q = p.src_amp * p.src[ax.o + bj.o + ck.o];
#pragma unroll
        for (int c = 0; c < 3; ++c)                    // (acc stays in registers)
          if (c == p.srcc) acc[c] -= q;
      }
    }
    if constexpr (ROW) {
      Sides3<double> l, r;
      cell_sides3<1, OpD>(v, ue, d, ed, p.k[1], l, r);
      if (ghost(1, j)) {
#pragma unroll
        for (int i = 0; i < 6; ++i) l.v[i] = r.v[i] = 0.0;
      }
      if constexpr (WHAT != ROWLO) {                  // face between rows j-1 and j
        face3<OpD>(yl, r, rcp_normal(epsr + eps), p.k[1], G);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double s = (i & 1) ? p.k[1][i / 2].sH : p.k[1][i / 2].sE;
          accp[face_comp<1>(i)] = fma(-s, G[i], accp[face_comp<1>(i)]);
          if (WHAT == FULLP) acc[face_comp<1>(i)] = fma(s, G[i], acc[face_comp<1>(i)]);
        }
        if (j > j0) {
#pragma unroll
          for (int c = 0; c < 6; ++c) st[((j - 1 - j0) * NST + 6 + c) * 32] = accp[c];
        }
      }
      yl = l;
      epsr = eps;
    }
    if constexpr (MAR) {
      double *q = st + (j - j0) * NST * 32;
      Sides3<double> l, r;
      cell_sides3<2, OpD>(v, ue, d, ed, p.k[2], l, r);
      if (ghost(2, k)) {
#pragma unroll
        for (int i = 0; i < 6; ++i) l.v[i] = r.v[i] = 0.0;
      }
      if constexpr (WHAT != MARLO) {                  // face between planes k-1 and k
        Sides3<double> zl;
#pragma unroll
        for (int i = 0; i < 6; ++i) zl.v[i] = q[i * 32];
        const int64_t om = ax.o + bj.o + cm.o;
        const double epsm = __ldg(p.eps + om);
        face3<OpD>(zl, r, rcp_normal(epsm + eps), p.k[2], G);
        if (k > k0) {                                 // completes plane k-1
          double nv[6];
#pragma unroll
          for (int c = 0; c < 6; ++c) nv[c] = q[(6 + c) * 32];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            nv[face_comp<2>(i)] = fma(-((i & 1) ? p.k[2][i / 2].sH : p.k[2][i / 2].sE), G[i],
                                      nv[face_comp<2>(i)]);
          const double ie = rcp_normal(epsm);
#pragma unroll
          for (int c = 0; c < 3; ++c) nv[c] = fma(nv[c], ie, __ldg(p.F[c] + om));
          if (store) {
#pragma unroll
            for (int c = 0; c < 6; ++c) {
              p.out[c][om] = nv[c];
              bad |= not_finite(nv[c]);
            }
          }
        }
        if constexpr (WHAT == FULLP) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            acc[face_comp<2>(i)] = fma((i & 1) ? p.k[2][i / 2].sH : p.k[2][i / 2].sE, G[i],
                                       acc[face_comp<2>(i)]);
        }
      }
      if constexpr (WHAT != MARHI) {
#pragma unroll
        for (int i = 0; i < 6; ++i) q[i * 32] = l.v[i];
      }
    }
    if constexpr (WHAT == FULLP) {
#pragma unroll
      for (int c = 0; c < 6; ++c) accp[c] = acc[c];
    }
  };

  for (int j = j0; j < j1; ++j) pass(std::integral_constant<int, MARLO>{}, j, k0 - 1);
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
#pragma unroll
    for (int c = 0; c < 6; ++c) accp[c] = 0.0;
    pass(std::integral_constant<int, ROWLO>{}, j0 - 1, k);
#pragma unroll 1
    for (int j = j0; j < j1; ++j) pass(std::integral_constant<int, FULLP>{}, j, k);
    pass(std::integral_constant<int, ROWHI>{}, j1, k);
  }
#pragma unroll 1
  for (int j = j0; j < j1; ++j) pass(std::integral_constant<int, MARHI>{}, j, k1);
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(p.flag, 1);
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

// Lane axis, rows per warp and planes per chunk: the least FP64 work on the busiest scheduler for
// one to four warps on each.  A chunk costs about 0.48 of a row (plane) more; one warp alone on a
// scheduler does not hide its loads (an eighth); strided access along the lanes costs a few
// percent.
struct Plan {
  int axis = 0, strips = 0, nrow = 0, nmarch = 0, R = 0, Z = 0;
};

Plan plan_march(const CartGeom &g) {
  const int n[3] = {g.nx, g.ny, g.nz};
  const int64_t sched = (int64_t)sm_count() * WARPS;
  double best = 1e300;
  Plan pl;
  for (int ax = 0; ax < 3; ++ax) {
    const int nl = n[ax], nr = n[(ax + 1) % 3], nm = n[(ax + 2) % 3];
    const int strips = (nl + WL - 1) / WL;
    for (int R0 = 1; R0 <= MAXR; ++R0) {
      const int nrow = (nr + R0 - 1) / R0, R = (nr + nrow - 1) / nrow;
      for (int m = 1; m <= 4; ++m) {
        const int64_t want = std::max<int64_t>(1, m * sched / ((int64_t)strips * nrow));
        const int Z = (int)((nm + want - 1) / want), nmarch = (nm + Z - 1) / Z;
        const int64_t nw = (int64_t)strips * nrow * nmarch;
        const double cost = (double)((nw + sched - 1) / sched) * (R + 0.48) * (Z + 0.48) *
                            (nw > sched ? 1.0 : 1.125) * (ax == 0 ? 1.0 : 1.25);
        if (cost < best * 0.999) {
          best = cost;
          pl.axis = ax; pl.strips = strips; pl.nrow = nrow; pl.nmarch = nmarch; pl.R = R; pl.Z = Z;
        }
      }
    }
  }
  return pl;
}

}  // namespace

// Fits to steps of 24 grids of 32^3 to 120^3 cells, within 10%: a row of a plane takes two warps of a
// scheduler 16.7 us together, a single one 12.1 (loads not hidden); lanes along y or z take 13% more.
double cart3d_tau0_f64_us(const CartGeom &g, bool limited) {
  const Plan pl = plan_march(g);
  const int64_t sched = (int64_t)sm_count() * WARPS;
  const int64_t waves = ((int64_t)pl.strips * pl.nrow * pl.nmarch + sched - 1) / sched;
  const double two = limited ? 30.5 : 16.7, one = limited ? 21.6 : 12.1;
  return (pl.R + 0.48) * (pl.Z + 0.48) * ((double)(waves / 2) * two + (double)(waves % 2) * one) *
         (pl.axis == 0 ? 1.0 : 1.13);
}

bool cart3d_tau0_f64_supported(const CartStepArgs &a) {
  return !a.mu && a.eps_normal && a.C[1] == 0.0 && a.C[3] == 0.0 && a.C[4] == 0.0 && a.C[0] > 0.0;
}

cudaError_t launch_cart3d_tau0_f64(const CartGeom &g, const CartStepArgs &a, cudaStream_t st) {
  static SharedLimit limit;
  const cudaError_t e = limit.raise(WARPS * MAXR * NST * 32 * 8, cart3d_tau0_f64_kernel<false>,
                                    cart3d_tau0_f64_kernel<true>);
  if (e != cudaSuccess) return e;
  Args p;
  const int n[3] = {g.nx, g.ny, g.nz};
  const int64_t stride[3] = {1, g.pitch, g.plane};
  const Plan pl = plan_march(g);
  const int lane_axis = pl.axis;
  p.strips = pl.strips; p.nrow = pl.nrow; p.nmarch = pl.nmarch; p.R = pl.R; p.Z = pl.Z;
  double h[3];
  for (int r = 0; r < 3; ++r) {
    const int ax = (lane_axis + r) % 3;
    for (int f = 0; f < 2; ++f) {
      p.F[3 * f + r] = static_cast<const double *>(a.V) + (3 * f + ax) * g.cstride;
      p.out[3 * f + r] = static_cast<double *>(a.Vout) + (3 * f + ax) * g.cstride;
    }
    p.n[r] = n[ax]; p.per[r] = g.periodic[ax]; p.s[r] = stride[ax];
    p.pec[2 * r] = g.pec[2 * ax]; p.pec[2 * r + 1] = g.pec[2 * ax + 1];
    p.sb[2 * r] = a.src_box[2 * ax]; p.sb[2 * r + 1] = a.src_box[2 * ax + 1];
    h[r] = g.h[ax];
    if (ax == 2) p.srcc = r;
  }
  for (int r = 0; r < 3; ++r)
    for (int q = 0; q < 2; ++q) p.k[r][q] = make_pair_k<double>(a.C, h, a.c, r, q);
  p.eps = static_cast<const double *>(a.eps);
  p.src = static_cast<const double *>(a.src);
  p.src_amp = a.src_amp;
  p.flag = a.flag;
  const int64_t nw = (int64_t)p.strips * p.nrow * p.nmarch;
  const int grid = (int)((nw + WARPS - 1) / WARPS), smem = WARPS * p.R * NST * 32 * 8;
  if (a.limiter)
    cart3d_tau0_f64_kernel<true><<<grid, WARPS * 32, smem, st>>>(p);
  else
    cart3d_tau0_f64_kernel<false><<<grid, WARPS * 32, smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace gks
