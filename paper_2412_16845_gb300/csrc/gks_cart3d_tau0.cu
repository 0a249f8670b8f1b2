// Fused 3-D GKS step on a Cartesian grid in FP32 for tau = 0 (Sec. 4.1) with mu = 1: the pair flux of
// gks_pair3.cuh in paired FP32 arithmetic, planes staged in shared memory.
//
// The march is that of cart3d_side_kernel (gks_cart3d_side.cu, which keeps tau > 0): a CTA owns 64
// columns x NWO rows of a chunk of z-planes; a row warp holds two adjacent cells per lane as the
// halves of a float2; two halo warps supply the y-sides of the rows below and above and, a plane
// ahead, the x-sides of the columns left and right of the tile; planes arrive by TMA into four slots.
// With tau = 0 a cell sends 6 values to a neighbour instead of 12 and a face carries 4 components
// instead of 6: 81 paired instructions a cell pair's worth of flux and update instead of 220, half the
// shuffles and shared-memory exchange, and the z-sides fit in registers (no tensor memory).
// Bound: latency at 12 warps an SM.  Issue slots are 49.5% active at 160^3; the stalls per issue are
// dependencies 1.5, shared memory 1.0 and the two CTA barriers a plane 0.8.  256^3: 310 to 334 us a step (back
// to back; with a state copied before and after ten steps), the side-split kernel 525; 14 row warps 348, two CTAs
// of 6 row warps 360.
#include <cuda_runtime.h>

#include "gks_internal.h"
#include "gks_pdl.cuh"
#include "gks_pair3.cuh"
#include "gks_rcp.cuh"
#include "gks_shared_limit.h"
#include "gks_tma.cuh"

namespace gks {
namespace {

constexpr int NWO = 10;                 // row warps per CTA
constexpr int NWARP = NWO + 2;          // plus the halo warps H0 (below) and H1 (above)
constexpr int NTH = NWARP * 32;
constexpr int CTAS = 1;                 // per SM
constexpr int TCOLS = 64;               // columns per CTA (two per lane)
constexpr int TW = 72;                  // staged columns X0-4 .. X0+67 (16-byte chunks)
constexpr int NR = NWO + 4;             // staged rows y0-2 .. y0+NWO+1
constexpr int NA = 7;                   // staged arrays: Ex, Ey, Ez, Hx, Hy, Hz, eps
constexpr int NSLOT = 4;
constexpr unsigned FULL = 0xffffffffu;
// wrapped entries of a staged plane on periodic sides: two layers beyond each side, every row
// for columns and every column for rows, all arrays
constexpr int kMaxFix = NA * (4 * NR + 4 * TW);

using f2 = float2;

__device__ __forceinline__ f2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ f2 vrcp(f2 s) { return pk(rcp_normal(s.x), rcp_normal(s.y)); }

// Paired FP32 arithmetic (two cells per value); a constant is a scalar kernel parameter replicated
// into both halves, which the paired FMA reads straight from the constant bank.
struct OpP {
  static __device__ __forceinline__ f2 fma(float k, f2 x, f2 a) { return __ffma2_rn(pk(k, k), x, a); }
  static __device__ __forceinline__ f2 fmav(f2 k, f2 x, f2 a) { return __ffma2_rn(k, x, a); }
  static __device__ __forceinline__ f2 add(f2 a, f2 b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ f2 sub(f2 a, f2 b) { return __ffma2_rn(b, pk(-1.f, -1.f), a); }
  static __device__ __forceinline__ f2 mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ f2 mulk(float k, f2 x) { return __fmul2_rn(pk(k, k), x); }
};
struct OpS {
  static __device__ __forceinline__ float fma(float k, float x, float a) { return fmaf(k, x, a); }
  static __device__ __forceinline__ float fmav(float k, float x, float a) { return fmaf(k, x, a); }
  static __device__ __forceinline__ float add(float a, float b) { return a + b; }
  static __device__ __forceinline__ float mul(float a, float b) { return a * b; }
  static __device__ __forceinline__ float mulk(float k, float x) { return k * x; }
};

struct Args {
  const float *V;                      // (not __restrict__: gks_pdl.cuh)
  float *Vout;
  const float *eps;
  const float *src;
  int sx0, sx1, sy0, sy1, sz0, sz1;
  float src_amp;
  int nx, ny, nz;
  int64_t pitch, plane, cstride;
  int per[3];
  int zchunk;
  int *flag;
  PairK<float> k[3][2];
};

// One staged plane in the TMA box order (array, row, column); slots start 128-byte aligned.
struct alignas(128) PlaneSlot {
  float a[NA][NR][TW];
};

struct Smem {
  PlaneSlot V[NSLOT];                  // staged planes
  unsigned long long bar[NSLOT];       // one mbarrier per slot
  int err;                             // a bounded wait ran out (shared by the CTA)
  f2 Y[NWO + 1][6][32];                // sides of each row toward the row below
  f2 F[NWO + 1][4][32];                // flux through the face above each row; [NWO]: below row 0
  float XL[2][NWO][7];                 // side of column X0-1 toward the tile, and its eps
  float XR[2][NWO][7];                 // side of column X0+64 toward the tile, and its eps
  // periodic sides: staged entries past the grid that hold wrapped cells (the TMA box leaves
  // them zero): position in a plane slot (array, row, column) and source offset in a plane
  unsigned short fixd[kMaxFix];
  int fixg[kMaxFix];
  int nfix;
};
static_assert(sizeof(Smem) <= 227 * 1024, "shared memory of one SM");

__device__ __forceinline__ int wrap_or_clamp(int i, int n, int periodic) {
  if (periodic) {
    i %= n;
    return i < 0 ? i + n : i;
  }
  return i < 0 ? 0 : (i >= n ? n - 1 : i);
}

constexpr unsigned kPlaneBytes = NA * NR * TW * 4;   // one staged plane (both tensor boxes)

// One thread: the tensor copies of plane gz into slot `slot` (fields box, then eps box), both
// completing on the slot's mbarrier.  Earlier generic-proxy reads of the slot are ordered before
// the copies by the CTA barrier that precedes the call and the proxy fence here.
__device__ __forceinline__ void tma_plane(Smem &s, const CUtensorMap *tmV,
                                          const CUtensorMap *tmE, int slot, int x, int y,
                                          int gz) {
  unsigned long long *b = &s.bar[slot];
  fence_proxy_async();
  mbar_expect_tx(b, kPlaneBytes);
  tma_load_4d(&s.V[slot].a[0][0][0], tmV, x, y, gz, 0, b);
  tma_load_3d(&s.V[slot].a[6][0][0], tmE, x, y, gz, b);
}

// Periodic sides: the list of staged entries that hold wrapped cells (x = -2, -1, nx, nx+1 on a
// periodic x axis, every row; y = -2, -1, ny, ny+1 on a periodic y axis, every column; all
// arrays).  The tensor copy leaves them zero.  Built once per CTA; non-reflecting sides need no
// entries, their reads are clamped instead.
__device__ __forceinline__ void build_fix_list(Smem &s, const Args &a, int X0, int y0,
                                               int tid) {
  unsigned cols = 0, rows = 0;        // up to four tile columns and rows, one byte each
  int nc = 0, nr = 0;
  for (int g = 1; g <= 2; ++g) {
    const int tl = -g - (X0 - 4), th = a.nx - 1 + g - (X0 - 4);
    const int rl = -g - (y0 - 2), rh = a.ny - 1 + g - (y0 - 2);
    if (a.per[0] && tl >= 0 && tl < TW) cols |= (unsigned)tl << (8 * nc++);
    if (a.per[0] && th >= 0 && th < TW) cols |= (unsigned)th << (8 * nc++);
    if (a.per[1] && rl >= 0 && rl < NR) rows |= (unsigned)rl << (8 * nr++);
    if (a.per[1] && rh >= 0 && rh < NR) rows |= (unsigned)rh << (8 * nr++);
  }
  const int n1 = NA * NR * nc, n = n1 + NA * nr * TW;
  for (int i = tid; i < n; i += NTH) {
    int arr, r, t;
    if (i < n1) {
      t = (cols >> (8 * (i % nc))) & 0xff;
      r = (i / nc) % NR;
      arr = i / (nc * NR);
    } else {
      const int j = i - n1;
      t = j % TW;
      r = (rows >> (8 * ((j / TW) % nr))) & 0xff;
      arr = j / (TW * nr);
    }
    const int gx = wrap_or_clamp(X0 - 4 + t, a.nx, a.per[0]);
    const int gy = wrap_or_clamp(y0 - 2 + r, a.ny, a.per[1]);
    s.fixd[i] = (unsigned short)((arr * NR + r) * TW + t);
    s.fixg[i] = gy * (int)a.pitch + gx;
  }
  if (tid == 0) s.nfix = n;
}

// Write the wrapped entries of plane gz into its slot (all threads; four loads in flight each).
__device__ __forceinline__ void fix_plane(Smem &s, const Args &a, int slot, int gz,
                                          int tid) {
  const int n = s.nfix;
  float *dst = &s.V[slot].a[0][0][0];
  for (int i0 = tid; i0 < n; i0 += 4 * NTH) {
    float v[4];
    int d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * NTH;
      d[u] = -1;
      v[u] = 0.f;
      if (i < n) {
        const int dd = s.fixd[i], arr = dd / (NR * TW);
        v[u] = __ldcg((arr < 6 ? a.V + arr * a.cstride : a.eps) + (int64_t)gz * a.plane + s.fixg[i]);
        d[u] = dd;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (d[u] >= 0) dst[d[u]] = v[u];
  }
}

// Where a lane reads the staged planes.  On a non-reflecting side the reads are clamped to the
// grid (the Green-Gauss ghost copy), so the zero-filled entries past the grid are never read;
// on a periodic side they are the wrapped entries the fix-up list writes.
struct Taps {
  int r, rm, rp;          // rows of the warp's cells and of their lower / upper neighbours
  int t0, t1;             // columns of the lane's two cells
  int tm, tp;             // left neighbour of the first cell, right neighbour of the second
  bool pair;              // the warp's two cells of every lane are adjacent and aligned
};

// The own pair (both columns of the lane) of one staged row: 6 fields and eps.
__device__ __forceinline__ void load_pair(const Smem &s, int slot, const Taps &q, f2 v[7]) {
  if (q.pair) {
#pragma unroll
    for (int m = 0; m < NA; ++m) v[m] = *reinterpret_cast<const f2 *>(&s.V[slot].a[m][q.r][q.t0]);
  } else {
#pragma unroll
    for (int m = 0; m < NA; ++m) v[m] = pk(s.V[slot].a[m][q.r][q.t0], s.V[slot].a[m][q.r][q.t1]);
  }
}

// Raw central differences of the lane's two cells in plane slot s0 (d[a][m], m not along a), the
// planes below (vm) and above (vp) in registers, and the eps-weighted E rows.
__device__ __forceinline__ void differences(const Smem &s, int s0, const Taps &q, const f2 v[7],
                                            const f2 vm[7], const f2 vp[7], f2 d[3][6], f2 ue[3],
                                            f2 ed[3][3]) {
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    if (m % 3 != 0) {
      const float xm = s.V[s0].a[m][q.r][q.tm], xp = s.V[s0].a[m][q.r][q.tp];
      d[0][m] = pk(v[m].y - xm, xp - v[m].x);
    }
    if (m % 3 != 1) {
      f2 ym, yp;
      if (q.pair) {
        ym = *reinterpret_cast<const f2 *>(&s.V[s0].a[m][q.rm][q.t0]);
        yp = *reinterpret_cast<const f2 *>(&s.V[s0].a[m][q.rp][q.t0]);
      } else {
        ym = pk(s.V[s0].a[m][q.rm][q.t0], s.V[s0].a[m][q.rm][q.t1]);
        yp = pk(s.V[s0].a[m][q.rp][q.t0], s.V[s0].a[m][q.rp][q.t1]);
      }
      d[1][m] = OpP::sub(yp, ym);
    }
    if (m % 3 != 2) d[2][m] = OpP::sub(vp[m], vm[m]);
  }
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    ue[m] = OpP::mul(v[6], v[m]);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a != m) ed[a][m] = OpP::mul(v[6], d[a][m]);
  }
}

// The x-side of one cell at tile column t, row r of plane slots (sm, s0, sp): the columns left and
// right of the tile, computed by the halo warps.  high: toward +x, else toward -x.
__device__ __forceinline__ void halo_x_cell(const Smem &s, int sm, int s0, int sp, int r, int rm,
                                            int rp, int t, int tm, int tp, const PairK<float> k[2],
                                            bool high, bool ghost, float out[7]) {
  float v[6], d[3][6], ue[3], ed[3][3];
  const float e = s.V[s0].a[6][r][t];
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    v[m] = s.V[s0].a[m][r][t];
    if (m % 3 != 0) d[0][m] = s.V[s0].a[m][r][tp] - s.V[s0].a[m][r][tm];
    if (m % 3 != 1) d[1][m] = s.V[s0].a[m][rp][t] - s.V[s0].a[m][rm][t];
    if (m % 3 != 2) d[2][m] = s.V[sp].a[m][r][t] - s.V[sm].a[m][r][t];
  }
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    ue[m] = e * v[m];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (a != m) ed[a][m] = e * d[a][m];
  }
  Sides3<float> l, r_;
  cell_sides3<0, OpS>(v, ue, d, ed, k, l, r_);
#pragma unroll
  for (int m = 0; m < 6; ++m) out[m] = ghost ? 0.f : (high ? l.v[m] : r_.v[m]);
  out[6] = e;
}

__device__ __forceinline__ void zero6(Sides3<f2> &a) {
#pragma unroll
  for (int m = 0; m < 6; ++m) a.v[m] = pk(0.f, 0.f);
}

__global__ void __launch_bounds__(NTH, CTAS)
    cart3d_tau0_kernel(const __grid_constant__ CUtensorMap tmV,
                       const __grid_constant__ CUtensorMap tmE, const __grid_constant__ Args a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  grid_wait();
  grid_trigger();
  Smem &s = *reinterpret_cast<Smem *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int X0 = blockIdx.x * TCOLS, y0 = blockIdx.y * NWO;
  const int z0 = blockIdx.z * a.zchunk;
  const int z1 = min(z0 + a.zchunk, a.nz);
  const bool owned = warp < NWO, h0 = warp == NWO, h1 = warp == NWO + 1;
  const int y = y0 - 2 + (owned ? warp + 2 : (h0 ? 1 : NWO + 2));   // the warp's grid row
  const int x = X0 + 2 * lane;                               // grid column of its first cell
  // non-reflecting ghosts (outside the grid on a non-periodic axis) carry no distributions
  const bool yghost = !a.per[1] && (y < 0 || y >= a.ny);
  const bool xg0 = !a.per[0] && x >= a.nx, xg1 = !a.per[0] && x + 1 >= a.nx;
  const bool st0 = x < a.nx, st1 = x + 1 < a.nx;            // columns this lane stores
  // read positions: clamped to the grid on non-reflecting sides
  auto trow = [&](int yy) { return (a.per[1] ? yy : min(max(yy, 0), a.ny - 1)) - (y0 - 2); };
  auto tcol = [&](int xx) { return (a.per[0] ? xx : min(max(xx, 0), a.nx - 1)) - (X0 - 4); };
  Taps q;
  q.r = trow(y);
  q.rm = trow(y - 1);
  q.rp = trow(y + 1);
  q.t0 = tcol(x);
  q.t1 = tcol(x + 1);
  q.tm = tcol(x - 1);
  q.tp = tcol(x + 2);
  q.pair = __all_sync(FULL, q.t1 == q.t0 + 1 && (q.t0 & 1) == 0);
  // the halo warps' x-halo cells: row y0 + lane, column X0 - 1 (H0) or X0 + 64 (H1)
  const int hy = y0 + lane;
  const int hr = trow(hy), hrm = trow(hy - 1), hrp = trow(hy + 1);
  const int hx = h0 ? X0 - 1 : X0 + TCOLS;
  const bool hghost = !a.per[0] && (hx < 0 || hx >= a.nx);
  const int ht = tcol(hx), htm = tcol(hx - 1), htp = tcol(hx + 1);

  // ---------------- prologue: planes z0-1 .. z0+2 staged; z-vectors of plane z0-1
  // plane p sits in slot p mod NSLOT; it is that slot's ((p - z0 + 1) / NSLOT)-th load
  auto slot_of = [](int p) { return (p + 2 * NSLOT) % NSLOT; };
  auto parity_of = [z0](int p) { return (unsigned)(((p - z0 + 1) / NSLOT) & 1); };
  auto zidx = [&a](int p) { return wrap_or_clamp(p, a.nz, a.per[2]); };
  const bool issuer = tid == NWO * 32;                       // lane 0 of H0 issues the copies
  const int last_plane = max(z0 + 3, z1 + 1);                // the last plane this CTA loads
  if (tid == 0) {
    for (int i = 0; i < NSLOT; ++i) mbar_init(&s.bar[i], 1);
    s.err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  build_fix_list(s, a, X0, y0, tid);
  __syncthreads();
  if (issuer)
    for (int p = z0 - 1; p <= z0 + 2; ++p)
      tma_plane(s, &tmV, &tmE, slot_of(p), X0 - 4, y0 - 2, zidx(p));
  // own pair at plane z0-2 (wrapped or clamped, always inside the grid), loaded while the
  // staged planes are in flight
  f2 Wm[7];
  {
    const int gz = wrap_or_clamp(z0 - 2, a.nz, a.per[2]);
    const int gy = wrap_or_clamp(y, a.ny, a.per[1]);
    const int c0 = wrap_or_clamp(x, a.nx, a.per[0]), c1 = wrap_or_clamp(x + 1, a.nx, a.per[0]);
    const int64_t o = (int64_t)gz * a.plane + (int64_t)gy * a.pitch;
#pragma unroll
    for (int m = 0; m < NA; ++m) {
      const float *base = (m < 6 ? a.V + m * a.cstride : a.eps) + o;
      Wm[m] = pk(__ldcg(base + c0), __ldcg(base + c1));
    }
  }
  {
    bool ok = true;
    for (int p = z0 - 1; p <= z0 + 2; ++p) ok &= mbar_wait(&s.bar[slot_of(p)], parity_of(p));
    if (!ok) { s.err = 1; atomicOr(a.flag, 2); }
    for (int p = z0 - 1; p <= z0 + 2; ++p) fix_plane(s, a, slot_of(p), zidx(p), tid);
  }
  __syncthreads();
  if (s.err) return;                                          // nothing else is in flight

  f2 W0[7], Wp[7];                      // own pair at planes k, k+1 (Wm: k-1)
  f2 B[6], Minv = pk(0.f, 0.f);         // pending update of plane k-1 (z-face components)
  Sides3<f2> zl;                        // sides of plane k-1 toward plane k
  load_pair(s, slot_of(z0 - 1), q, W0);
  load_pair(s, slot_of(z0), q, Wp);
#pragma unroll
  for (int m = 0; m < 6; ++m) B[m] = pk(0.f, 0.f);
  if (owned) {
    f2 d[3][6], ue[3], ed[3][3];
    Sides3<f2> r;
    differences(s, slot_of(z0 - 1), q, W0, Wm, Wp, d, ue, ed);
    cell_sides3<2, OpP>(W0, ue, d, ed, a.k[2], zl, r);
    if (!a.per[2] && z0 == 0) zero6(zl);
  } else if (lane < NWO) {
    // x-halo sides of plane z0 (slots z0-1, z0, z0+1)
    float o[7];
    halo_x_cell(s, slot_of(z0 - 1), slot_of(z0), slot_of(z0 + 1), hr, hrm, hrp, ht, htm, htp, a.k[0],
                h0, hghost, o);
    float *dst = h0 ? s.XL[z0 & 1][lane] : s.XR[z0 & 1][lane];
#pragma unroll
    for (int u = 0; u < 7; ++u) dst[u] = o[u];
  }
#pragma unroll
  for (int m = 0; m < NA; ++m) { Wm[m] = W0[m]; W0[m] = Wp[m]; }
  __syncthreads();

  bool bad = false;
  const bool store_row = owned && y < a.ny;
  float *out = a.Vout + (int64_t)z0 * a.plane + (int64_t)y * a.pitch + x;   // plane k
  auto put = [&](float *o, f2 v) {
    if (st1)
      *reinterpret_cast<f2 *>(o) = v;
    else if (st0)
      *o = v.x;
  };
  auto check = [&](f2 v) {
    if (st1) bad |= !(isfinite(v.x) && isfinite(v.y));
    else if (st0) bad |= !isfinite(v.x);
  };
  // ---------------- march: plane k's x- and y-faces, the z-face below it (completing k-1)
#pragma unroll 1
  for (int k = z0; k <= z1; ++k) {
    const bool last = k == z1;                 // only the z-face below plane z1 remains
    if (issuer && k + 3 <= last_plane)         // plane k-1's slot is free
      tma_plane(s, &tmV, &tmE, slot_of(k + 3), X0 - 4, y0 - 2, zidx(k + 3));
    const int s0 = slot_of(k), sp = slot_of(k + 1);
    load_pair(s, sp, q, Wp);
    f2 acc[6];
    if (owned) {
      f2 d[3][6], ue[3], ed[3][3], G[4];
      differences(s, s0, q, W0, Wm, Wp, d, ue, ed);
#pragma unroll
      for (int m = 0; m < 6; ++m) acc[m] = m < 3 ? pk(0.f, 0.f) : W0[m];
      // z: the face below plane k; completes plane k-1
      {
        Sides3<f2> l, r;
        cell_sides3<2, OpP>(W0, ue, d, ed, a.k[2], l, r);
        if (!a.per[2] && k == a.nz) zero6(r);
        face3<OpP>(zl, r, vrcp(OpP::add(Wm[6], W0[6])), a.k[2], G);
        if (k > z0 && store_row) {
          f2 sum = pk(0.f, 0.f);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = face_comp<2>(i);
            const f2 nv = (i & 1) ? OpP::fma(a.k[2][i / 2].mH, G[i], B[c])
                                  : OpP::fmav(Minv, OpP::mulk(a.k[2][i / 2].mE, G[i]), B[c]);
            put(out + c * a.cstride - a.plane, nv);
            sum = OpP::add(sum, nv);
          }
          check(sum);
        }
        if (last) break;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = face_comp<2>(i);
          acc[c] = OpP::fma((i & 1) ? a.k[2][i / 2].sH : a.k[2][i / 2].sE, G[i], acc[c]);
        }
        zl = l;
      }
      // x: faces x+1/2 of both cells; the second needs the next lane's first cell
      {
        Sides3<f2> l, r;
        cell_sides3<0, OpP>(W0, ue, d, ed, a.k[0], l, r);
        if (xg0 | xg1) {                        // ghost columns past the high x side
#pragma unroll
          for (int m = 0; m < 6; ++m) {
            if (xg0) l.v[m].x = r.v[m].x = 0.f;
            if (xg1) l.v[m].y = r.v[m].y = 0.f;
          }
        }
        const int par = k & 1;
        Sides3<f2> rn;                          // sides of the cells to the right
        float re = __shfl_down_sync(FULL, W0[6].x, 1);
#pragma unroll
        for (int m = 0; m < 6; ++m) {
          rn.v[m].x = r.v[m].y;
          rn.v[m].y = __shfl_down_sync(FULL, r.v[m].x, 1);
        }
        if (lane == 31) {                       // column X0+64 (halo warp H1)
#pragma unroll
          for (int m = 0; m < 6; ++m) rn.v[m].y = s.XR[par][warp][m];
          re = s.XR[par][warp][6];
        }
        face3<OpP>(l, rn, vrcp(OpP::add(W0[6], pk(W0[6].y, re))), a.k[0], G);
        float Gm[4];                            // the face left of the first cell
#pragma unroll
        for (int i = 0; i < 4; ++i) Gm[i] = __shfl_up_sync(FULL, G[i].y, 1);
        if (lane == 0) {                        // column X0-1 (H0)
          Sides3<float> hl, hr_;
#pragma unroll
          for (int m = 0; m < 6; ++m) {
            hl.v[m] = s.XL[par][warp][m];
            hr_.v[m] = r.v[m].x;
          }
          face3<OpS>(hl, hr_, rcp_normal(s.XL[par][warp][6] + W0[6].x), a.k[0], Gm);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = face_comp<0>(i);
          acc[c] = OpP::fma((i & 1) ? a.k[0][i / 2].mH : a.k[0][i / 2].mE,
                            pk(G[i].x - Gm[i], G[i].y - G[i].x), acc[c]);
        }
      }
      // y: sides published for the row below; the face above waits for the barrier
      Sides3<f2> l, r;
      cell_sides3<1, OpP>(W0, ue, d, ed, a.k[1], l, r);
      if (yghost) {
        zero6(l);
        zero6(r);
      }
#pragma unroll
      for (int m = 0; m < 6; ++m) s.Y[warp][m][lane] = r.v[m];
      __syncthreads();                          // B1: the sides of every row
      {
        const f2 eu = q.pair ? *reinterpret_cast<const f2 *>(&s.V[s0].a[6][q.rp][q.t0])
                             : pk(s.V[s0].a[6][q.rp][q.t0], s.V[s0].a[6][q.rp][q.t1]);
        Sides3<f2> up;
#pragma unroll
        for (int m = 0; m < 6; ++m) up.v[m] = s.Y[warp + 1][m][lane];
        face3<OpP>(l, up, vrcp(OpP::add(W0[6], eu)), a.k[1], G);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = face_comp<1>(i);
          s.F[warp][i][lane] = G[i];
          acc[c] = OpP::fma((i & 1) ? a.k[1][i / 2].mH : a.k[1][i / 2].mE, G[i], acc[c]);
        }
      }
    } else {
      // halo warps: the y-sides of their row, and the x-halo columns of plane k+1
      if (last) break;
      f2 d[3][6], ue[3], ed[3][3];
      Sides3<f2> l, r;
      differences(s, s0, q, W0, Wm, Wp, d, ue, ed);
      cell_sides3<1, OpP>(W0, ue, d, ed, a.k[1], l, r);
      if (yghost) {
        zero6(l);
        zero6(r);
      }
      if (h1) {
#pragma unroll
        for (int m = 0; m < 6; ++m) s.Y[NWO][m][lane] = r.v[m];
      }
      if (lane < NWO) {
        float o[7];
        halo_x_cell(s, s0, sp, slot_of(k + 2), hr, hrm, hrp, ht, htm, htp, a.k[0], h0, hghost, o);
        float *dst = h0 ? s.XL[(k + 1) & 1][lane] : s.XR[(k + 1) & 1][lane];
#pragma unroll
        for (int u = 0; u < 7; ++u) dst[u] = o[u];
      }
      __syncthreads();                          // B1
      if (h0) {                                 // face below row y0
        const f2 eu = q.pair ? *reinterpret_cast<const f2 *>(&s.V[s0].a[6][q.rp][q.t0])
                             : pk(s.V[s0].a[6][q.rp][q.t0], s.V[s0].a[6][q.rp][q.t1]);
        Sides3<f2> up;
        f2 G[4];
#pragma unroll
        for (int m = 0; m < 6; ++m) up.v[m] = s.Y[0][m][lane];
        face3<OpP>(l, up, vrcp(OpP::add(W0[6], eu)), a.k[1], G);
#pragma unroll
        for (int i = 0; i < 4; ++i) s.F[NWO][i][lane] = G[i];
      }
    }
    if (k + 3 <= last_plane) {
      if (!mbar_wait(&s.bar[slot_of(k + 3)], parity_of(k + 3))) {
        s.err = 1;                              // plane k+3 never landed
        atomicOr(a.flag, 2);
      } else if (s.nfix) {
        fix_plane(s, a, slot_of(k + 3), zidx(k + 3), tid);   // periodic sides: wrapped cells
      }
    }
    __syncthreads();                            // B2: face fluxes; plane k+3 visible
    if (s.err) break;                           // leave together; no copy is in flight
    if (owned) {
      const int below = warp == 0 ? NWO : warp - 1;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = face_comp<1>(i);
        acc[c] = OpP::fma((i & 1) ? a.k[1][i / 2].sH : a.k[1][i / 2].sE, s.F[below][i][lane], acc[c]);
      }
      if (a.src && y >= a.sy0 && y < a.sy1 && k >= a.sz0 && k < a.sz1) {
        const int64_t o = (int64_t)k * a.plane + (int64_t)y * a.pitch;
        if (x >= a.sx0 && x < a.sx1) acc[2].x -= a.src_amp * a.src[o + x];
        if (x + 1 >= a.sx0 && x + 1 < a.sx1) acc[2].y -= a.src_amp * a.src[o + x + 1];
      }
      Minv = vrcp(W0[6]);
#pragma unroll
      for (int m = 0; m < 6; ++m) B[m] = m < 3 ? OpP::fmav(Minv, acc[m], W0[m]) : acc[m];
      if (store_row) {                          // no z-face changes E_z and H_z
        put(out + 2 * a.cstride, B[2]);
        put(out + 5 * a.cstride, B[5]);
        check(OpP::add(B[2], B[5]));
      }
      out += a.plane;
    }
#pragma unroll
    for (int m = 0; m < NA; ++m) Wm[m] = W0[m];
    load_pair(s, sp, q, W0);                   // plane k+1 (still staged) is the next W0
  }
  if (__any_sync(FULL, bad) && lane == 0) atomicOr(a.flag, 1);
}

// Tensor map of `rank` dims over a [ncomp][nz][ny][pitch] FP32 array: dims (nx, ny, nz[, 6]),
// box (TW, NR, 1[, 6]); entries past the grid read as zero.
bool encode_map(CUtensorMap *m, const float *base, const CartGeom &g, int rank) {
  const cuuint64_t dim[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, 6};
  const cuuint64_t stride[3] = {(cuuint64_t)g.pitch * 4, (cuuint64_t)g.plane * 4,
                                (cuuint64_t)g.cstride * 4};
  const cuuint32_t box[4] = {TW, NR, 1, 6};
  return encode_f32_map(m, base, rank, dim, stride, box);
}

}  // namespace

bool cart3d_tau0_supported(const CartGeom &g, const CartStepArgs &a) {
  return cart3d_side_supported(g, a, false) && a.eps_normal && a.C[1] == 0.0 && a.C[3] == 0.0 &&
         a.C[4] == 0.0 && a.C[0] > 0.0;
}

cudaError_t launch_cart3d_tau0(const CartGeom &g, const CartStepArgs &a, cudaStream_t st) {
  Args p;
  p.V = static_cast<const float *>(a.V);
  p.Vout = static_cast<float *>(a.Vout);
  p.eps = static_cast<const float *>(a.eps);
  p.src = static_cast<const float *>(a.src);
  p.sx0 = a.src_box[0]; p.sx1 = a.src_box[1];
  p.sy0 = a.src_box[2]; p.sy1 = a.src_box[3];
  p.sz0 = a.src_box[4]; p.sz1 = a.src_box[5];
  p.src_amp = float(a.src_amp);
  p.nx = g.nx; p.ny = g.ny; p.nz = g.nz;
  p.pitch = g.pitch; p.plane = g.plane; p.cstride = g.cstride;
  for (int d = 0; d < 3; ++d) p.per[d] = g.periodic[d];
  p.flag = a.flag;
  for (int A = 0; A < 3; ++A)
    for (int q = 0; q < 2; ++q) p.k[A][q] = make_pair_k<float>(a.C, g.h, a.c, A, q);
  const int gx = (g.nx + TCOLS - 1) / TCOLS, gy = (g.ny + NWO - 1) / NWO;
  const int smem = (int)sizeof(Smem);
  static SharedLimit limit;
  const cudaError_t e = limit.raise(smem, cart3d_tau0_kernel);
  if (e != cudaSuccess) return e;
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = sms > 0 ? sms * CTAS : 1;
  }
  // z chunks: one CTA per SM; pick the chunk count that fills whole waves best.  A CTA's fixed
  // cost -- staging its first four planes with nothing to overlap them, the z-vectors of the
  // plane below its chunk and the closing z-face -- counts as 2.7 planes of work.  The rule takes the fastest
  // count of 1 to 32 at four sizes (us a step): 256^3 7 chunks 310, 4: 317, 16: 326, 1: 410; 160^3 3: 106,
  // 5: 120; 200 x 128 x 90 5: 72, 2: 88; 300 x 200 x 100 3: 143, 5: 154.
  constexpr double kChunkCost = 2.7;
  const int64_t tiles = (int64_t)gx * gy;
  int zchunks = 1;
  double best = -1.0;
  for (int zc = 1; zc <= 64 && zc <= g.nz; ++zc) {
    const int len = (g.nz + zc - 1) / zc;
    const int nzc = (g.nz + len - 1) / len;
    const int64_t ctas = tiles * nzc;
    const double waves = (double)((ctas + sms - 1) / sms);
    const double eff =
        (double)ctas / (waves * sms) * (double)g.nz / ((double)nzc * (len + kChunkCost));
    if (eff > best + 1e-9) { best = eff; zchunks = nzc; }
  }
  p.zchunk = (g.nz + zchunks - 1) / zchunks;
  zchunks = (g.nz + p.zchunk - 1) / p.zchunk;
  CUtensorMap tmV, tmE;
  if (!encode_map(&tmV, p.V, g, 4) || !encode_map(&tmE, p.eps, g, 3)) return cudaErrorInvalidValue;
  dim3 grid(gx, gy, zchunks);
  return launch_pdl(cart3d_tau0_kernel, grid, NTH, smem, st, tmV, tmE, p);
}

}  // namespace gks
