// Face flux of the 3-D Cartesian step for tau = 0 (Sec. 4.1) and mu = 1, by pairs of components.
//
// For tau -> 0 only F = C1 <u g0> + C3 <u g_t> is left, the D3Q4 third moment drops out with C2 and
// C5, and the flux of E_n and H_n through a face of normal n vanishes.  The four tangential
// components split into two pairs, (E_e, H_h) = (E_{n+1}, H_{n+2}) with S = +1 and (E_{n+2}, H_{n+1})
// with S = -1 (indices modulo 3), each of the form of the 2-D TM flux.  With r = 1/(eps_l + eps_r)
//     GE = (P_l + P_r) + kE r (QE_l + QE_r)     F_E = sE GE
//     GH = r (QH_l + QH_r)                      F_H = sH GH
// and a cell's values toward its high (l, upper signs) and its low face (r), d_a the raw central
// differences along axis a, ic = 1/c, lam = C3/(2 h_n C1):
//     P  = (H + S ic d_n E/4) +- (d_n H + 4 S ic E)/4
//     QE = (eps d_n E_e - (h_n/h_e) eps d_e E_n) +- S ic d_n H
//     QH = (eps E + S (ic/4 - lam) d_n H + S lam (h_n/h_h) d_h H_n)
//          +- (eps d_n E + 4 S ic H - 4 lam ic d_n E)/4
// : 13 operations a pair and cell.  All three axes have the same form under a cyclic renaming.
#pragma once

#include <cuda_runtime.h>

namespace gks {

// Constants of one pair of one axis (signs folded in).
template <typename T>
struct PairK {
  T q, ic4, mk, ic, mic, c0, lk, l4, kE, sE, sH, mE, mH;   // mE = -sE, mH = -sH
};

template <typename T>
inline PairK<T> make_pair_k(const double C[5], const double h[3], double c, int n, int pair) {
  const double S = pair == 0 ? 1.0 : -1.0, ic = 1.0 / c, lam = C[2] / (2.0 * h[n] * C[0]);
  const int e = (n + 1 + pair) % 3, hh = (n + 2 - pair) % 3;
  PairK<T> k;
  k.q = T(0.25 * S * ic); k.ic4 = T(4.0 * S * ic); k.mk = T(-h[n] / h[e]);
  k.ic = T(S * ic); k.mic = T(-S * ic);
  k.c0 = T(S * (0.25 * ic - lam)); k.lk = T(S * lam * h[n] / h[hh]); k.l4 = T(-4.0 * lam * ic);
  k.kE = T(-2.0 * S * lam); k.sE = T(0.5 * S * C[0] / h[n]); k.sH = T(S * C[0] / h[n]);
  k.mE = -k.sE; k.mH = -k.sH;
  return k;
}

// A cell's values for one of its faces: the two pairs' P, QE, QH.
template <typename V>
struct Sides3 {
  V v[6];
};

// OP supplies fma(k, x, a) for a constant k, add, mul(x, y), mulk(k, x).
template <class OP, typename V, typename T>
__device__ __forceinline__ void pair_sides(const V &e, const V &h, const V &ue, const V &ne,
                                           const V &nh, const V &une, const V &edt, const V &dht,
                                           const PairK<T> &k, V *l, V *r) {
  const V ev = OP::fma(k.q, ne, h), od = OP::fma(k.ic4, e, nh);
  l[0] = OP::fma(T(0.25), od, ev);
  r[0] = OP::fma(T(-0.25), od, ev);
  const V x = OP::fma(k.mk, edt, une);
  l[1] = OP::fma(k.ic, nh, x);
  r[1] = OP::fma(k.mic, nh, x);
  const V eq = OP::fma(k.lk, dht, OP::fma(k.c0, nh, ue));
  const V oq = OP::fma(k.l4, ne, OP::fma(k.ic4, h, une));
  l[2] = OP::fma(T(0.25), oq, eq);
  r[2] = OP::fma(T(-0.25), oq, eq);
}

// Both sides of a cell along axis N: v its (E, H), ue = eps E, d[a] the raw differences along axis a,
// ed[a] those of E times eps (only d[a][m] with m not along a are read).
template <int N, class OP, typename V, typename T>
__device__ __forceinline__ void cell_sides3(const V v[6], const V ue[3], const V d[3][6],
                                            const V ed[3][3], const PairK<T> k[2], Sides3<V> &l,
                                            Sides3<V> &r) {
  constexpr int P = (N + 1) % 3, Q = (N + 2) % 3;
  pair_sides<OP>(v[P], v[3 + Q], ue[P], d[N][P], d[N][3 + Q], ed[N][P], ed[P][N], d[Q][3 + N], k[0],
                 l.v, r.v);
  pair_sides<OP>(v[Q], v[3 + P], ue[Q], d[N][Q], d[N][3 + P], ed[N][Q], ed[Q][N], d[P][3 + N], k[1],
                 l.v + 3, r.v + 3);
}

// G = (GE, GH) of the two pairs of a face with inv = 1/(eps_l + eps_r).
template <class OP, typename V, typename T>
__device__ __forceinline__ void face3(const Sides3<V> &l, const Sides3<V> &r, const V &inv,
                                      const PairK<T> k[2], V G[4]) {
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const V *a = l.v + 3 * p, *b = r.v + 3 * p;
    G[2 * p] = OP::fmav(OP::mulk(k[p].kE, inv), OP::add(a[1], b[1]), OP::add(a[0], b[0]));
    G[2 * p + 1] = OP::mul(inv, OP::add(a[2], b[2]));
  }
}

// Components (0..5: E, H) that G[0..3] of a face of normal N advance.
template <int N>
__device__ __forceinline__ constexpr int face_comp(int g) {
  return g == 0 ? (N + 1) % 3 : g == 1 ? 3 + (N + 2) % 3 : g == 2 ? (N + 2) % 3 : 3 + (N + 1) % 3;
}

}  // namespace gks
