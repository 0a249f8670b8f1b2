// Constants of the 2-D TM flux for tau = 0 and mu = 1 (see gks_cart2d_tau0.cu), shared by the step, its
// several-step form on small grids and its adjoint.
#pragma once

namespace gks {

// Constants of one axis, with ic = +-1/c, k3 = +-C3/(2 h_n C1), ka = -+C3/(2 h_t C1) (x upper, y
// lower signs): mic = -ic, mq = -ic/4, m4 = -4 ic, c0 = k3 - ic/4, l4 = -4 k3 ic, kE = 2 k3 and the
// flux scales sE = -+C1/(2 h_n), sH = -+C1/h_n.
template <typename T>
struct AxisK {
  T ic, mic, mq, m4, c0, l4, ka, kE, sE, sH;
};

template <typename T>
AxisK<T> make_axis(const double C[5], double c, double hn, double ht, double sign) {
  const double ic = sign / c, k3 = sign * C[2] / (2.0 * hn * C[0]);
  AxisK<T> k;
  k.ic = T(ic); k.mic = T(-ic); k.mq = T(-0.25 * ic); k.m4 = T(-4.0 * ic);
  k.c0 = T(k3 - 0.25 * ic); k.l4 = T(-4.0 * k3 * ic);
  k.ka = T(-sign * C[2] / (2.0 * ht * C[0])); k.kE = T(2.0 * k3);
  k.sE = T(-sign * 0.5 * C[0] / hn); k.sH = T(-sign * C[0] / hn);
  return k;
}

}  // namespace gks
