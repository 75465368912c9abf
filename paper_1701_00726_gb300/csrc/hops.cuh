// Per-offset constants of the Brillouin stencil and the spin algebra of its
// hops, shared by the stencil kernel and the adjoint (force) kernel.
#pragma once

#include "stencil.cuh"

namespace bri {

// Stored offsets nu = 1..40 with their identity weight -2^{-k-3} and the
// signed gamma weights c_k s_mu, c_k = 4^{2-k}/27.
template <typename R> struct HopTable {
  int site_d[40][4];
  R a[40];
  R cs[40][4];
};
template <typename R> void fill_hops(HopTable<R>& h) {
  for (int j = 0; j < 40; ++j) {
    const int d[4] = {j % 3 - 1, (j / 3) % 3 - 1, (j / 9) % 3 - 1, (j / 27) % 3 - 1};
    int k = 0;
    for (int mu = 0; mu < 4; ++mu) k += d[mu] != 0;
    const double c = double(1 << (2 * (4 - k))) / 432.0;
    h.a[j] = (R)(-1.0 / double(1 << (k + 3)));
    for (int mu = 0; mu < 4; ++mu) {
      h.site_d[j][mu] = d[mu];
      h.cs[j][mu] = (R)(c * d[mu]);
    }
  }
}

// The table of one precision, built once per process on the host and passed
// to the kernels by value (a __grid_constant__ parameter, read from the
// constant bank), so no translation unit has device state to upload.
template <typename R> const HopTable<R>& hop_table() {
  static const HopTable<R> t = [] {
    HopTable<R> h;
    fill_hops(h);
    return h;
  }();
  return t;
}

// In the chiral basis sum_mu s_mu gamma_mu = [[0, B], [B^dagger, 0]],
// B = s_4 - i (s_1 sigma_1 + s_2 sigma_2 + s_3 sigma_3).
// acc += c gamma_mu v over one colour (four spins), chiral basis:
// MU = 1..4.
template <int MU, typename R>
__device__ __forceinline__ void gamma_term(C<R> acc[4], const C<R> v[4], R c) {
  if constexpr (MU == 1) {
    acc[0].re = fma(c, v[3].im, acc[0].re); acc[0].im = fma(-c, v[3].re, acc[0].im);
    acc[1].re = fma(c, v[2].im, acc[1].re); acc[1].im = fma(-c, v[2].re, acc[1].im);
    acc[2].re = fma(-c, v[1].im, acc[2].re); acc[2].im = fma(c, v[1].re, acc[2].im);
    acc[3].re = fma(-c, v[0].im, acc[3].re); acc[3].im = fma(c, v[0].re, acc[3].im);
  } else if constexpr (MU == 2) {
    acc[0].re = fma(-c, v[3].re, acc[0].re); acc[0].im = fma(-c, v[3].im, acc[0].im);
    acc[1].re = fma(c, v[2].re, acc[1].re); acc[1].im = fma(c, v[2].im, acc[1].im);
    acc[2].re = fma(c, v[1].re, acc[2].re); acc[2].im = fma(c, v[1].im, acc[2].im);
    acc[3].re = fma(-c, v[0].re, acc[3].re); acc[3].im = fma(-c, v[0].im, acc[3].im);
  } else if constexpr (MU == 3) {
    acc[0].re = fma(c, v[2].im, acc[0].re); acc[0].im = fma(-c, v[2].re, acc[0].im);
    acc[1].re = fma(-c, v[3].im, acc[1].re); acc[1].im = fma(c, v[3].re, acc[1].im);
    acc[2].re = fma(-c, v[0].im, acc[2].re); acc[2].im = fma(c, v[0].re, acc[2].im);
    acc[3].re = fma(c, v[1].im, acc[3].re); acc[3].im = fma(-c, v[1].re, acc[3].im);
  } else {
    acc[0].re = fma(c, v[2].re, acc[0].re); acc[0].im = fma(c, v[2].im, acc[0].im);
    acc[1].re = fma(c, v[3].re, acc[1].re); acc[1].im = fma(c, v[3].im, acc[1].im);
    acc[2].re = fma(c, v[0].re, acc[2].re); acc[2].im = fma(c, v[0].im, acc[2].im);
    acc[3].re = fma(c, v[1].re, acc[3].re); acc[3].im = fma(c, v[1].im, acc[3].im);
  }
}

}  // namespace bri
