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

// The 40 stored offsets in the order the stencils take them, with the gamma
// weights for V = -(P - Q), c_mu = -(sign) c_k s_mu.  The offsets come with the most
// hops (the smallest weights) first, so the accumulator stays small for most of its
// roundings (FP32, relative error against FP64 at 16^3 x 32 and 24^3 x 48: 7.5e-8
// sorted, 1.0e-7 in storage order).  Among those of equal weight, each aligned four
// have at most three directions between them where that is possible: the four
// thread groups of a warp then skip the same gamma terms (bri_split.cuh).
template <typename R> struct PairHops {
  int j[40];     // index of the stored offset
  int d[40][4];  // displacement signs
  R a[40];
  R c[40][4];
};
template <typename R> const PairHops<R>& pair_hops(int dagger) {
  static const auto make = [](R sgn) {
    PairHops<R> t;
    const HopTable<R>& h = hop_table<R>();
    constexpr int masks[15] = {15, 7, 11, 13, 14, 3, 5, 6, 10, 9, 12, 1, 2, 4, 8};  // directions of an offset
    int i = 0;
    for (int m : masks)
      for (int j = 0; j < 40; ++j) {
        int dirs = 0;
        for (int mu = 0; mu < 4; ++mu) dirs |= (h.site_d[j][mu] != 0) << mu;
        if (dirs != m) continue;
        t.j[i] = j;
        t.a[i] = h.a[j];
        for (int mu = 0; mu < 4; ++mu) {
          t.d[i][mu] = h.site_d[j][mu];
          t.c[i][mu] = -sgn * h.cs[j][mu];
        }
        ++i;
      }
    return t;
  };
  static const PairHops<R> t0 = make((R)1), t1 = make((R)-1);
  return dagger ? t1 : t0;
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
