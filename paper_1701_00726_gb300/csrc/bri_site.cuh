// The Brillouin stencil at one site for NR right-hand sides (CUDA cores, scalar
// FMAs), templated on spinor precision R and link storage LS: the per-site
// function of the batched work-list kernel, whose right-hand sides belong to
// lattices of different volume.
//
// D_bri x(n) = sum_{d != 0} W_d(n) M_d x(n+d) + (15/8 + m0) x(n) + C(n) x(n)   (Eq. def_bril)
//   M_d = -2^{-k-3} 1 + (4^{2-k}/27) sum_{mu: d_mu != 0} sign(d_mu) gamma_mu,  k = |d|_1
// (the momentum forms of App. A expanded into plane waves).  D^dagger = gamma5 D
// gamma5 only flips the sign of the gamma part.
//
// A runtime loop visits the 40 stored offsets d (nu = 1..40 of App. C); each
// iteration also handles the opposite hop -d, whose transporter is the stored
// link of d at the neighbour n-d, daggered (W_{82-nu}(n) = W_nu(n-d)^dagger).
// Both hops of a pair have the same weights a_k, c_k and spin matrix G = sum_mu
// s_mu gamma_mu up to the sign of G, so the two source spinors are
// colour-transported first (P = W x(n+d), Q = W'^dagger x(n-d), Q accumulated
// onto P) and the spin structure is applied once: acc += a_k (P + Q) + c_k G (P
// - Q), with P - Q = 2P - (P + Q).  The FP64 instance skips the gamma terms
// whose s_mu vanishes.  The loop is not unrolled so that the compiler does not
// hoist loads across hops, which keeps the live register set bounded.
#pragma once

#include "hops.cuh"

namespace bri {

// One hop pair (stored offset d and its opposite) for NR right-hand sides:
// acc += a (P + Q) + c G (P - Q) with P = W_d(n) x(n+d), Q = W_d(n-d)^dagger x(n-d),
// G = sum_mu s_mu gamma_mu, both links already in registers (w = W_d(n),
// wm = W_d(n-d)); mp, mm are the sites n+d and n-d.
template <typename R, int NR>
__device__ __forceinline__ void bri_pair(Spinor<R> (&acc)[NR], const R* __restrict__ xin, int64_t rstride, int mp,
                                         int mm, const C<R> (&w)[3][3], const C<R> (&wm)[3][3], R a, R c1, R c2,
                                         R c3, R c4) {
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    Spinor<R> xp, xm;
    load_spinor(xp, xin + r * rstride + (int64_t)mp * 24);
    load_spinor(xm, xin + r * rstride + (int64_t)mm * 24);
    // u = P + Q (Q accumulated onto P), vn = u - 2P = -(P - Q): the gamma
    // part takes vn with negated weights.
    if constexpr (sizeof(R) == 8) {
      // FP64 is bound by the FP64 pipe: gamma terms whose weight vanishes
      // (s_mu = 0 for 4 - k of the four directions) are skipped with
      // branches that are uniform across the grid.
      C<R> vn[3][4];
#pragma unroll
      for (int aa = 0; aa < 3; ++aa)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          C<R> p = w[aa][0] * xp.v[s][0];
          cfma(p, w[aa][1], xp.v[s][1]);
          cfma(p, w[aa][2], xp.v[s][2]);
          C<R> q = p;
          cfma_cj(q, wm[0][aa], xm.v[s][0]);
          cfma_cj(q, wm[1][aa], xm.v[s][1]);
          cfma_cj(q, wm[2][aa], xm.v[s][2]);
          acc[r].v[s][aa].re = fma(a, q.re, acc[r].v[s][aa].re);
          acc[r].v[s][aa].im = fma(a, q.im, acc[r].v[s][aa].im);
          vn[aa][s] = C<R>{fma((R)-2, p.re, q.re), fma((R)-2, p.im, q.im)};
        }
      const R cn[4] = {-c1, -c2, -c3, -c4};
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        C<R> col[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) col[s] = acc[r].v[s][aa];
        if (cn[0] != (R)0) gamma_term<1>(col, vn[aa], cn[0]);
        if (cn[1] != (R)0) gamma_term<2>(col, vn[aa], cn[1]);
        if (cn[2] != (R)0) gamma_term<3>(col, vn[aa], cn[2]);
        if (cn[3] != (R)0) gamma_term<4>(col, vn[aa], cn[3]);
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[r].v[s][aa] = col[s];
      }
    } else {
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        C<R> u[4], vn[4], col[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          C<R> p = w[aa][0] * xp.v[s][0];
          cfma(p, w[aa][1], xp.v[s][1]);
          cfma(p, w[aa][2], xp.v[s][2]);
          C<R> q = p;
          cfma_cj(q, wm[0][aa], xm.v[s][0]);
          cfma_cj(q, wm[1][aa], xm.v[s][1]);
          cfma_cj(q, wm[2][aa], xm.v[s][2]);
          u[s] = q;
          vn[s] = C<R>{fma((R)-2, p.re, q.re), fma((R)-2, p.im, q.im)};
          col[s] = acc[r].v[s][aa];
        }
        add_pair_terms(col, u, vn, a, -c1, -c2, -c3, -c4);
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[r].v[s][aa] = col[s];
      }
    }
  }
}

// The stencil at one site n for NR right-hand sides: xin and yout point at
// the first right-hand side, the others follow at xstride (input) and ystride
// (output) reals.
template <typename R, typename LS, int NR>
__device__ __forceinline__ void bri_site(const Geom& g, int n, R* __restrict__ yout, const R* __restrict__ xin,
                                         int64_t xstride, int64_t ystride, const LS* __restrict__ W,
                                         const R* __restrict__ cl, R diag, R sgn, const HopTable<R>& H) {
  const int V = (int)g.V;
  int co[4], L[4], str[4];
  {
    int r = n;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
      co[mu] = r % g.L[mu];
      r /= g.L[mu];
    }
    co[3] = r;
  }
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    L[mu] = g.L[mu];
    str[mu] = (int)g.str[mu];
  }
  Spinor<R> acc[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) zero(acc[r]);
  auto sites = [&](int j, int& mp, int& mm) {
    mp = 0;
    mm = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int d = H.site_d[j][mu];
      mp += wrap(co[mu] + d, L[mu]) * str[mu];
      mm += wrap(co[mu] - d, L[mu]) * str[mu];
    }
  };
  // The pair of opposite hops shares a, c and G = sum_mu s_mu gamma_mu:
  //   W x+ M_d + W'^dagger M_{-d} x- = a (P + Q) + c G (P - Q),
  //   P = W_d(n) x(n+d),  Q = W_d(n-d)^dagger x(n-d)   (M_{+-d} = a +- c G).
  // both links and both source spinors are loaded before any arithmetic, so
  // one memory latency is exposed per pair of hops
#pragma unroll 1
  for (int j = 0; j < 40; ++j) {
    int mp, mm;
    sites(j, mp, mm);
    C<R> w[3][3], wm[3][3];
    load_stored_link<R, LS>(w, W, j, n, V);
    load_stored_link<R, LS>(wm, W, j, mm, V);
    bri_pair<R, NR>(acc, xin, xstride, mp, mm, w, wm, H.a[j], sgn * H.cs[j][0], sgn * H.cs[j][1],
                    sgn * H.cs[j][2], sgn * H.cs[j][3]);
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    Spinor<R> xc;
    load_spinor(xc, xin + r * xstride + (int64_t)n * 24);
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        acc[r].v[s][aa].re = fma(diag, xc.v[s][aa].re, acc[r].v[s][aa].re);
        acc[r].v[s][aa].im = fma(diag, xc.v[s][aa].im, acc[r].v[s][aa].im);
      }
    if (cl) add_clover(acc[r], xc, cl, g.V, n);
    store_spinor(yout + r * ystride + (int64_t)n * 24, acc[r]);
  }
}

}  // namespace bri
