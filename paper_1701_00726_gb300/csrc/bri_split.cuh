// Brillouin stencil with the 40 hop pairs of a site split over a block's
// groups of threads (spinors in their own layout, FP64 or FP32):
// S sites x G groups, group k takes the offsets k, k + G, ...; the groups' sums
// meet in shared memory, where one thread per site and spinor component adds
// the diagonal and clover terms (and the solver's epilogue).
//
// FP64 runs it at every size: the FP64 pipe (1/64 of the FP32 rate) is busy
// with a few warps, so what counts is that every SM gets the same number of
// sites, which blocks of 8..32 sites give where blocks of 128 leave a partly
// filled last wave.  FP32 runs it, in blocks of 8 sites, on lattices too small to
// fill the chip with a thread per site, where the serial chain of 40 gathers per
// thread was the whole time.
#pragma once

#include "hops.cuh"

namespace bri {

// y = D x on the S sites of block blk for one right-hand side (x, y, p0 its
// vectors); EPI: y = D x + sg p0, returns this thread's part of Re<p0, y>.
template <typename R, typename LS, int S, int G, bool EPI>
__device__ __forceinline__ double split_block(const Geom& g, int blk, R* __restrict__ yout, const R* __restrict__ xin,
                                              const LS* __restrict__ W, const R* __restrict__ cl, R diag,
                                              const PairHops<R>& H, const R* __restrict__ p0, R sg) {
  __shared__ R red[G][24][S];
  const int V = (int)g.V;
  {
    const int site = threadIdx.x % S, grp = threadIdx.x / S;
    const int n = min(blk * S + site, V - 1);
    int up[4], dn[4];
    {
      int r = n;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        const int L = g.L[mu], st = (int)g.str[mu];
        const int c = mu < 3 ? r % L : r;
        if (mu < 3) r /= L;
        up[mu] = c == L - 1 ? -(L - 1) * st : st;
        dn[mu] = c == 0 ? (L - 1) * st : -st;
      }
    }
    C<R> acc[3][4];
#pragma unroll
    for (int aa = 0; aa < 3; ++aa)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[aa][q] = C<R>{0, 0};
#pragma unroll 1
    for (int i = grp; i < 40; i += G) {
      const int j = H.j[i];
      int mp = n, mm = n;
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        const int d = H.d[i][mu];
        mp += d > 0 ? up[mu] : (d < 0 ? dn[mu] : 0);
        mm += d > 0 ? dn[mu] : (d < 0 ? up[mu] : 0);
      }
      C<R> w[3][3], wm[3][3];
      Spinor<R> xp, xm;
      load_stored_link<R, LS>(w, W, j, n, V);
      load_spinor(xp, xin + (int64_t)mp * 24);
      load_stored_link<R, LS>(wm, W, j, mm, V);
      load_spinor(xm, xin + (int64_t)mm * 24);
      const R a = H.a[i], a2 = 2 * a;
      // P = w x+, V = wm^dagger x- - P, acc += 2 a P + a V - c G V
      C<R> v[3][4];
#pragma unroll
      for (int aa = 0; aa < 3; ++aa)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          C<R> p = w[aa][0] * xp.v[q][0];
          cfma(p, w[aa][1], xp.v[q][1]);
          cfma(p, w[aa][2], xp.v[q][2]);
          acc[aa][q].re = fma(a2, p.re, acc[aa][q].re);
          acc[aa][q].im = fma(a2, p.im, acc[aa][q].im);
          v[aa][q] = C<R>{-p.re, -p.im};
        }
#pragma unroll
      for (int aa = 0; aa < 3; ++aa)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          cfma_cj(v[aa][q], wm[0][aa], xm.v[q][0]);
          cfma_cj(v[aa][q], wm[1][aa], xm.v[q][1]);
          cfma_cj(v[aa][q], wm[2][aa], xm.v[q][2]);
          acc[aa][q].re = fma(a, v[aa][q].re, acc[aa][q].re);
          acc[aa][q].im = fma(a, v[aa][q].im, acc[aa][q].im);
        }
      // gamma terms of vanishing weight are skipped (uniform within a group,
      // and nearly so within a warp, see pair_hops)
      const R c1 = H.c[i][0], c2 = H.c[i][1], c3 = H.c[i][2], c4 = H.c[i][3];
      if (c1 != (R)0)
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) gamma_term<1>(acc[aa], v[aa], c1);
      if (c2 != (R)0)
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) gamma_term<2>(acc[aa], v[aa], c2);
      if (c3 != (R)0)
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) gamma_term<3>(acc[aa], v[aa], c3);
      if (c4 != (R)0)
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) gamma_term<4>(acc[aa], v[aa], c4);
    }
#pragma unroll
    for (int aa = 0; aa < 3; ++aa)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        red[grp][2 * (q * 3 + aa)][site] = acc[aa][q].re;
        red[grp][2 * (q * 3 + aa) + 1][site] = acc[aa][q].im;
      }
  }
  __syncthreads();
  double dot = 0.0;
  for (int i = threadIdx.x; i < 12 * S; i += S * G) {
    const int site = i % S, e = i / S;  // component e = 3 spin + colour
    const int n = blk * S + site;
    if (n >= V) continue;
    C<R> o{0, 0};
#pragma unroll
    for (int k = 0; k < G; ++k) {
      o.re += red[k][2 * e][site];
      o.im += red[k][2 * e + 1][site];
    }
    const C<R>* xn = reinterpret_cast<const C<R>*>(xin + (int64_t)n * 24);
    const C<R> xe = xn[e];
    o.re = fma(diag, xe.re, o.re);
    o.im = fma(diag, xe.im, o.im);
    if (cl) {  // row of the packed Hermitian 6x6 block (clover_block)
      const int h = e / 6, row = e - 6 * h;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const C<R> xk = xn[6 * h + k];
        if (k == row) {
          const R d = clover_real(cl, V, n, h, k);
          o.re = fma(d, xk.re, o.re);
          o.im = fma(d, xk.im, o.im);
        } else {
          const int i0 = min(k, row), j0 = max(k, row);
          const int at = 6 + 2 * (i0 * 5 - i0 * (i0 - 1) / 2 + j0 - i0 - 1);
          C<R> cij{clover_real(cl, V, n, h, at), clover_real(cl, V, n, h, at + 1)};
          if (k < row) cij.im = -cij.im;
          cfma(o, cij, xk);
        }
      }
    }
    const int64_t at = (int64_t)n * 24 + 2 * e;
    if constexpr (EPI) {
      const C<R> p = *reinterpret_cast<const C<R>*>(p0 + at);
      o.re = fma(sg, p.re, o.re);
      o.im = fma(sg, p.im, o.im);
      dot += (double)fma(p.re, o.re, p.im * o.im);
    }
    *reinterpret_cast<C<R>*>(yout + at) = o;
  }
  return dot;
}

template <typename R, typename LS, int S, int G, bool EPI>
__global__ void __launch_bounds__(S* G, sizeof(R) == 8 ? 2 : 3)
    bri_split_kernel(Geom g, R* __restrict__ y, const R* __restrict__ x, const LS* __restrict__ W,
                     const R* __restrict__ cl, R diag, int gfirst, const __grid_constant__ PairHops<R> H,
                     ShiftDot<R> sd) {
  const int s = gfirst ? blockIdx.x : blockIdx.y, blk = gfirst ? blockIdx.y : blockIdx.x;
  const int64_t o = s * (g.V * 24);
  double dot = split_block<R, LS, S, G, EPI>(g, blk, y + o, x + o, W, cl, diag, H, EPI ? sd.p + o : nullptr,
                                             EPI ? (R)sd.sig[s] : (R)0);
  if constexpr (EPI) {
    __shared__ double sh[(S * G + 31) / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = dot;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < S * G / 32; ++k) t += sh[k];
      sd.part[(int64_t)s * (gfirst ? gridDim.y : gridDim.x) + blk] = t;
    }
  }
}

template <typename R, typename LS, int S, int G>
inline void launch_split_sg(const Geom& g, R* y, const R* x, const LS* W, const R* cl, R diag, int dagger, int nrhs,
                            cudaStream_t st, const ShiftDot<R>* sd) {
  const StencilGrid sg = stencil_grid(blocks_for(g.V, S), nrhs);
  if (sd)
    bri_split_kernel<R, LS, S, G, true><<<sg.grid, S * G, 0, st>>>(g, y, x, W, cl, diag, sg.gfirst, pair_hops<R>(dagger), *sd);
  else
    bri_split_kernel<R, LS, S, G, false><<<sg.grid, S * G, 0, st>>>(g, y, x, W, cl, diag, sg.gfirst, pair_hops<R>(dagger),
                                                                   ShiftDot<R>{nullptr, nullptr, nullptr});
  note_launch();
}

// Sites per block: 32 while that still gives every SM several blocks, else 16 or 8.
inline int split_sites(int64_t site_rhs) {
  constexpr int64_t kBlocks = 4 * 152;
  return site_rhs >= 32 * kBlocks ? 32 : (site_rhs >= 16 * kBlocks ? 16 : 8);
}

template <typename R, typename LS>
inline int launch_split(const Geom& g, R* y, const R* x, const LS* W, const R* cl, R diag, int nrhs, int dagger,
                        cudaStream_t st, const ShiftDot<R>* sd, int* sd_blocks) {
  // (FP32 is here for small calls, and for a solve that has no memory for packed vectors)
  const int S = sizeof(R) == 4 ? 8 : split_sites(g.V * nrhs);
  if (sd_blocks) *sd_blocks = blocks_for(g.V, S);
  if constexpr (sizeof(R) == 8) {
    if (S == 32) launch_split_sg<R, LS, 32, 5>(g, y, x, W, cl, diag, dagger, nrhs, st, sd);
    if (S == 16) launch_split_sg<R, LS, 16, 10>(g, y, x, W, cl, diag, dagger, nrhs, st, sd);
  }
  if (S == 8) launch_split_sg<R, LS, 8, 20>(g, y, x, W, cl, diag, dagger, nrhs, st, sd);
  BRI_LAUNCH_CHECK("bri_split_kernel");
  return BRI_OK;
}

}  // namespace bri
