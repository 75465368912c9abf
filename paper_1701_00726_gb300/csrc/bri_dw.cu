// Brillouin stencil in double-word FP32 arithmetic (a value is the unevaluated
// sum h + l of two floats, about 48 significant bits), for FP64-class operator
// applications on the FP32 pipe.  GB300 runs FP64 at 1/64 of its FP32 rate,
// so the FP64 residuals of the mixed-precision scheme are cheaper this way.
//
// Arithmetic, from published error-free transformations:
//  * TwoSum (Knuth, TAOCP vol. 2, 4.2.2; Moller 1965): s + e = a + b exactly,
//    six operations, no ordering condition;
//  * Fast2Sum (Dekker 1971): s + e = a + b exactly when |a| >= |b|;
//  * TwoProduct with a fused multiply-add (Ogita, Rump and Oishi, "Accurate
//    sum and dot product", SIAM J. Sci. Comput. 26 (2005)): p + e = a b exactly;
//  * their Dot2 accumulation: the leading parts of the products are summed by
//    TwoSum, and every rounding error (of the sums and of the products) is
//    collected in a second FP32 word.  With double-word operands the two cross
//    products u_h v_l + u_l v_h join that word too (their own rounding is
//    ~2^-48 of the product).  The accumulators are renormalised by Fast2Sum
//    once per hop pair.
// The products and sums of the transformations are written with the _rn
// intrinsics, which the compiler never contracts into fused operations.
//
// The transformations run on fma/add/mul.rn.f32x2: a word holds the two spins of
// a chirality (A, B), the link elements are broadcast to both, so half of the
// instructions do the same arithmetic and no component is moved between
// registers (bri_pair.cuh has the FP32 form of the same scheme).
//
// The stencil (Eq. def_bril, App. C) takes the two hops of a stored offset
// together, colour transport first:
//   P = W_d(n) x(n+d),  V = W_d(n-d)^dagger x(n-d) - P,
//   acc += 2 a_k P + a_k V - c_k S_d V,   S_d = sum_mu d_mu gamma_mu.
// a_k = -2^{-k-3} is a power of two (exact scaling); c_k = 4^{2-k}/27 is carried
// as a double-word constant.
//
// Storage: spinors as [rhs][V/32][12][32] 16-byte words (re_A, re_B, im_A, im_B),
// rows 0..5 the leading words of (chirality, colour), rows 6..11 the second
// ones; links [V/32][40][9][32] words (re_h, re_l, im_h, im_l); clover
// [V/32][2][36][32] pairs (h, l).
//
// Bound: the FP32 pipe, about 4600 operations per hop pair, site and right-hand
// side (12 per real multiply-add; 2.4 ms for 4 right-hand sides at 16^3 x 32).
// GB300, 16^3 x 32, 4 rhs, with the split and join passes: 4.46 ms with scalar
// arithmetic, spin combination before each of the two transports and strided
// links, 3.28 ms now; error against FP64 1.4e-14 -> 0.96e-14.  12 warps per SM with
// the colour loop unrolled; rolled 3.37 ms, both hops unrolled 3.51 ms
// (instruction fetch), 16 warps 3.42 ms (spills).
#include "stencil.cuh"
#include "bri_pair.cuh"

#include <string>

namespace bri {

namespace {

struct DW {
  float h, l;
};
// two double-word values (A, B): leading and second words
struct DP {
  float2 h, l;
};
struct CDP {
  DP re, im;
};

__device__ __forceinline__ float2 d_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 d_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 d_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 d_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 d_neg(float2 a) { return make_float2(-a.x, -a.y); }

// acc += u v (one Dot2 step with double-word operands)
__device__ __forceinline__ void mac(DP& acc, float2 uh, float2 ul, float2 vh, float2 vl) {
  const float2 p = d_mul(uh, vh);
  const float2 pe = d_fma(uh, vh, d_neg(p));
  const float2 s = d_add(acc.h, p);
  const float2 bb = d_sub(s, acc.h);
  float2 t = d_add(d_sub(acc.h, d_sub(s, bb)), d_sub(p, bb));
  acc.h = s;
  t = d_add(t, pe);
  t = d_fma(uh, vl, t);
  t = d_fma(ul, vh, t);
  acc.l = d_add(acc.l, t);
}
// acc += k t for a factor k of powers of two (the products are exact)
__device__ __forceinline__ void add(DP& acc, const DP& t, float2 k) {
  const float2 s = d_fma(t.h, k, acc.h);
  const float2 bb = d_sub(s, acc.h);
  const float2 e = d_add(d_sub(acc.h, d_sub(s, bb)), d_fma(t.h, k, d_neg(bb)));
  acc.h = s;
  acc.l = d_add(d_fma(t.l, k, acc.l), e);
}
// Fast2Sum
__device__ __forceinline__ void renorm(DP& a) {
  const float2 s = d_add(a.h, a.l);
  a.l = d_sub(a.l, d_sub(s, a.h));
  a.h = s;
}
// TwoSum
__device__ __forceinline__ void finish(DP& a) {
  const float2 s = d_add(a.h, a.l);
  const float2 bb = d_sub(s, a.h);
  a.l = d_add(d_sub(a.h, d_sub(s, bb)), d_sub(a.l, bb));
  a.h = s;
}
__device__ __forceinline__ DP swapped(const DP& a) { return DP{pr_swp(a.h), pr_swp(a.l)}; }
__device__ __forceinline__ DP zero_dp() { return DP{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

// word rows r (leading) and r + 6 (second) of a packed spinor
__device__ __forceinline__ CDP ld_cdp(const float4* __restrict__ x, int r) {
  const float4 h = __ldg(x + r * kPackBlock), l = __ldg(x + (r + 6) * kPackBlock);
  return CDP{DP{make_float2(h.x, h.y), make_float2(l.x, l.y)}, DP{make_float2(h.z, h.w), make_float2(l.z, l.w)}};
}
// acc += w v, w = (re_h, re_l, im_h, im_l)
__device__ __forceinline__ void cmac(CDP& acc, const float4& w, const CDP& v) {
  const float2 rh = pr_bc(w.x), rl = pr_bc(w.y), ih = pr_bc(w.z), il = pr_bc(w.w);
  mac(acc.re, rh, rl, v.re.h, v.re.l);
  mac(acc.im, rh, rl, v.im.h, v.im.l);
  mac(acc.re, d_neg(ih), d_neg(il), v.im.h, v.im.l);
  mac(acc.im, ih, il, v.re.h, v.re.l);
}

// Per-offset constants: signs, a_k (exact in FP32), c_k as a double-word pair.
struct HopTableDW {
  int d[40][4];
  float a[40];
  float ch[40], cl[40];
};

const HopTableDW& hop_table_dw() {
  static const HopTableDW t = [] {
    const HopTable<double>& h = hop_table<double>();
    HopTableDW t;
    for (int j = 0; j < 40; ++j) {
      double c = 0.0;
      for (int mu = 0; mu < 4; ++mu) {
        t.d[j][mu] = h.site_d[j][mu];
        if (h.cs[j][mu] != 0.0) c = h.cs[j][mu] > 0 ? h.cs[j][mu] : -h.cs[j][mu];
      }
      t.a[j] = (float)h.a[j];
      t.ch[j] = (float)c;
      t.cl[j] = (float)(c - (double)t.ch[j]);
    }
    return t;
  }();
  return t;
}

constexpr int kDwLinkWords = 9 * kLinkBlock;  // one offset of one block of sites

// One thread per site and right-hand side (grid groups = right-hand sides, in
// the order of stencil_grid), or KS groups of threads that share a site's offsets
// and meet in shared memory, where the first two finish one chirality each.  The
// hop loop is rolled so that the body fits the instruction cache.
template <int KS>
__global__ void __launch_bounds__(128, 3)
    bri_kernel_dw(Geom g, float4* __restrict__ y, const float4* __restrict__ x, const float4* __restrict__ W,
                  const float2* __restrict__ cl, DW diag, float sgn, int gfirst, const __grid_constant__ HopTableDW H) {
  const int grp = gfirst ? blockIdx.x : blockIdx.y, blk = gfirst ? blockIdx.y : blockIdx.x;
  constexpr int SB = 128 / KS;
  const int n0 = blk * SB + threadIdx.x % SB;
  if (KS == 1 && n0 >= g.V) return;
  const int n = KS == 1 ? n0 : min(n0, (int)g.V - 1), ksg = KS == 1 ? 0 : threadIdx.x / SB;
  const int64_t roff = (int64_t)grp * packed_words(g.V, 12);
  const float4* xin = x + roff;
  int up[4], dn[4];
  {
    int r = n;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int L = g.L[mu], s = (int)g.str[mu];
      const int c = mu < 3 ? r % L : r;
      if (mu < 3) r /= L;
      up[mu] = c == L - 1 ? -(L - 1) * s : s;
      dn[mu] = c == 0 ? (L - 1) * s : -s;
    }
  }
  CDP acc[2][3];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) acc[q][aa] = CDP{zero_dp(), zero_dp()};

#pragma unroll 1
  for (int j = ksg; j < 40; j += KS) {
    int mp = n, mm = n;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int d = H.d[j][mu];
      mp += d > 0 ? up[mu] : (d < 0 ? dn[mu] : 0);
      mm += d > 0 ? dn[mu] : (d < 0 ? up[mu] : 0);
    }
    const float a = H.a[j];
    CDP P[2][3];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) P[q][aa] = CDP{zero_dp(), zero_dp()};
    // hop 0: P = W_d(n) x(n+d); hop 1: V = W_d(n-d)^dagger x(n-d) - P (conj(w) = (w_re, -w_im))
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      const int m = h ? mm : n;
      const float4* wp = W + ((int64_t)(m / kLinkBlock) * 40 + j) * kDwLinkWords + m % kLinkBlock;
      const float4* xs = xin + packed_at<12>(h ? mm : mp);
      const float cs = h ? -1.f : 1.f;
      const int wb = (h ? 3 : 1) * kLinkBlock, wa = (h ? 1 : 3) * kLinkBlock;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const CDP x0 = ld_cdp(xs, b), x1 = ld_cdp(xs, 3 + b);
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) {
          float4 w = __ldg(wp + b * wb + aa * wa);
          w.z *= cs;
          w.w *= cs;
          cmac(P[0][aa], w, x0);
          cmac(P[1][aa], w, x1);
        }
      }
      // acc += 2 a P and P -> -P (hop 0), acc += a V (hop 1)
      const float2 k = pr_bc(h ? a : 2.f * a), f = pr_bc(-cs);
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) {
          add(acc[q][aa].re, P[q][aa].re, k);
          add(acc[q][aa].im, P[q][aa].im, k);
          P[q][aa].re = DP{d_mul(P[q][aa].re.h, f), d_mul(P[q][aa].re.l, f)};
          P[q][aa].im = DP{d_mul(P[q][aa].im.h, f), d_mul(P[q][aa].im.l, f)};
        }
    }
    // V times c_k, then the signed spin permutations of -S_d (bri_pair.cuh)
    const float2 ch = pr_bc(H.ch[j]), clo = pr_bc(H.cl[j]);
    auto scale = [&](DP& v) {
      const float2 h = d_mul(v.h, ch);
      float2 e = d_fma(v.h, ch, d_neg(h));
      e = d_fma(v.l, ch, e);
      v.l = d_fma(v.h, clo, e);
      v.h = h;
    };
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        scale(P[q][aa].re);
        scale(P[q][aa].im);
      }
    const float s1 = -sgn * (float)H.d[j][0], s2 = -sgn * (float)H.d[j][1], s3 = -sgn * (float)H.d[j][2], s4 = -sgn * (float)H.d[j][3];
    if (s1 != 0.f) {
      const float2 p = pr_bc(s1), m = pr_bc(-s1);
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        add(acc[0][aa].re, swapped(P[1][aa].im), p);
        add(acc[0][aa].im, swapped(P[1][aa].re), m);
        add(acc[1][aa].re, swapped(P[0][aa].im), m);
        add(acc[1][aa].im, swapped(P[0][aa].re), p);
      }
    }
    if (s2 != 0.f) {
      const float2 k = make_float2(-s2, s2), m = make_float2(s2, -s2);
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        add(acc[0][aa].re, swapped(P[1][aa].re), k);
        add(acc[0][aa].im, swapped(P[1][aa].im), k);
        add(acc[1][aa].re, swapped(P[0][aa].re), m);
        add(acc[1][aa].im, swapped(P[0][aa].im), m);
      }
    }
    if (s3 != 0.f) {
      const float2 k = make_float2(s3, -s3), m = make_float2(-s3, s3);
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        add(acc[0][aa].re, P[1][aa].im, k);
        add(acc[0][aa].im, P[1][aa].re, m);
        add(acc[1][aa].re, P[0][aa].im, m);
        add(acc[1][aa].im, P[0][aa].re, k);
      }
    }
    if (s4 != 0.f) {
      const float2 k = pr_bc(s4);
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        add(acc[0][aa].re, P[1][aa].re, k);
        add(acc[0][aa].im, P[1][aa].im, k);
        add(acc[1][aa].re, P[0][aa].re, k);
        add(acc[1][aa].im, P[0][aa].im, k);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        renorm(acc[q][aa].re);
        renorm(acc[q][aa].im);
      }
  }
  if constexpr (KS > 1) {
    __shared__ float4 red[KS][12][SB];
    const int l = threadIdx.x % SB;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const CDP& v = acc[i / 3][i % 3];
      red[ksg][2 * i][l] = make_float4(v.re.h.x, v.re.h.y, v.re.l.x, v.re.l.y);
      red[ksg][2 * i + 1][l] = make_float4(v.im.h.x, v.im.h.y, v.im.l.x, v.im.l.y);
    }
    __syncthreads();
    if (ksg >= 2 || n0 >= g.V) return;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      CDP t{zero_dp(), zero_dp()};
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        const float4 r = red[k][6 * ksg + 2 * i][l], m = red[k][6 * ksg + 2 * i + 1][l];
        add(t.re, DP{make_float2(r.x, r.y), make_float2(r.z, r.w)}, pr_bc(1.f));
        add(t.im, DP{make_float2(m.x, m.y), make_float2(m.z, m.w)}, pr_bc(1.f));
      }
      renorm(t.re);
      renorm(t.im);
      acc[0][i] = t;  // this group's chirality, whichever it is
      acc[1][i] = t;
    }
  }
  // diagonal and clover terms at the site itself.  A chirality's clover block is
  // [[X, M], [M^dagger, -X]] on its two spins: X (3 reals, 3 complex above the
  // diagonal) acts with the signs (+, -), M and M^dagger on the exchanged spins.
  const float4* xo = xin + packed_at<12>(n);
  float4* yo = y + roff + packed_at<12>(n);
  const float2 dh = pr_bc(diag.h), dl = pr_bc(diag.l);
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (KS > 1 && q != ksg) continue;
    CDP in[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      in[b] = ld_cdp(xo, 3 * q + b);
      mac(acc[q][b].re, dh, dl, in[b].re.h, in[b].re.l);
      mac(acc[q][b].im, dh, dl, in[b].im.h, in[b].im.l);
    }
    if (cl) {
      const float2* cb = cl + ((int64_t)(n / kCloverBlock * 2 + q) * 36) * kCloverBlock + n % kCloverBlock;
      auto real = [&](int k) { return __ldg(cb + k * kCloverBlock); };
      auto at = [](int i, int j) { return 6 + 2 * (i * 5 - i * (i - 1) / 2 + j - i - 1); };
      const float2 pm = make_float2(1.f, -1.f);
      // (+-) X: entry (a, b) as a complex double-word number, conjugated below the diagonal
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        CDP v = in[b];  // signs (+, -) on the two spins
        v.re = DP{d_mul(v.re.h, pm), d_mul(v.re.l, pm)};
        v.im = DP{d_mul(v.im.h, pm), d_mul(v.im.l, pm)};
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) {
          if (aa == b) {
            const float2 d = real(aa);
            mac(acc[q][aa].re, pr_bc(d.x), pr_bc(d.y), v.re.h, v.re.l);
            mac(acc[q][aa].im, pr_bc(d.x), pr_bc(d.y), v.im.h, v.im.l);
          } else {
            const int k = aa < b ? at(aa, b) : at(b, aa);
            const float2 r = real(k), i = real(k + 1);
            const float sg = aa < b ? 1.f : -1.f;
            cmac(acc[q][aa], make_float4(r.x, r.y, sg * i.x, sg * i.y), v);
          }
        }
      }
      // out_A += M in_B, out_B += M^dagger in_A: pair operands (M[aa][b], conj M[b][aa])
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const DP vr = swapped(in[b].re), vi = swapped(in[b].im);
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) {
          const float2 ra = real(at(aa, 3 + b)), ia = real(at(aa, 3 + b) + 1);
          const float2 rb = real(at(b, 3 + aa)), ib = real(at(b, 3 + aa) + 1);
          const float2 rh = make_float2(ra.x, rb.x), rl = make_float2(ra.y, rb.y);
          const float2 ih = make_float2(ia.x, -ib.x), il = make_float2(ia.y, -ib.y);
          mac(acc[q][aa].re, rh, rl, vr.h, vr.l);
          mac(acc[q][aa].im, rh, rl, vi.h, vi.l);
          mac(acc[q][aa].re, d_neg(ih), d_neg(il), vi.h, vi.l);
          mac(acc[q][aa].im, ih, il, vr.h, vr.l);
        }
      }
    }
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) {
      CDP o = acc[q][aa];
      finish(o.re);
      finish(o.im);
      yo[(3 * q + aa) * kPackBlock] = make_float4(o.re.h.x, o.re.h.y, o.im.h.x, o.im.h.y);
      yo[(3 * q + aa + 6) * kPackBlock] = make_float4(o.re.l.x, o.re.l.y, o.im.l.x, o.im.l.y);
    }
  }
}

__device__ __forceinline__ float2 split_dw(double v) {
  const float h = __double2float_rn(v);
  return make_float2(h, __double2float_rn(v - (double)h));
}

// FP64 spinors [rhs][V][12] -> packed double-word spinors and back; one thread
// per site, chirality and colour, blockIdx.y = right-hand side.
__global__ void __launch_bounds__(256) k_split_dw(int64_t V, const double2* __restrict__ in, float4* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V * 6) return;
  const int64_t n = i / 6;
  const int q = (int)(i - n * 6);
  const double2* p = in + (blockIdx.y * V + n) * 12 + q + 3 * (q / 3);
  const double2 u = __ldg(p), v = __ldg(p + 3);
  const float2 ur = split_dw(u.x), ui = split_dw(u.y), vr = split_dw(v.x), vi = split_dw(v.y);
  float4* o = out + (int64_t)blockIdx.y * packed_words(V, 12) + packed_at<12>((int)n) + q * kPackBlock;
  o[0] = make_float4(ur.x, vr.x, ui.x, vi.x);
  o[6 * kPackBlock] = make_float4(ur.y, vr.y, ui.y, vi.y);
}
__global__ void __launch_bounds__(256) k_join_dw(int64_t V, const float4* __restrict__ in, double2* __restrict__ out) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V * 6) return;
  const int64_t n = i / 6;
  const int q = (int)(i - n * 6);
  const float4* o = in + (int64_t)blockIdx.y * packed_words(V, 12) + packed_at<12>((int)n) + q * kPackBlock;
  const float4 h = __ldg(o), l = __ldg(o + 6 * kPackBlock);
  double2* p = out + (blockIdx.y * V + n) * 12 + q + 3 * (q / 3);
  p[0] = make_double2((double)h.x + (double)l.x, (double)h.z + (double)l.z);
  p[3] = make_double2((double)h.y + (double)l.y, (double)h.w + (double)l.w);
}
// FP64 links [40][9][V] and clover [2][36][V] into the chunked double-word
// layouts, one thread per element and site.
__global__ void __launch_bounds__(256) k_links_dw(int64_t V, const double2* __restrict__ in, float4* __restrict__ out) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= V) return;
  const int je = blockIdx.y;
  const double2 v = in[(int64_t)je * V + n];
  const float2 r = split_dw(v.x), m = split_dw(v.y);
  out[(n / kLinkBlock * 360 + je) * kLinkBlock + n % kLinkBlock] = make_float4(r.x, r.y, m.x, m.y);
}
__global__ void __launch_bounds__(256) k_clover_dw(int64_t V, const double* __restrict__ in, float2* __restrict__ out) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= V) return;
  out[(n / kCloverBlock * 72 + blockIdx.y) * kCloverBlock + n % kCloverBlock] = split_dw(in[(int64_t)blockIdx.y * V + n]);
}

}  // namespace

size_t dw_vector_bytes(int64_t V) { return sizeof(float4) * (size_t)packed_words(V, 12); }

// Double-word copies of the FP64 links and clover, made on first use after
// each bri_build_links.
int ensure_dw_links(bri_ctx* c) {
  if (c->dw_valid) return BRI_OK;
  const int64_t V = c->g.V;
  cudaStream_t st = c->stream;
  auto alloc = [&](void** p, size_t bytes) -> int {
    if (*p) return BRI_OK;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error(std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
      return BRI_ERR_OOM;
    }
    note_device_alloc();
    return BRI_OK;
  };
  int rc;
  const int64_t Vp = link_blocks(V) * kLinkBlock;
  if ((rc = alloc(&c->Wdw, sizeof(float4) * 360 * Vp))) return rc;
  k_links_dw<<<dim3(blocks_for(V, 256), 360), 256, 0, st>>>(V, c->W64, (float4*)c->Wdw); note_launch();
  if (c->have_clover) {
    if ((rc = alloc(&c->Cdw, sizeof(float2) * 72 * Vp))) return rc;
    k_clover_dw<<<dim3(blocks_for(V, 256), 72), 256, 0, st>>>(V, c->C64, (float2*)c->Cdw); note_launch();
  }
  BRI_LAUNCH_CHECK("double-word links");
  c->dw_valid = true;
  return BRI_OK;
}

// Four groups of threads per site until one thread per site fills several waves.
// GB300, us with one group / four (conversions included): 8^4 x 1 rhs 158 / 56, 8^3.16
// x 1 162 / 84, 12^4 x 1 296 / 195, 16^4 x 1 567 / 489, 8^3.16 x 12 739 / 662, 16^4 x 2
// 911 / 884, 16^3.32 x 2 1749 / 1711, x 4 3289 / 3315.
static int dw_groups(int64_t site_rhs) { return site_rhs <= 393216 ? 4 : 1; }

// y = D x or D^dagger x on double-word vectors (Brillouin kernel).
int dirac_bri_dw(bri_ctx* c, void* y, const void* x, int nrhs, double m0, int dagger, cudaStream_t s) {
  int rc = ensure_dw_links(c);
  if (rc) return rc;
  const double dg = 15.0 / 8.0 + m0;
  DW diag;
  diag.h = (float)dg;
  diag.l = (float)(dg - (double)diag.h);
  const int ks = dw_groups(c->g.V * nrhs);
  const StencilGrid sg = stencil_grid(blocks_for(c->g.V, 128 / ks), nrhs);
  auto run = [&](auto kernel) {
    kernel<<<sg.grid, 128, 0, s>>>(c->g, (float4*)y, (const float4*)x, (const float4*)c->Wdw,
                                   c->have_clover ? (const float2*)c->Cdw : nullptr, diag, dagger ? -1.f : 1.f, sg.gfirst,
                                   hop_table_dw());
  };
  if (ks == 4) run(bri_kernel_dw<4>);
  else run(bri_kernel_dw<1>);
  note_launch();
  BRI_LAUNCH_CHECK("bri_kernel_dw");
  return BRI_OK;
}

// FP64 in, FP64 out: split, stencil, join (tmp: two double-word vectors of
// nrhs right-hand sides).
int dirac_bri_dw64(bri_ctx* c, double* y, const double* x, int nrhs, double m0, int dagger, void* tmp,
                   cudaStream_t s) {
  const int64_t V = c->g.V;
  const dim3 eg(blocks_for(V * 6, 256), nrhs);
  float4* xa = (float4*)tmp;
  float4* ya = xa + packed_words(V, 12) * nrhs;
  k_split_dw<<<eg, 256, 0, s>>>(V, (const double2*)x, xa); note_launch();
  int rc = dirac_bri_dw(c, ya, xa, nrhs, m0, dagger, s);
  if (rc) return rc;
  k_join_dw<<<eg, 256, 0, s>>>(V, ya, (double2*)y); note_launch();
  BRI_LAUNCH_CHECK("double-word apply");
  return BRI_OK;
}

// A x = D^dagger D x on FP64 vectors through double-word stencils; out = A x
// (FP64).  t1, t2: double-word scratch of nrhs vectors each.
int normal_op_dw(bri_ctx* c, double* out, const double* x, int nrhs, double m0, void* t1, void* t2, cudaStream_t s) {
  const int64_t V = c->g.V;
  const dim3 eg(blocks_for(V * 6, 256), nrhs);
  k_split_dw<<<eg, 256, 0, s>>>(V, (const double2*)x, (float4*)t1); note_launch();
  int rc = dirac_bri_dw(c, t2, t1, nrhs, m0, 0, s);
  if (rc) return rc;
  rc = dirac_bri_dw(c, t1, t2, nrhs, m0, 1, s);
  if (rc) return rc;
  k_join_dw<<<eg, 256, 0, s>>>(V, (const float4*)t1, (double2*)out); note_launch();
  BRI_LAUNCH_CHECK("double-word normal operator");
  return BRI_OK;
}

}  // namespace bri
