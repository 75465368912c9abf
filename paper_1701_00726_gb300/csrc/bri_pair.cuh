// Brillouin stencil on packed FP32 spinors: every 16-byte word holds one
// complex number of two spinor components, (re_A, re_B, im_A, im_B), so that
// fma.rn.f32x2 works on two components at a time with the link element
// broadcast to both halves (a free operand form), a factor i only exchanges the
// re and im registers (signs go into the scalar weights), and no register pair
// has to be built or rotated.
//
//   two right-hand sides (RP): A, B = the two right-hand sides of a pair,
//       [group][V/32][12][32] words, row 3 s + c (spin s, colour c);
//   one right-hand side (SP):  A, B = the two spins of a chirality,
//       [rhs][V/32][6][32] words, row 3 h + c (chirality h, colour c).
//
// A warp of 32 consecutive sites reads whole 512-byte rows without bank
// conflicts at immediate offsets from one address (the array-of-structs spinor
// costs a 96-byte stride: 1.7x the L1 wavefronts).
//
// D_bri x(n) = sum_{d != 0} W_d(n) M_d x(n+d) + (15/8 + m0) x(n) + C(n) x(n)   (Eq. def_bril, App. C)
//
// Per stored offset d the two opposite hops are taken together, in place:
//   P = W_d(n) x(n+d),  V = W_d(n-d)^dagger x(n-d) - P,
//   acc += 2 a_k P + a_k V - c_k sum_mu s_mu gamma_mu V
// (a_k (P + Q) + c_k G (P - Q) with Q = V + P), so one colour-transported
// spinor is live besides the accumulator.  The next offset's links are loaded
// into the registers of the present ones as soon as those are dead.
//
// Bound: the FP32 pipe (432 paired FMAs per hop pair and pair of right-hand
// sides; 71 % busy at 16^3 x 32, L1 46 %, DRAM 19 %), for one right-hand side
// at 24^3 x 48 also the link stream.  GB300, packing pass included, against the
// kernels before it (array-of-structs spinors, links as five strided streams):
// 16^3 x 32, 12 rhs 1208 -> 1015 us; 24^3 x 48, 1 rhs 653 -> 560 us; BF16
// links, 18.15.14.21, 3 rhs 278 -> 178 us (237 with one thread group per site).  Two right-hand sides per thread run
// at 12 warps per SM (168 registers), one at 16 (128); more warps with spills
// were slower (0.80 against 0.62 ns per site and rhs), as were blocks that
// stage a 4D tile and its halo in shared memory (0.78: filling the halo takes
// longer than the gathers it saves), branches around vanishing gamma terms
// (0.71 against 0.65) and sites numbered by 4D tiles (0.69: rows of 8 sites
// straddle more lines).
#pragma once

#include "hops.cuh"
#include "sum3.cuh"

namespace bri {

__device__ __forceinline__ float2 pr_bc(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 pr_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pr_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pr_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 pr_swp(float2 a) { return make_float2(a.y, a.x); }

// One complex number of the two components of a word.
struct CP {
  float2 re, im;
};
__device__ __forceinline__ CP cp_of(const float4& v) { return CP{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 cp_word(const CP& v) { return make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }
// o += c v, o += i c v
__device__ __forceinline__ void cp_add(CP& o, const CP& v, float c) {
  o.re = pr_fma(v.re, pr_bc(c), o.re);
  o.im = pr_fma(v.im, pr_bc(c), o.im);
}
__device__ __forceinline__ void cp_addi(CP& o, const CP& v, float c) {
  o.re = pr_fma(v.im, pr_bc(-c), o.re);
  o.im = pr_fma(v.re, pr_bc(c), o.im);
}

constexpr int kPackBlock = 32;
// 16-byte words of one group (rows = 12: a pair of right-hand sides, 6: one)
__host__ __device__ __forceinline__ int64_t packed_words(int64_t V, int rows) {
  return (V + kPackBlock - 1) / kPackBlock * kPackBlock * rows;
}
template <int ROWS> __device__ __forceinline__ int packed_at(int m) {
  return (m / kPackBlock) * (ROWS * kPackBlock) + m % kPackBlock;
}

// The words of a spinor in one of two layouts: rows of a block of sites as above, or
// (OWN, single right-hand sides) the caller's 96 bytes of a site, whose spins meet in
// registers.  OWN needs no packed copy of x: 16^3 x 32, 4 and 12 rhs 422 and 1205 us
// against 382 and 1023 with one (packing included), 24^3 x 48, 1 rhs 621 against 565,
// 16^4, 1 rhs 68 against 70; its 16-byte words in order 510 and 1472 us, 3 blocks per SM 446
// and 1291; the split kernel (bri_split.cuh), which needs no copy either, 713 and 2056.
template <int R, bool OWN> struct SpinorWords {
  CP v[R][3];
  // Neighbouring lanes are 96 bytes apart: the lanes with bit 2 set read each pair of
  // words the other way round, so that no two of eight meet in a bank.
  __device__ __forceinline__ void load(const float4* __restrict__ x) {
    if constexpr (OWN) {
      static_assert(R == 2, "single right-hand sides");
      const int odd = (threadIdx.x >> 2) & 1;
      float4 u[6];
#pragma unroll
      for (int i = 0; i < 6; i += 2) {
        const float4 a = __ldg(x + i + odd), b = __ldg(x + i + 1 - odd);
        u[i] = make_float4(odd ? b.x : a.x, odd ? b.y : a.y, odd ? b.z : a.z, odd ? b.w : a.w);
        u[i + 1] = make_float4(odd ? a.x : b.x, odd ? a.y : b.y, odd ? a.z : b.z, odd ? a.w : b.w);
      }
#pragma unroll
      for (int q = 0; q < R; ++q) join(u[3 * q], u[3 * q + 1], u[3 * q + 2], v[q]);
    }
  }
  __device__ __forceinline__ static void join(const float4& a, const float4& b, const float4& c, CP (&o)[3]) {
    o[0] = CP{make_float2(a.x, b.z), make_float2(a.y, b.w)};
    o[1] = CP{make_float2(a.z, c.x), make_float2(a.w, c.y)};
    o[2] = CP{make_float2(b.x, c.z), make_float2(b.y, c.w)};
  }
  __device__ __forceinline__ static void load_half(const float4* __restrict__ x, int q, CP (&o)[3]) {
    if constexpr (OWN) {
      join(__ldg(x + 3 * q), __ldg(x + 3 * q + 1), __ldg(x + 3 * q + 2), o);
    } else {
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) o[aa] = cp_of(__ldg(x + (q * 3 + aa) * kPackBlock));
    }
  }
  __device__ __forceinline__ CP word(const float4* __restrict__ x, int q, int b) const {
    if constexpr (OWN) return v[q][b];
    else return cp_of(__ldg(x + (q * 3 + b) * kPackBlock));
  }
  __device__ __forceinline__ static int at(int m) { return OWN ? m * 6 : packed_at<3 * R>(m); }
};

// P = w x (rows of x: R spinor rows, component q at row 3 q + colour)
template <int R, bool OWN> __device__ __forceinline__ void pr_fwd(CP (&P)[R][3], const float4* __restrict__ x, const C<float> (&w)[3][3]) {
  SpinorWords<R, OWN> xs;
  xs.load(x);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    CP v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = xs.word(x, q, b);
#pragma unroll
    for (int q = 0; q < R; ++q) {
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        const float2 wr = pr_bc(w[aa][b].re), wi = pr_bc(w[aa][b].im);
        P[q][aa].re = b == 0 ? pr_mul(v[q].re, wr) : pr_fma(v[q].re, wr, P[q][aa].re);
        P[q][aa].im = b == 0 ? pr_mul(v[q].re, wi) : pr_fma(v[q].re, wi, P[q][aa].im);
      }
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        const float2 wr = pr_bc(w[aa][b].re), nw = pr_bc(-w[aa][b].im);
        P[q][aa].im = pr_fma(v[q].im, wr, P[q][aa].im);
        P[q][aa].re = pr_fma(v[q].im, nw, P[q][aa].re);
      }
    }
  }
}
// P = w^dagger x - P
template <int R, bool OWN> __device__ __forceinline__ void pr_bwd(CP (&P)[R][3], const float4* __restrict__ x, const C<float> (&w)[3][3]) {
  SpinorWords<R, OWN> xs;
  xs.load(x);
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    CP v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = xs.word(x, q, b);
#pragma unroll
    for (int q = 0; q < R; ++q) {
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        const float2 wr = pr_bc(w[b][aa].re), nw = pr_bc(-w[b][aa].im);
        P[q][aa].re = pr_fma(v[q].re, wr, b == 0 ? pr_neg(P[q][aa].re) : P[q][aa].re);
        P[q][aa].im = pr_fma(v[q].re, nw, b == 0 ? pr_neg(P[q][aa].im) : P[q][aa].im);
      }
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        const float2 wr = pr_bc(w[b][aa].re), wi = pr_bc(w[b][aa].im);
        P[q][aa].im = pr_fma(v[q].im, wr, P[q][aa].im);
        P[q][aa].re = pr_fma(v[q].im, wi, P[q][aa].re);
      }
    }
  }
}
template <int R> __device__ __forceinline__ void pr_axpy(CP (&acc)[R][3], const CP (&v)[R][3], float k) {
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) cp_add(acc[q][aa], v[q][aa], k);
}
// acc += sum_mu c_mu gamma_mu V, chiral basis (hops.cuh), on two right-hand sides
__device__ __forceinline__ void pr_gamma(CP (&acc)[4][3], const CP (&v)[4][3], float c1, float c2, float c3, float c4) {
#pragma unroll
  for (int aa = 0; aa < 3; ++aa) {
    cp_addi(acc[0][aa], v[3][aa], -c1);
    cp_addi(acc[1][aa], v[2][aa], -c1);
    cp_addi(acc[2][aa], v[1][aa], c1);
    cp_addi(acc[3][aa], v[0][aa], c1);
    cp_add(acc[0][aa], v[3][aa], -c2);
    cp_add(acc[1][aa], v[2][aa], c2);
    cp_add(acc[2][aa], v[1][aa], c2);
    cp_add(acc[3][aa], v[0][aa], -c2);
    cp_addi(acc[0][aa], v[2][aa], -c3);
    cp_addi(acc[1][aa], v[3][aa], c3);
    cp_addi(acc[2][aa], v[0][aa], c3);
    cp_addi(acc[3][aa], v[1][aa], -c3);
    cp_add(acc[0][aa], v[2][aa], c4);
    cp_add(acc[1][aa], v[3][aa], c4);
    cp_add(acc[2][aa], v[0][aa], c4);
    cp_add(acc[3][aa], v[1][aa], c4);
  }
}
// the same on two spins per word: gamma_1 and gamma_2 exchange the spins of a
// chirality, gamma_3 and gamma_4 do not
__device__ __forceinline__ void pr_gamma(CP (&acc)[2][3], const CP (&v)[2][3], float c1, float c2, float c3, float c4) {
  const float2 p1 = pr_bc(c1), m1 = pr_bc(-c1), p4 = pr_bc(c4);
  const float2 k2 = make_float2(-c2, c2), n2 = make_float2(c2, -c2), k3 = make_float2(c3, -c3), n3 = make_float2(-c3, c3);
#pragma unroll
  for (int aa = 0; aa < 3; ++aa) {
    const float2 s0r = pr_swp(v[0][aa].re), s0i = pr_swp(v[0][aa].im);
    const float2 s1r = pr_swp(v[1][aa].re), s1i = pr_swp(v[1][aa].im);
    acc[0][aa].re = pr_fma(s1i, p1, acc[0][aa].re);
    acc[0][aa].im = pr_fma(s1r, m1, acc[0][aa].im);
    acc[1][aa].re = pr_fma(s0i, m1, acc[1][aa].re);
    acc[1][aa].im = pr_fma(s0r, p1, acc[1][aa].im);
    acc[0][aa].re = pr_fma(s1r, k2, acc[0][aa].re);
    acc[0][aa].im = pr_fma(s1i, k2, acc[0][aa].im);
    acc[1][aa].re = pr_fma(s0r, n2, acc[1][aa].re);
    acc[1][aa].im = pr_fma(s0i, n2, acc[1][aa].im);
    acc[0][aa].re = pr_fma(v[1][aa].im, k3, acc[0][aa].re);
    acc[0][aa].im = pr_fma(v[1][aa].re, n3, acc[0][aa].im);
    acc[1][aa].re = pr_fma(v[0][aa].im, n3, acc[1][aa].re);
    acc[1][aa].im = pr_fma(v[0][aa].re, k3, acc[1][aa].im);
    acc[0][aa].re = pr_fma(v[1][aa].re, p4, acc[0][aa].re);
    acc[0][aa].im = pr_fma(v[1][aa].im, p4, acc[0][aa].im);
    acc[1][aa].re = pr_fma(v[0][aa].re, p4, acc[1][aa].re);
    acc[1][aa].im = pr_fma(v[0][aa].im, p4, acc[1][aa].im);
  }
}

// Sum over the hops at site n into acc (all 80, or those of every KS-th offset
// pair from i0 on); x = packed vector (R = 4: a pair of right-hand sides, R = 2: one).
template <int R, typename LS, int KS, bool OWN>
__device__ __forceinline__ void pr_hops(CP (&acc)[R][3], const Geom& g, int n, const float4* __restrict__ x,
                                        const LS* __restrict__ W, const PairHops<float>& H, int i0) {
  const int V = (int)g.V;
  // index steps to the neighbours in each direction (periodic)
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
  auto sites = [&](int j, int& mp, int& mm) {
    mp = n;
    mm = n;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int d = H.d[j][mu];
      mp += d > 0 ? up[mu] : (d < 0 ? dn[mu] : 0);
      mm += d > 0 ? dn[mu] : (d < 0 ? up[mu] : 0);
    }
  };
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) acc[q][aa] = CP{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  C<float> w[3][3], wm[3][3];
  int mp, mm;
  if constexpr (KS == 1) i0 = 0;
  sites(i0, mp, mm);
  load_stored_link<float, LS>(w, W, H.j[i0], n, V);
  load_stored_link<float, LS>(wm, W, H.j[i0], mm, V);
#pragma unroll 1
  for (int j = i0; j < 40; j += KS) {
    const int jn = KS == 1 ? (j < 39 ? j + 1 : 39) : (j < 40 - KS ? j + KS : j);
    const float a = H.a[j];
    const int op = SpinorWords<R, OWN>::at(mp), om = SpinorWords<R, OWN>::at(mm);
    CP P[R][3];
    pr_fwd<R, OWN>(P, x + op, w);
    sites(jn, mp, mm);
    load_stored_link<float, LS>(w, W, H.j[jn], n, V);
    pr_axpy<R>(acc, P, 2.f * a);
    pr_bwd<R, OWN>(P, x + om, wm);
    load_stored_link<float, LS>(wm, W, H.j[jn], mm, V);
    pr_axpy<R>(acc, P, a);
    pr_gamma(acc, P, H.c[j][0], H.c[j][1], H.c[j][2], H.c[j][3]);
  }
}

// Sum of v over the block (FP64, fixed order), valid in thread 0.
__device__ __forceinline__ double pr_block_total(double v) {
  __shared__ double sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

// One chirality's clover block on a pair of right-hand sides, o = C in, its
// reals used as they arrive (held in an array first they cost the main loop
// registers: 0.68 against 0.64 ns per site and rhs).
__device__ __forceinline__ void pr_clover(CP (&o)[6], const float* __restrict__ cl, int64_t n, int h, const CP (&in)[6]) {
  const float4* q = reinterpret_cast<const float4*>(cl + clover_at32(n, h, 0));
  float4 v = __ldg(q);
  const float4 v1 = __ldg(q + kCloverBlock);
  o[0] = CP{pr_mul(in[0].re, pr_bc(v.x)), pr_mul(in[0].im, pr_bc(v.x))};
  o[1] = CP{pr_mul(in[1].re, pr_bc(v.y)), pr_mul(in[1].im, pr_bc(v.y))};
  o[2] = CP{pr_mul(in[2].re, pr_bc(v.z)), pr_mul(in[2].im, pr_bc(v.z))};
  o[3] = CP{pr_mul(in[3].re, pr_bc(v.w)), pr_mul(in[3].im, pr_bc(v.w))};
  o[4] = CP{pr_mul(in[4].re, pr_bc(v1.x)), pr_mul(in[4].im, pr_bc(v1.x))};
  o[5] = CP{pr_mul(in[5].re, pr_bc(v1.y)), pr_mul(in[5].im, pr_bc(v1.y))};
  v = v1;
  int k = 6;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      if (k % 4 == 0) v = __ldg(q + k / 4 * kCloverBlock);
      const float r = k % 4 == 0 ? v.x : v.z, m = k % 4 == 0 ? v.y : v.w;
      cp_add(o[i], in[j], r);
      cp_addi(o[i], in[j], m);
      cp_add(o[j], in[i], r);
      cp_addi(o[j], in[i], -m);
      k += 2;
    }
}

// The solver's epilogue on packed vectors: y = D x + sig_s p_s and the site
// block's partial of Re<p_s, y> in part[s * blocks + block].  A thread's products are
// summed in FP32 (EPI = 1, one lattice) or to FP64 accuracy and range (EPI = 2,
// batched lattices: sum3.cuh, p and y scaled by 2^k2).
struct PackedDot {
  const float4* p;    // packed base directions
  const double* sig;  // per system
  double* part;       // [nsys][blocks]
};

// The thread group of a 128-thread block; a warp is of one group.  Told so, the
// compiler keeps the offset's constants in uniform registers (16^3.32 x 12, two
// groups: 1089 -> 1027 us).
template <int KS> __device__ __forceinline__ int pr_group() {
  if constexpr (KS == 1) return 0;
  return __shfl_sync(0xffffffffu, threadIdx.x / (128 / KS), 0);
}

// D x at the sites of block blk of one packed group, a site's offset pairs split
// over KS thread groups: each takes every KS-th pair, their sums meet in shared
// memory and the groups 0 and 1 finish one chirality each.  x, yp: the group's
// packed vectors, y0: its first right-hand side in the spinors' own layout (OUT =
// 0 writes y0, OUT = 1 yp).  EPI > 0 (R = 2, OUT = 1): the epilogue of system s, p at
// word po of sd.p.
template <int R, typename LS, int OUT, int EPI, int KS, bool OWN = false>
__device__ __forceinline__ void pr_block(const Geom& g, int blk, float* __restrict__ y0, float4* __restrict__ yp,
                                         const float4* __restrict__ x, const LS* __restrict__ W,
                                         const float* __restrict__ cl, float diag, const PairHops<float>& H, const PackedDot& sd,
                                         int64_t po, int s, int nb, int k2 = 0) {
  static_assert(R == 2 || (OUT == 0 && KS == 1), "pairs: spinors' own layout out, one thread per site");
  static_assert(!EPI || OUT == 1, "the epilogue writes packed vectors");
  constexpr int SB = 128 / KS;
  constexpr bool STAGE = R == 2 && OUT == 0 && KS == 1;
  const int n0 = blk * SB + (KS == 1 ? threadIdx.x : threadIdx.x % SB);
  const bool valid = n0 < g.V;
  if (R == 4 && !valid) return;  // else every thread takes part in the block's exchanges
  const int n = valid ? n0 : 0, grp = pr_group<KS>();
  CP acc[R][3];
  pr_hops<R, LS, KS, OWN>(acc, g, n, x, W, H, grp);
  if constexpr (KS > 1) {
    __shared__ float4 red[KS][6][SB];
    const int l = threadIdx.x % SB;
#pragma unroll
    for (int i = 0; i < 6; ++i) red[grp][i][l] = cp_word(acc[i / 3][i % 3]);
    __syncthreads();
    if (grp < 2) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        CP t = cp_of(red[0][grp * 3 + i][l]);
#pragma unroll
        for (int k = 1; k < KS; ++k) {
          const CP u = cp_of(red[k][grp * 3 + i][l]);
          t.re = make_float2(t.re.x + u.re.x, t.re.y + u.re.y);
          t.im = make_float2(t.im.x + u.im.x, t.im.y + u.im.y);
        }
        acc[0][i] = t;  // this group's chirality, whichever it is
        acc[1][i] = t;
      }
    }
  }
  const float4* xo = x + SpinorWords<R, OWN>::at(n);
  if constexpr (R == 4) {
    const int64_t rs = g.V * 24;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      CP own[6], out[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        own[i] = cp_of(__ldg(xo + (h * 6 + i) * kPackBlock));
        out[i] = acc[h * 2 + i / 3][i % 3];
        cp_add(out[i], own[i], diag);
      }
      if (cl) {
        CP co[6];
        pr_clover(co, cl, n, h, own);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          out[i].re = make_float2(out[i].re.x + co[i].re.x, out[i].re.y + co[i].re.y);
          out[i].im = make_float2(out[i].im.x + co[i].im.x, out[i].im.y + co[i].im.y);
        }
      }
      float4* ya = reinterpret_cast<float4*>(y0 + (int64_t)n * 24 + h * 12);
      float4* yb = reinterpret_cast<float4*>(y0 + rs + (int64_t)n * 24 + h * 12);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        ya[i] = make_float4(out[2 * i].re.x, out[2 * i].im.x, out[2 * i + 1].re.x, out[2 * i + 1].im.x);
        yb[i] = make_float4(out[2 * i].re.y, out[2 * i].im.y, out[2 * i + 1].re.y, out[2 * i + 1].im.y);
      }
    }
  } else {
    __shared__ float4 stage[STAGE ? 128 * 7 : 1];
    const float sig = EPI ? (float)sd.sig[s] : 0.f;
    float dA = 0.f, dB = 0.f;
    Sum3 sum = sum3_zero();
    const float2 sc = pr_bc(exp2_float(k2));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (KS > 1 && h != grp) continue;
      C<float> in[6], out[6];
      CP xh[3];
      SpinorWords<R, OWN>::load_half(xo, h, xh);
#pragma unroll
      for (int aa = 0; aa < 3; ++aa) {
        const CP own = xh[aa];
        cp_add(acc[h][aa], own, diag);
        in[aa] = C<float>{own.re.x, own.im.x};
        in[3 + aa] = C<float>{own.re.y, own.im.y};
        out[aa] = C<float>{acc[h][aa].re.x, acc[h][aa].im.x};
        out[3 + aa] = C<float>{acc[h][aa].re.y, acc[h][aa].im.y};
      }
      if (cl) {
        C<float> co[6];
        float c[36];
        load_clover(c, cl, g.V, n, h);
        clover_block(co, c, in);
#pragma unroll
        for (int i = 0; i < 6; ++i) out[i] = out[i] + co[i];
      }
      if constexpr (OUT == 1) {
#pragma unroll
        for (int aa = 0; aa < 3; ++aa) {
          const int at = packed_at<6>(n) + (h * 3 + aa) * kPackBlock;
          CP v{make_float2(out[aa].re, out[3 + aa].re), make_float2(out[aa].im, out[3 + aa].im)};
          if constexpr (EPI) {
            const CP pv = cp_of(__ldg(sd.p + po + at));
            v.re = pr_fma(pv.re, pr_bc(sig), v.re);
            v.im = pr_fma(pv.im, pr_bc(sig), v.im);
            if constexpr (EPI == 1) {
              dA = fmaf(pv.re.x, v.re.x, dA);
              dB = fmaf(pv.re.y, v.re.y, dB);
              dA = fmaf(pv.im.x, v.im.x, dA);
              dB = fmaf(pv.im.y, v.im.y, dB);
            } else {
              sum3_add(sum, pr_mul(pv.re, sc), pr_mul(v.re, sc));
              sum3_add(sum, pr_mul(pv.im, sc), pr_mul(v.im, sc));
            }
          }
          if (valid) yp[at] = cp_word(v);
        }
      } else {
        float4* ya = STAGE ? stage + threadIdx.x * 7 + h * 3 : reinterpret_cast<float4*>(y0 + (int64_t)n * 24 + h * 12);
        if (STAGE || valid) {
#pragma unroll
          for (int i = 0; i < 3; ++i)
            ya[i] = make_float4(out[2 * i].re, out[2 * i].im, out[2 * i + 1].re, out[2 * i + 1].im);
        }
      }
    }
    if constexpr (STAGE) {
      // a warp's 32 sites are 3 KB of y, stored in whole sectors (16^3.32 x 12: 1063 -> 1019 us)
      __syncwarp();
      const int lane = threadIdx.x & 31, w0 = threadIdx.x - lane, m = ((int)g.V - blk * SB - w0) * 6;
      float4* yw = reinterpret_cast<float4*>(y0 + (int64_t)(blk * SB + w0) * 24);
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        const int k = i * 32 + lane;
        if (k < m) yw[k] = stage[(w0 + k / 6) * 7 + k % 6];
      }
    }
    if constexpr (EPI) {
      const double d = EPI == 1 ? (double)dA + (double)dB : sum3_total(sum);
      const double t = pr_block_total(valid ? d : 0.0);
      if (threadIdx.x == 0) sd.part[(int64_t)s * nb + blk] = EPI == 1 ? t : t * exp2_square(k2);
    }
  }
}

// y = D x on `groups` packed groups of one lattice; the first one holds right-hand
// side rhs0 (and rhs0 + 1).  OWN: x in its own layout, a group one right-hand side.
template <int R, typename LS, int KS, bool OWN = false>
__global__ void __launch_bounds__(128, R == 4 ? 3 : 4)
    bri_pair_kernel(Geom g, float* __restrict__ y, const float4* __restrict__ x, const LS* __restrict__ W,
                    const float* __restrict__ cl, float diag, int rhs0, int gfirst, const __grid_constant__ PairHops<float> H) {
  const int grp = gfirst ? blockIdx.x : blockIdx.y, blk = gfirst ? blockIdx.y : blockIdx.x;
  pr_block<R, LS, 0, 0, KS, OWN>(g, blk, y + (int64_t)(rhs0 + grp * (R / 2)) * g.V * 24, nullptr,
                                x + (int64_t)grp * (OWN ? g.V * 6 : packed_words(g.V, 3 * R)), W, cl, diag, H,
                                PackedDot{nullptr, nullptr, nullptr}, 0, 0, 0);
}

// Spinors [nrhs][V][12] complex64 -> packed groups; group g holds the
// right-hand sides rhs0 + 2g, rhs0 + 2g + 1 (R = 4) or rhs0 + g (R = 2).
template <int R> __global__ void __launch_bounds__(256) k_pack(int64_t V, const float* __restrict__ x, int rhs0, float4* __restrict__ X) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;  // 16-byte word (R = 4) or spin pair (R = 2) of a site
  if (i >= V * 6) return;
  const int64_t n = i / 6;
  const int q = (int)(i - n * 6);
  float4* o = X + (int64_t)blockIdx.y * packed_words(V, 3 * R) + packed_at<3 * R>((int)n);
  if constexpr (R == 4) {
    const float* p = x + (rhs0 + 2 * (int64_t)blockIdx.y) * V * 24 + i * 4;
    const float4 u = __ldg(reinterpret_cast<const float4*>(p));
    const float4 v = __ldg(reinterpret_cast<const float4*>(p + V * 24));
    o[(2 * q) * kPackBlock] = make_float4(u.x, v.x, u.y, v.y);
    o[(2 * q + 1) * kPackBlock] = make_float4(u.z, v.z, u.w, v.w);
  } else {
    const int h = q / 3, b = q - 3 * h;
    const float2* p = reinterpret_cast<const float2*>(x + (rhs0 + (int64_t)blockIdx.y) * V * 24 + n * 24) + h * 6 + b;
    const float2 u = __ldg(p), v = __ldg(p + 3);
    o[q * kPackBlock] = make_float4(u.x, v.x, u.y, v.y);
  }
}

template <int R> inline void launch_pack(int64_t V, const float* x, int rhs0, int groups, float4* X, cudaStream_t s) {
  k_pack<R><<<dim3(blocks_for(V * 6, 256), groups), 256, 0, s>>>(V, x, rhs0, X);
  note_launch();
}
// y = D x for `groups` pairs of right-hand sides starting at rhs0.
template <typename LS>
inline void launch_pairs(const Geom& g, float* y, const float4* X, const LS* W, const float* cl, float diag, int dagger,
                         int rhs0, int groups, cudaStream_t s) {
  const StencilGrid sg = stencil_grid(blocks_for(g.V, 128), groups);
  bri_pair_kernel<4, LS, 1><<<sg.grid, 128, 0, s>>>(g, y, X, W, cl, diag, rhs0, sg.gfirst, pair_hops<float>(dagger));
  note_launch();
}

// y = D x for `n` single right-hand sides starting at rhs0; OWN: X is x itself.
template <typename LS, bool OWN = false>
inline void launch_singles(const Geom& g, float* y, const float4* X, const LS* W, const float* cl, float diag, int dagger,
                           int rhs0, int n, cudaStream_t s) {
  const int ks = pack_groups(g.V * n);
  const StencilGrid sg = stencil_grid(blocks_for(g.V, pack_sites(ks)), n);
  with_groups(ks, [&](auto k) {
    bri_pair_kernel<2, LS, decltype(k)::value, OWN><<<sg.grid, 128, 0, s>>>(g, y, X, W, cl, diag, rhs0, sg.gfirst, pair_hops<float>(dagger));
  });
  note_launch();
}

}  // namespace bri
