// Wilson stencil (Eq. def_wils) with spin projection (App. C, Wilson operator
// flop count): for each of the 8 hops the 4-spinor is projected to 2 spin
// components with (1 -+ gamma_mu), transported, and rebuilt.
//
// FP32: links and clover come in 16-byte words of 32-site chunks; a block works on
// 64 sites of two right-hand sides, whose links the second finds in L1.  HBM could
// deliver its bytes (thin links 288, clover 288 and two spinors of 96 per site) in
// 94 us at 24^3 x 48, 2 rhs, clover; what bounds it is the latency of the gathers
// (12 to 16 warps per SM, DRAM and L2 half busy).  GB300, that case: 302 us with
// element-wise link and clover streams read once per right-hand side, 168 us with
// two right-hand sides per thread, 154 us now.  Against this: spinor words in order
// (load_words; L1 83 % busy instead of 56) 168 us; one block of 128 sites per rhs
// 176; 2, 4, 5 and 6 blocks per SM 187, 156, 174 and 186; prefetching a block's links and
// clover into L2 188 (two rhs per thread).
#include "stencil.cuh"

namespace bri {
namespace {

template <typename R> struct Nb {
  int64_t o[4][3];  // stride-scaled coordinates of x-1, x, x+1 (etc.), periodic
};

template <typename R>
__device__ __forceinline__ void neighbours(const Geom& g, int64_t n, Nb<R>& nb) {
  int64_t r = n;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    int L = g.L[mu];
    int c = (mu < 3) ? (int)(r % L) : (int)r;
    if (mu < 3) r /= L;
    int cm = c == 0 ? L - 1 : c - 1;
    int cp = c == L - 1 ? 0 : c + 1;
    nb.o[mu][0] = cm * g.str[mu];
    nb.o[mu][1] = c * g.str[mu];
    nb.o[mu][2] = cp * g.str[mu];
  }
}

// Spin projection (chiral basis): (1 -+ gamma_mu) x is fixed by its upper half
// h = x_up -+ e_mu x_low (e_k = -i sigma_k, e_4 = 1); its lower half is
// -+ e_mu^dagger h.  U acts on h only (2 spins), then the lower half is rebuilt.
template <typename R> __device__ __forceinline__ C<R> mul_i(C<R> a) { return C<R>{-a.im, a.re}; }
template <typename R> __device__ __forceinline__ C<R> neg(C<R> a) { return C<R>{-a.re, -a.im}; }

// PLUS = true for (1 + gamma_mu), false for (1 - gamma_mu)
template <int MU, bool PLUS, typename R>
__device__ __forceinline__ void project(const Spinor<R>& x, C<R> h[2][3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const C<R> x0 = x.v[0][c], x1 = x.v[1][c], x2 = x.v[2][c], x3 = x.v[3][c];
    if constexpr (MU == 0) {
      h[0][c] = PLUS ? x0 - mul_i(x3) : x0 + mul_i(x3);
      h[1][c] = PLUS ? x1 - mul_i(x2) : x1 + mul_i(x2);
    } else if constexpr (MU == 1) {
      h[0][c] = PLUS ? x0 - x3 : x0 + x3;
      h[1][c] = PLUS ? x1 + x2 : x1 - x2;
    } else if constexpr (MU == 2) {
      h[0][c] = PLUS ? x0 - mul_i(x2) : x0 + mul_i(x2);
      h[1][c] = PLUS ? x1 + mul_i(x3) : x1 - mul_i(x3);
    } else {
      h[0][c] = PLUS ? x0 + x2 : x0 - x2;
      h[1][c] = PLUS ? x1 + x3 : x1 - x3;
    }
  }
}

// acc += -1/2 * (projected, transported) spinor reconstructed from uh
template <int MU, bool PLUS, typename R>
__device__ __forceinline__ void reconstruct(Spinor<R>& acc, const C<R> uh[2][3]) {
  const R hf = (R)-0.5;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    C<R> h0 = uh[0][c], h1 = uh[1][c], v2, v3;
    if constexpr (MU == 0) {
      v2 = PLUS ? mul_i(h1) : neg(mul_i(h1));
      v3 = PLUS ? mul_i(h0) : neg(mul_i(h0));
    } else if constexpr (MU == 1) {
      v2 = PLUS ? h1 : neg(h1);
      v3 = PLUS ? neg(h0) : h0;
    } else if constexpr (MU == 2) {
      v2 = PLUS ? mul_i(h0) : neg(mul_i(h0));
      v3 = PLUS ? neg(mul_i(h1)) : mul_i(h1);
    } else {
      v2 = PLUS ? h0 : neg(h0);
      v3 = PLUS ? h1 : neg(h1);
    }
    acc.v[0][c] = acc.v[0][c] + hf * h0;
    acc.v[1][c] = acc.v[1][c] + hf * h1;
    acc.v[2][c] = acc.v[2][c] + hf * v2;
    acc.v[3][c] = acc.v[3][c] + hf * v3;
  }
}

__device__ __forceinline__ void load_thin(C<double> u[3][3], const double2* __restrict__ U, int mu, int64_t m, int64_t V) {
#pragma unroll
  for (int e = 0; e < 9; ++e) u[e / 3][e % 3] = ld2(U + ((int64_t)mu * 9 + e) * V + m);
}
__device__ __forceinline__ void load_thin(C<float> u[3][3], const float2* __restrict__ U, int mu, int64_t m, int64_t) {
  load_link_chunk<4>(u, U, mu, (int)m);
}

// N 16-byte words of a lane's spinor.  Neighbouring lanes are 96 bytes apart, so
// of eight lanes that read the same word two at a time meet in a bank; the lanes
// with bit 2 set take each pair of words the other way round, and none do.
template <int N> __device__ __forceinline__ void load_words(float4 (&v)[N], const float4* __restrict__ q) {
  const int odd = (threadIdx.x >> 2) & 1;
#pragma unroll
  for (int i = 0; i + 1 < N; i += 2) {
    const float4 a = __ldg(q + i + odd), b = __ldg(q + i + 1 - odd);
    v[i] = make_float4(odd ? b.x : a.x, odd ? b.y : a.y, odd ? b.z : a.z, odd ? b.w : a.w);
    v[i + 1] = make_float4(odd ? a.x : b.x, odd ? a.y : b.y, odd ? a.z : b.z, odd ? a.w : b.w);
  }
  if constexpr (N % 2 == 1) v[N - 1] = __ldg(q + N - 1);
}
__device__ __forceinline__ void load_site(Spinor<float>& s, const float* p) {
  float4 v[6];
  load_words<6>(v, reinterpret_cast<const float4*>(p));
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    s.v[2 * i / 3][2 * i % 3] = C<float>{v[i].x, v[i].y};
    s.v[(2 * i + 1) / 3][(2 * i + 1) % 3] = C<float>{v[i].z, v[i].w};
  }
}
__device__ __forceinline__ void load_site(Spinor<double>& s, const double* p) { load_spinor(s, p); }
// the six components of chirality h
__device__ __forceinline__ void load_chirality(C<float> (&o)[6], const float* p, int h) {
  float4 v[3];
  load_words<3>(v, reinterpret_cast<const float4*>(p) + 3 * h);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    o[2 * i] = C<float>{v[i].x, v[i].y};
    o[2 * i + 1] = C<float>{v[i].z, v[i].w};
  }
}
__device__ __forceinline__ void load_chirality(C<double> (&o)[6], const double* p, int h) {
#pragma unroll
  for (int i = 0; i < 6; ++i) o[i] = ld2(reinterpret_cast<const double2*>(p) + 6 * h + i);
}

// forward: -1/2 (1 - gamma_mu) U_mu(n) x(n+mu); backward: -1/2 (1 + gamma_mu) U_mu(n-mu)^+ x(n-mu)
// (dagger swaps the two projectors).
template <int MU, typename R, typename LS, bool DAG>
__device__ __forceinline__ void wil_dir(Spinor<R>& acc, const R* __restrict__ xin, const LS* __restrict__ U, int64_t V, int64_t n,
                                        const Nb<R>& nb) {
  const int64_t mf = nb.o[0][1] + nb.o[1][1] + nb.o[2][1] + nb.o[3][1] - nb.o[MU][1] + nb.o[MU][2];
  const int64_t mb = nb.o[0][1] + nb.o[1][1] + nb.o[2][1] + nb.o[3][1] - nb.o[MU][1] + nb.o[MU][0];
  C<R> u[3][3], h[2][3], uh[2][3];
  Spinor<R> xs;
  load_thin(u, U, MU, n, V);
  load_site(xs, xin + mf * 24);
  project<MU, DAG>(xs, h);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      uh[s][a] = C<R>{0, 0};
#pragma unroll
      for (int b = 0; b < 3; ++b) cfma(uh[s][a], u[a][b], h[s][b]);
    }
  reconstruct<MU, DAG>(acc, uh);
  load_thin(u, U, MU, mb, V);
  load_site(xs, xin + mb * 24);
  project<MU, !DAG>(xs, h);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      uh[s][a] = C<R>{0, 0};
#pragma unroll
      for (int b = 0; b < 3; ++b) cfma_cj(uh[s][a], u[b][a], h[s][b]);
    }
  reconstruct<MU, !DAG>(acc, uh);
}

// RB right-hand sides per block of 128 threads, one per thread
template <typename R, typename LS, int RB, bool DAG, bool CLOV>
__global__ void __launch_bounds__(128, sizeof(R) == 8 ? 1 : 3) wil_kernel(Geom g, R* __restrict__ y, const R* __restrict__ x, int rhs0,
                                                  const LS* __restrict__ U, const R* __restrict__ cl, R diag) {
  constexpr int SB = 128 / RB;
  const int64_t n = blockIdx.x * (int64_t)SB + threadIdx.x % SB;
  if (n >= g.V) return;
  const int64_t rhs_off = (rhs0 + (int64_t)blockIdx.y * RB + threadIdx.x / SB) * g.V * 24;
  const R* xin = x + rhs_off;
  Nb<R> nb;
  neighbours(g, n, nb);
  Spinor<R> acc;
  load_site(acc, xin + n * 24);
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) acc.v[s][a] = diag * acc.v[s][a];
  wil_dir<0, R, LS, DAG>(acc, xin, U, g.V, n, nb);
  wil_dir<1, R, LS, DAG>(acc, xin, U, g.V, n, nb);
  wil_dir<2, R, LS, DAG>(acc, xin, U, g.V, n, nb);
  wil_dir<3, R, LS, DAG>(acc, xin, U, g.V, n, nb);
  if constexpr (CLOV) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      R c[36];
      load_clover(c, cl, g.V, n, h);
      C<R> in[6], out[6];
      load_chirality(in, xin + n * 24, h);
      clover_block(out, c, in);
#pragma unroll
      for (int i = 0; i < 6; ++i) acc.v[2 * h + i / 3][i % 3] = acc.v[2 * h + i / 3][i % 3] + out[i];
    }
  }
  store_spinor(y + rhs_off + n * 24, acc);
}

template <typename R, typename LS, int RB>
void launch_wil_rb(const Geom& g, R* y, const R* x, int rhs0, int groups, const LS* U, const R* cl, R diag, int dagger,
                   cudaStream_t s) {
  const int th = 128;
  const dim3 grid(blocks_for(g.V, th / RB), groups);
  if (dagger) {
    if (cl) wil_kernel<R, LS, RB, true, true><<<grid, th, 0, s>>>(g, y, x, rhs0, U, cl, diag);
    else wil_kernel<R, LS, RB, true, false><<<grid, th, 0, s>>>(g, y, x, rhs0, U, cl, diag);
  } else {
    if (cl) wil_kernel<R, LS, RB, false, true><<<grid, th, 0, s>>>(g, y, x, rhs0, U, cl, diag);
    else wil_kernel<R, LS, RB, false, false><<<grid, th, 0, s>>>(g, y, x, rhs0, U, cl, diag);
  }
  note_launch();
}

}  // namespace

template <typename R, typename LS>
int launch_wil_t(const Geom& g, R* y, const R* x, const LS* U, const R* cl, R diag, int nrhs, int dagger,
                 cudaStream_t s) {
  constexpr int RB = sizeof(R) == 4 ? 2 : 1;
  const int groups = nrhs / RB;
  if (groups) launch_wil_rb<R, LS, RB>(g, y, x, 0, groups, U, cl, diag, dagger, s);
  if (nrhs > groups * RB) launch_wil_rb<R, LS, 1>(g, y, x, groups * RB, nrhs - groups * RB, U, cl, diag, dagger, s);
  BRI_LAUNCH_CHECK("wil_kernel");
  return BRI_OK;
}

template int launch_wil_t<double, double2>(const Geom&, double*, const double*, const double2*, const double*,
                                           double, int, int, cudaStream_t);
template int launch_wil_t<float, float2>(const Geom&, float*, const float*, const float2*, const float*, float, int,
                                         int, cudaStream_t);

}  // namespace bri
