// Device helpers shared by the Brillouin and Wilson stencil kernels.
#pragma once

#include "internal.cuh"
#include "cplx.cuh"

namespace bri {

template <typename R> struct Spinor {
  C<R> v[4][3];
};

// AoS spinor [4][3] complex: 24 reals, 16-byte vector loads.
__device__ __forceinline__ void load_spinor(Spinor<float>& s, const float* p) {
  const float4* q = reinterpret_cast<const float4*>(p);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    float4 v = __ldg(q + i);
    int e0 = 2 * i, e1 = 2 * i + 1;  // complex element index 0..11
    s.v[e0 / 3][e0 % 3] = C<float>{v.x, v.y};
    s.v[e1 / 3][e1 % 3] = C<float>{v.z, v.w};
  }
}
__device__ __forceinline__ void load_spinor(Spinor<double>& s, const double* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
  for (int e = 0; e < 12; ++e) {
    double2 v = __ldg(q + e);
    s.v[e / 3][e % 3] = C<double>{v.x, v.y};
  }
}
__device__ __forceinline__ void store_spinor(float* p, const Spinor<float>& s) {
  float4* q = reinterpret_cast<float4*>(p);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    int e0 = 2 * i, e1 = 2 * i + 1;
    q[i] = make_float4(s.v[e0 / 3][e0 % 3].re, s.v[e0 / 3][e0 % 3].im, s.v[e1 / 3][e1 % 3].re,
                       s.v[e1 / 3][e1 % 3].im);
  }
}
__device__ __forceinline__ void store_spinor(double* p, const Spinor<double>& s) {
  double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
  for (int e = 0; e < 12; ++e) q[e] = make_double2(s.v[e / 3][e % 3].re, s.v[e / 3][e % 3].im);
}

// One 3x3 FP64 link in structure-of-arrays storage: element e of the link at site
// n sits at p[e*V] (p already offset by n).
__device__ __forceinline__ void load_link(C<double> w[3][3], const double2* __restrict__ p, int V) {
#pragma unroll
  for (int e = 0; e < 9; ++e) w[e / 3][e % 3] = ld2(p + e * V);
}

// Stored link of offset j at site m.  FP64 links are [40][9][V] (element e at
// (j*9 + e)*V + m).  FP32 and BF16 links come in blocks of 32 sites, one
// contiguous chunk per offset and block: four (two) rows of 32 16-byte words
// holding elements 2k, 2k+1 (4k..4k+3), then a row of 32 words with the ninth
// element.  A link takes five (three) wide loads at immediate offsets from one
// address, and a warp reads one contiguous 2304-byte (1152-byte) chunk.
constexpr int kLinkBlock = 32;
constexpr int kLinkBytes32 = 72, kLinkBytes16 = 36;
__host__ __device__ __forceinline__ int64_t link_blocks(int64_t V) { return (V + kLinkBlock - 1) / kLinkBlock; }

// FP32 link j of the n a block of sites holds (40 stored off-axis links, 4 thin links).
template <int N> __device__ __forceinline__ void load_link_chunk(C<float> w[3][3], const float2* __restrict__ W, int j, int m) {
  const char* q = reinterpret_cast<const char*>(W) + ((int64_t)(m / kLinkBlock) * N + j) * (kLinkBlock * kLinkBytes32);
  const int lane = m % kLinkBlock;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(q) + k * kLinkBlock + lane);
    const int e0 = 2 * k, e1 = 2 * k + 1;
    w[e0 / 3][e0 % 3] = C<float>{v.x, v.y};
    w[e1 / 3][e1 % 3] = C<float>{v.z, v.w};
  }
  const float2 v = __ldg(reinterpret_cast<const float2*>(q + 64 * kLinkBlock) + lane);
  w[2][2] = C<float>{v.x, v.y};
}

template <typename R, typename LS>
__device__ __forceinline__ void load_stored_link(C<R> w[3][3], const LS* __restrict__ W, int j, int m, int V) {
  if constexpr (sizeof(R) == 4 && sizeof(LS) == 8) {
    load_link_chunk<40>(w, W, j, m);
  } else if constexpr (sizeof(LS) == 4) {
    const char* q = reinterpret_cast<const char*>(W) +
                    ((int64_t)(m / kLinkBlock) * 40 + j) * (kLinkBlock * kLinkBytes16);
    const int lane = m % kLinkBlock;
    const unsigned last = __ldg(reinterpret_cast<const unsigned*>(q + 32 * kLinkBlock) + lane);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(q) + k * kLinkBlock + lane);
      const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)  // BF16 is the upper half of an FP32 word
        w[(4 * k + i) / 3][(4 * k + i) % 3] =
            C<R>{(R)__uint_as_float(u[i] << 16), (R)__uint_as_float(u[i] & 0xffff0000u)};
    }
    w[2][2] = C<R>{(R)__uint_as_float(last << 16), (R)__uint_as_float(last & 0xffff0000u)};
  } else {
    load_link(w, W + (int64_t)j * 9 * V + m, V);
  }
}

__device__ __forceinline__ int wrap(int c, int L) { return c < 0 ? c + L : (c >= L ? c - L : c); }

// Clover storage: per chirality 36 reals (6 diagonal, then 15 upper
// off-diagonal complex, row by row).  FP64 [2][36][V]; FP32 in chunks of 32
// sites, [V/32][2][9][32] words of 16 bytes (reals 4r..4r+3 of a block).
constexpr int kCloverBlock = 32;
__host__ __device__ __forceinline__ int64_t clover_words32(int64_t V) { return (V + kCloverBlock - 1) / kCloverBlock * kCloverBlock * 18; }
__device__ __forceinline__ int64_t clover_at32(int64_t n, int h, int k) {
  return (((n / kCloverBlock * 18 + 9 * h + k / 4) * kCloverBlock) + n % kCloverBlock) * 4 + k % 4;
}
__device__ __forceinline__ double clover_real(const double* __restrict__ cl, int64_t V, int64_t n, int h, int k) {
  return __ldg(cl + ((int64_t)h * 36 + k) * V + n);
}
__device__ __forceinline__ float clover_real(const float* __restrict__ cl, int64_t, int64_t n, int h, int k) {
  return __ldg(cl + clover_at32(n, h, k));
}
// The 36 reals of block h at site n.
__device__ __forceinline__ void load_clover(double (&c)[36], const double* __restrict__ cl, int64_t V, int64_t n, int h) {
#pragma unroll
  for (int k = 0; k < 36; ++k) c[k] = clover_real(cl, V, n, h, k);
}
__device__ __forceinline__ void load_clover(float (&c)[36], const float* __restrict__ cl, int64_t V, int64_t n, int h) {
  const float4* q = reinterpret_cast<const float4*>(cl + clover_at32(n, h, 0));
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    const float4 v = __ldg(q + r * kCloverBlock);
    c[4 * r] = v.x;
    c[4 * r + 1] = v.y;
    c[4 * r + 2] = v.z;
    c[4 * r + 3] = v.w;
  }
}
// out = C in for one chirality block.
template <typename R>
__device__ __forceinline__ void clover_block(C<R> out[6], const R (&c)[36], const C<R> in[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) out[i] = C<R>{c[i] * in[i].re, c[i] * in[i].im};
  int k = 6;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      const C<R> cij{c[k], c[k + 1]};
      cfma(out[i], cij, in[j]);
      cfma_cj(out[j], cij, in[i]);
      k += 2;
    }
}

// Fused solver epilogue of a stencil launch: q = D x + sigma_s p_s at every
// site, and per block the partial sums of Re<p_s, q> in FP64 (the inner
// product of the multi-shift CG), written to part[s * blocks + site block] for
// the launch's right-hand side s.  p has the spinors' layout.
template <typename R> struct ShiftDot {
  const R* p;          // base search directions p_s (nullptr: no epilogue)
  const double* sig;   // per-system shift sigma_s
  double* part;        // [nsys][site blocks]
};

// Grid of a stencil launch: the right-hand-side groups in x (fastest, so the
// groups of one site block run together and reuse its links from L2) and the
// site blocks in y, unless there are more site blocks than a grid's y extent
// allows; gfirst tells the kernel which order was chosen.
struct StencilGrid {
  dim3 grid;
  int gfirst;
};
inline StencilGrid stencil_grid(int64_t site_blocks, int groups) {
  if (site_blocks <= 65535) return StencilGrid{dim3((unsigned)groups, (unsigned)site_blocks), 1};
  return StencilGrid{dim3((unsigned)site_blocks, (unsigned)groups), 0};
}

// Host-side launchers (one translation unit per precision).  sd (optional): the
// fused solver epilogue; sd_blocks receives the number of its partials per
// system, at most blocks_for(V, kMinSiteBlock).
constexpr int kMinSiteBlock = 8;
int launch_bri_f64(const Geom& g, double* y, const double* x, const double2* W, const double* cl, double diag, int nrhs,
                   int dagger, cudaStream_t s, const ShiftDot<double>* sd = nullptr, int* sd_blocks = nullptr);
template <typename LS>
int launch_bri_f32(const Geom& g, float* y, const float* x, const LS* W, const float* cl, float diag, int nrhs,
                   int dagger, cudaStream_t s, const ShiftDot<float>* sd = nullptr, int* sd_blocks = nullptr);
// Packed FP32 vectors of single right-hand sides (bri_pair.cuh) for the solver,
// which keeps its vectors in that form: whether a launch of nrhs right-hand sides
// takes the packed kernels, and packing.  pack_groups(V * nrhs): the thread groups
// that share a site's offsets, pack_sites of it: the sites of a block.
bool bri_f32_packed(int64_t V, int nrhs);
int pack_groups(int64_t site_rhs);
inline int pack_sites(int ks) { return 128 / ks; }
template <typename F> inline void with_groups(int ks, F&& f) {
  if (ks == 4) f(std::integral_constant<int, 4>());
  else if (ks == 2) f(std::integral_constant<int, 2>());
  else f(std::integral_constant<int, 1>());
}
int bri_f32_pack(int64_t V, const float* x, int nrhs, void* X, cudaStream_t s);
int bri_f32_unpack(int64_t V, const void* X, int nrhs, float* x, cudaStream_t s);
template <typename R, typename LS>
int launch_wil_t(const Geom& g, R* y, const R* x, const LS* U, const R* cl, R diag, int nrhs, int dagger,
                 cudaStream_t s);

}  // namespace bri
