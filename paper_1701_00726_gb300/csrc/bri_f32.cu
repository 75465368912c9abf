// FP32-spinor Brillouin stencil (FP32 and BF16 link storage): which kernel a
// launch takes, and the packed vectors the large ones run on.
#include "bri_pair.cuh"
#include "bri_split.cuh"

#include <algorithm>

namespace bri {

// The packed kernels cost a packing pass, and below some thousand sites they
// leave the chip idle where the split kernel's 5..20 threads per site do not.
// Measured on GB300 (us, split / packed with its packing pass): 4^4 x 1 rhs 6.5 /
// 15, 8^4 x 1 14.7 / 15.5, 8^4 x 2 20.8 / 19.9; above the line 6^4 x 12 33 / 25,
// 8^4 x 4 31 / 24, 12^4 x 1 39 / 30, 16^4 x 1 102 / 66.
bool bri_f32_packed(int64_t V, int nrhs) { return V * nrhs > 8192; }

// More thread groups per site give more blocks, fewer sites per block share less
// of each other's cache lines.  Measured on GB300 (us, 1 / 2 / 4 groups, packed
// out): 8^4 x 1 25 / 15 / 10.6, 8^4 x 4 25 / 19 / 19, 12^4 x 4 81 / 70 / 69, 16^4 x
// 1 66 / 61 / 62, 8^3.16 x 12 84 / 74 / 72, 16^3.32 x 1 109 / 109 / 109, x 2 191 /
// 187 / 193, x 4 349 / 354 / 368, x 12 998 / 1023 / 1064, 24^3.48 x 1 521 / 524 / 542.
int pack_groups(int64_t site_rhs) { return site_rhs <= 98304 ? 4 : (site_rhs <= 393216 ? 2 : 1); }

// Pairs of right-hand sides share a link's loads, single ones have twice the
// threads.  Measured on GB300 (us, spinors' own layout out, pairs / the better of
// one and two groups of singles): 16^3.32 x 4 359 / 355, x 12 993 / 1019, 24^3.48 x 4
// 1760 / 1811.  (Packed out the pairs lose: 381 / 349, 1048 / 998, 1853 / 1768.)
static bool take_pairs(int64_t V, int nrhs) { return nrhs > 1 && V * nrhs > 786432; }

int bri_f32_pack(int64_t V, const float* x, int nrhs, void* X, cudaStream_t s) {
  launch_pack<2>(V, x, 0, nrhs, (float4*)X, s);
  BRI_LAUNCH_CHECK("k_pack");
  return BRI_OK;
}

// Packed single right-hand sides -> spinors [nrhs][V][12] complex64.
static __global__ void __launch_bounds__(256) k_unpack(int64_t V, const float4* __restrict__ X, float* __restrict__ x) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= V * 6) return;
  const int64_t n = i / 6;
  const int q = (int)(i - n * 6);
  const float4 u = __ldg(X + (int64_t)blockIdx.y * packed_words(V, 6) + packed_at<6>((int)n) + q * kPackBlock);
  float2* p = reinterpret_cast<float2*>(x + (int64_t)blockIdx.y * V * 24 + n * 24) + q + 3 * (q / 3);
  p[0] = make_float2(u.x, u.z);
  p[3] = make_float2(u.y, u.w);
}

int bri_f32_unpack(int64_t V, const void* X, int nrhs, float* x, cudaStream_t s) {
  k_unpack<<<dim3(blocks_for(V * 6, 256), nrhs), 256, 0, s>>>(V, (const float4*)X, x);
  note_launch();
  BRI_LAUNCH_CHECK("k_unpack");
  return BRI_OK;
}

// Under capture an allocation would become a node of the caller's graph, which then
// could be no child graph, no body of a conditional node and be instantiated only once.
static bool may_allocate(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) return cap == cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return false;
}

// Spinors in their own layout in and out.  The packed copy of x lives in a
// stream-ordered allocation of at most kChunk right-hand sides; where there is
// no memory for it, or under capture, the kernels read x as it is.
template <typename LS>
int launch_bri_f32(const Geom& g, float* y, const float* x, const LS* W, const float* cl, float diag, int nrhs, int dagger,
                   cudaStream_t s, const ShiftDot<float>* sd, int* sd_blocks) {
  constexpr int kChunk = 16;
  if (!sd && bri_f32_packed(g.V, nrhs) && may_allocate(s)) {
    void* X = nullptr;
    if (scratch_alloc(&X, sizeof(float4) * packed_words(g.V, 6) * std::min(nrhs, kChunk), s) == cudaSuccess) {
      float4* X4 = (float4*)X;
      for (int r0 = 0; r0 < nrhs; r0 += kChunk) {
        const int nr = std::min(kChunk, nrhs - r0), pairs = take_pairs(g.V, nr) ? nr / 2 : 0, one = nr - 2 * pairs;
        float4* X1 = X4 + packed_words(g.V, 12) * pairs;
        if (pairs) {
          launch_pack<4>(g.V, x, r0, pairs, X4, s);
          launch_pairs<LS>(g, y, X4, W, cl, diag, dagger, r0, pairs, s);
        }
        if (one) {
          const int r1 = r0 + 2 * pairs;
          launch_pack<2>(g.V, x, r1, one, X1, s);
          launch_singles<LS>(g, y, X1, W, cl, diag, dagger, r1, one, s);
        }
      }
      cudaFreeAsync(X, s);
      BRI_LAUNCH_CHECK("bri_pair_kernel");
      return BRI_OK;
    }
  }
  if (!sd && bri_f32_packed(g.V, nrhs)) {
    launch_singles<LS, true>(g, y, (const float4*)x, W, cl, diag, dagger, 0, nrhs, s);
    BRI_LAUNCH_CHECK("bri_pair_kernel");
    return BRI_OK;
  }
  return launch_split<float, LS>(g, y, x, W, cl, diag, nrhs, dagger, s, sd, sd_blocks);
}
template int launch_bri_f32<float2>(const Geom&, float*, const float*, const float2*, const float*, float, int, int, cudaStream_t,
                                    const ShiftDot<float>*, int*);
template int launch_bri_f32<__nv_bfloat162>(const Geom&, float*, const float*, const __nv_bfloat162*, const float*, float, int,
                                            int, cudaStream_t, const ShiftDot<float>*, int*);

}  // namespace bri
