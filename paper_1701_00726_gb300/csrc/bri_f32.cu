// FP32-spinor Brillouin stencil (FP32 and BF16 link storage): which kernel a
// launch takes, and the packed vectors the large ones run on.
#include "bri_pair.cuh"
#include "bri_split.cuh"

#include <algorithm>

namespace bri {

// The packed kernels need a thread per site and pair of right-hand sides to
// fill the chip; below that the split kernel's 5..20 threads per site win.
// Measured on GB300 (us, split / packed with its packing pass): 4^4 x 1 rhs
// 6.5 / 26, 8^4 x 1 12 / 29, 8^4 x 4 31 / 39, 9.7.8.16 x 3 41 / 76, 12^4 x 1
// 35 / 41; above the line 16^4 x 1 113 / 72, 8^3.16 x 12 118 / 84.
bool bri_f32_packed(int64_t V, int nrhs) { return V * nrhs > 24576; }

// A packed vector of nrhs right-hand sides: nrhs / 2 pairs, then the odd one.
size_t bri_f32_packed_bytes(int64_t V, int nrhs) {
  return sizeof(float4) * (size_t)(packed_words(V, 12) * (nrhs / 2) + (nrhs % 2 ? packed_words(V, 6) : 0));
}

int bri_f32_pack(int64_t V, const float* x, int nrhs, void* X, cudaStream_t s) {
  const int pairs = nrhs / 2;
  float4* X4 = (float4*)X;
  if (pairs) launch_pack<4>(V, x, 0, pairs, X4, s);
  if (nrhs % 2) launch_pack<2>(V, x, nrhs - 1, 1, X4 + packed_words(V, 12) * pairs, s);
  BRI_LAUNCH_CHECK("k_pack");
  return BRI_OK;
}

int bri_f32_unpack(int64_t V, const void* X, int nrhs, float* x, cudaStream_t s) {
  const int pairs = nrhs / 2;
  const float4* X4 = (const float4*)X;
  if (pairs) launch_unpack<4>(V, X4, 0, pairs, x, s);
  if (nrhs % 2) launch_unpack<2>(V, X4 + packed_words(V, 12) * pairs, nrhs - 1, 1, x, s);
  BRI_LAUNCH_CHECK("k_unpack");
  return BRI_OK;
}

// y (spinors' layout) or yp (packed) = D x for the first na of nrhs right-hand
// sides of the packed vector X (a pair whose second member is not asked for is
// still computed whole).  With p (packed; yp only) the fused epilogue of
// ShiftDot, sd_blocks partials per system.
template <typename LS>
int bri_f32_on_packed(const Geom& g, float* y, void* yp, const void* X, const LS* W, const float* cl, float diag, int nrhs,
                      int na, int dagger, cudaStream_t s, const void* p, const double* sig, double* part, int* sd_blocks) {
  const int pairs = nrhs / 2, act = std::min(pairs, (na + 1) / 2);
  const int64_t o = packed_words(g.V, 12) * pairs;
  const float4 *X4 = (const float4*)X, *P4 = (const float4*)p;
  float4* Y4 = (float4*)yp;
  if (sd_blocks) *sd_blocks = blocks_for(g.V, 128);
  PackedDot sd{P4, sig, part};
  if (act) launch_pair<4, LS>(g, y, Y4, X4, W, cl, diag, dagger, 0, act, s, p ? &sd : nullptr);
  if (nrhs % 2 && na == nrhs) {
    sd.p = P4 + (p ? o : 0);
    launch_pair<2, LS>(g, y, Y4 ? Y4 + o : nullptr, X4 + o, W, cl, diag, dagger, nrhs - 1, 1, s, p ? &sd : nullptr);
  }
  BRI_LAUNCH_CHECK("bri_pair_kernel");
  return BRI_OK;
}
template int bri_f32_on_packed<float2>(const Geom&, float*, void*, const void*, const float2*, const float*, float, int, int,
                                       int, cudaStream_t, const void*, const double*, double*, int*);
template int bri_f32_on_packed<__nv_bfloat162>(const Geom&, float*, void*, const void*, const __nv_bfloat162*, const float*,
                                               float, int, int, int, cudaStream_t, const void*, const double*, double*, int*);

// Spinors in their own layout in and out.  The packed copy of x lives in a
// stream-ordered allocation of at most kChunk right-hand sides; where there is
// no memory for it the split kernel, which needs none, takes over.
template <typename LS>
int launch_bri_f32(const Geom& g, float* y, const float* x, const LS* W, const float* cl, float diag, int nrhs, int dagger,
                   cudaStream_t s, const ShiftDot<float>* sd, int* sd_blocks) {
  constexpr int kChunk = 16;
  if (!sd && bri_f32_packed(g.V, nrhs)) {
    configure_pool_once();
    void* X = nullptr;
    if (cudaMallocAsync(&X, bri_f32_packed_bytes(g.V, std::min(nrhs, kChunk)), s) == cudaSuccess) {
      note_device_alloc();
      int rc = BRI_OK;
      for (int r0 = 0; r0 < nrhs && rc == BRI_OK; r0 += kChunk) {
        const int nr = std::min(kChunk, nrhs - r0);
        const int64_t at = r0 * g.V * 24;
        rc = bri_f32_pack(g.V, x + at, nr, X, s);
        if (rc == BRI_OK) rc = bri_f32_on_packed<LS>(g, y + at, nullptr, X, W, cl, diag, nr, nr, dagger, s);
      }
      cudaFreeAsync(X, s);
      return rc;
    }
    cudaGetLastError();
  }
  return launch_split<float, LS>(g, y, x, W, cl, diag, nrhs, dagger, s, sd, sd_blocks);
}
template int launch_bri_f32<float2>(const Geom&, float*, const float*, const float2*, const float*, float, int, int, cudaStream_t,
                                    const ShiftDot<float>*, int*);
template int launch_bri_f32<__nv_bfloat162>(const Geom&, float*, const float*, const __nv_bfloat162*, const float*, float, int,
                                            int, cudaStream_t, const ShiftDot<float>*, int*);

}  // namespace bri
