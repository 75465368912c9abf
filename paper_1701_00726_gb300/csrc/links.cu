// Link preparation (once per gauge configuration):
//  * thin links with the time boundary applied, structure-of-arrays;
//  * the 40 stored path-averaged off-axis transporters W_d(n) (App. C: average
//    over the k! shortest paths, no SU(3) back-projection), built level by level
//    with the last-step recursion
//        W_d(n) = (1/k) sum_{mu: d_mu != 0} W_{d - s_mu e_mu}(n) U_step(n + d - s_mu e_mu, mu, s_mu)
//    which groups the k! paths by their final hop; a lower transporter that is
//    not stored is the mirrored one, W_{82-nu}(n) = W_nu(n + d)^dagger.  FP64, and
//    FP32 and BF16 copies from the same registers;
//  * the clover term -(c_SW/2) sum_{mu<nu} sigma_{mu nu} F_{mu nu} (Eq. def_bril)
//    in the chiral basis, two Hermitian 6x6 blocks per site, its leaves products
//    of the two-hop paths of the link construction.
//
// The construction is bound by FP64 arithmetic (104 products of 3x3 complex
// matrices per site for the links, 24 for the clover leaves: 2.9 ms at 16^3 x 32
// at the measured FP64 rate).  GB300, 16^3 x 32 with clover, construction and
// export of the stored links: 10.6 ms with all 80 transporters in a scratch array
// (allocated and freed on each call), twelve products per clover plane and a
// strided export, 4.4 ms now.
#include "stencil.cuh"

namespace bri {
namespace {

struct SiteCoord {
  int c[4];
};

__device__ __forceinline__ SiteCoord coords(const Geom& g, int64_t n) {
  SiteCoord s;
  int64_t r = n;
  s.c[0] = (int)(r % g.L[0]); r /= g.L[0];
  s.c[1] = (int)(r % g.L[1]); r /= g.L[1];
  s.c[2] = (int)(r % g.L[2]); r /= g.L[2];
  s.c[3] = (int)r;
  return s;
}

__device__ __forceinline__ int64_t site_of(const Geom& g, const int c[4]) {
  int64_t n = 0;
#pragma unroll
  for (int mu = 3; mu >= 0; --mu) {
    int v = c[mu] % g.L[mu];
    if (v < 0) v += g.L[mu];
    n = n * g.L[mu] + v;
  }
  return n;
}

__device__ __forceinline__ int64_t displaced(const Geom& g, const SiteCoord& s, int dx, int dy, int dz, int dt) {
  int c[4] = {s.c[0] + dx, s.c[1] + dy, s.c[2] + dz, s.c[3] + dt};
  return site_of(g, c);
}

__device__ __forceinline__ M3<double> load_soa(const double2* base, int64_t V, int64_t n) {
  M3<double> m;
#pragma unroll
  for (int e = 0; e < 9; ++e) m.m[e / 3][e % 3] = ld2(base + (int64_t)e * V + n);
  return m;
}

__device__ __forceinline__ void store_soa(double2* base, int64_t V, int64_t n, const M3<double>& m) {
#pragma unroll
  for (int e = 0; e < 9; ++e) base[(int64_t)e * V + n] = make_double2(m.m[e / 3][e % 3].re, m.m[e / 3][e % 3].im);
}

// One FP32 link into row-of-32 chunk c at lane (load_link_chunk's layout).
__device__ __forceinline__ void store_link_chunk(float2* W, int64_t c, int lane, const float2 (&f)[9]) {
  char* q = reinterpret_cast<char*>(W) + c * (kLinkBlock * kLinkBytes32);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    reinterpret_cast<float4*>(q)[k * kLinkBlock + lane] = make_float4(f[2 * k].x, f[2 * k].y, f[2 * k + 1].x, f[2 * k + 1].y);
  reinterpret_cast<float2*>(q + 64 * kLinkBlock)[lane] = f[8];
}

// AoS caller layout [V][4][3][3] complex128 -> SoA [4][9][V] FP64 and chunked
// FP32, with the antiperiodic sign on U_t of the last time slice.
__global__ void thin_links_kernel(Geom g, const double2* __restrict__ U, double2* U64, float2* U32, int anti) {
  int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  int t = (int)(n / g.str[3]);
  for (int mu = 0; mu < 4; ++mu) {
    double sgn = (anti && mu == 3 && t == g.L[3] - 1) ? -1.0 : 1.0;
    float2 f[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      double2 v = U[(n * 4 + mu) * 9 + e];
      v.x *= sgn;
      v.y *= sgn;
      U64[((int64_t)mu * 9 + e) * g.V + n] = v;
      f[e] = make_float2((float)v.x, (float)v.y);
    }
    store_link_chunk(U32, n / kLinkBlock * 4 + mu, (int)(n % kLinkBlock), f);
  }
}

__device__ __forceinline__ int nu_of(int dx, int dy, int dz, int dt) {
  return (dx + 1) + 3 * (dy + 1) + 9 * (dz + 1) + 27 * (dt + 1);
}

// One-hop transporters: W_{+mu}(n) = U_mu(n), W_{-mu}(n) = U_mu(n - mu)^dagger.
__global__ void level1_kernel(Geom g, const double2* __restrict__ U64, double2* T) {
  int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  SiteCoord s = coords(g, n);
  for (int mu = 0; mu < 4; ++mu) {
    int e[4] = {0, 0, 0, 0};
    e[mu] = 1;
    M3<double> fwd = load_soa(U64 + (int64_t)mu * 9 * g.V, g.V, n);
    int64_t nb = displaced(g, s, -e[0], -e[1], -e[2], -e[3]);
    M3<double> bwd = adj(load_soa(U64 + (int64_t)mu * 9 * g.V, g.V, nb));
    store_soa(T + (int64_t)nu_of(e[0], e[1], e[2], e[3]) * 9 * g.V, g.V, n, fwd);
    store_soa(T + (int64_t)nu_of(-e[0], -e[1], -e[2], -e[3]) * 9 * g.V, g.V, n, bwd);
  }
}

}  // namespace

LevelList level_list(int k) {
  LevelList lst;
  lst.count = 0;
  for (int nu = 0; nu < 81; ++nu) {
    int d[4] = {nu % 3 - 1, (nu / 3) % 3 - 1, (nu / 9) % 3 - 1, (nu / 27) % 3 - 1};
    int h = (d[0] != 0) + (d[1] != 0) + (d[2] != 0) + (d[3] != 0);
    if (h == k) lst.nu[lst.count++] = nu;
  }
  return lst;
}

// The stored ones among them (nu <= 40).
static LevelList stored_level(int k) {
  LevelList all = level_list(k), lst;
  lst.count = 0;
  for (int i = 0; i < all.count; ++i)
    if (all.nu[i] < 40) lst.nu[lst.count++] = all.nu[i];
  return lst;
}

namespace {

// k-hop transporters from (k-1)-hop ones at the same site (last-step recursion),
// all 80 offsets (the adjoint's recursion needs them).
__global__ void levelk_kernel(Geom g, const double2* __restrict__ U64, double2* T, LevelList lst, int k) {
  int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int which = blockIdx.y;
  if (n >= g.V || which >= lst.count) return;
  int nu = lst.nu[which];
  int d[4] = {nu % 3 - 1, (nu / 3) % 3 - 1, (nu / 9) % 3 - 1, (nu / 27) % 3 - 1};
  SiteCoord s = coords(g, n);
  M3<double> acc;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) acc.m[i][j] = C<double>{0.0, 0.0};
  for (int mu = 0; mu < 4; ++mu) {
    if (d[mu] == 0) continue;
    int sg = d[mu];
    int dp[4] = {d[0], d[1], d[2], d[3]};
    dp[mu] -= sg;  // d' = d - s e_mu
    M3<double> wprev = load_soa(T + (int64_t)nu_of(dp[0], dp[1], dp[2], dp[3]) * 9 * g.V, g.V, n);
    M3<double> step;
    if (sg > 0) {  // U_mu(n + d')
      int64_t m = displaced(g, s, dp[0], dp[1], dp[2], dp[3]);
      step = load_soa(U64 + (int64_t)mu * 9 * g.V, g.V, m);
    } else {       // U_mu(n + d' - mu)^dagger
      int q[4] = {dp[0], dp[1], dp[2], dp[3]};
      q[mu] -= 1;
      int64_t m = displaced(g, s, q[0], q[1], q[2], q[3]);
      step = adj(load_soa(U64 + (int64_t)mu * 9 * g.V, g.V, m));
    }
    madd(acc, mmul(wprev, step));
  }
  double inv = 1.0 / k;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) acc.m[i][j] = inv * acc.m[i][j];
  store_soa(T + (int64_t)nu * 9 * g.V, g.V, n, acc);
}

// One stored link: FP64 structure-of-arrays element planes and the FP32 and BF16
// chunks that load_stored_link reads.
__device__ __forceinline__ void store_link(double2* W64, float2* W32, __nv_bfloat162* W16, int64_t V, int64_t n, int j,
                                           const M3<double>& m) {
  float2 f[9];
  unsigned h[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const C<double> v = m.m[e / 3][e % 3];
    W64[((int64_t)j * 9 + e) * V + n] = make_double2(v.re, v.im);
    f[e] = make_float2((float)v.re, (float)v.im);
    const __nv_bfloat162 b = __floats2bfloat162_rn(f[e].x, f[e].y);
    memcpy(&h[e], &b, 4);
  }
  const int64_t blk = n / kLinkBlock * 40 + j;
  const int lane = (int)(n % kLinkBlock);
  store_link_chunk(W32, blk, lane, f);
  char* s = reinterpret_cast<char*>(W16) + blk * (kLinkBlock * kLinkBytes16);
#pragma unroll
  for (int k = 0; k < 2; ++k)
    reinterpret_cast<uint4*>(s)[k * kLinkBlock + lane] = make_uint4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
  reinterpret_cast<unsigned*>(s + 32 * kLinkBlock)[lane] = h[8];
}

// acc += a b, and acc += a b^dagger
__device__ __forceinline__ void mmac(M3<double>& acc, const M3<double>& a, const M3<double>& b) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) cfma(acc.m[i][j], a.m[i][k], b.m[k][j]);
}
__device__ __forceinline__ void mzero(M3<double>& a) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) a.m[i][j] = C<double>{0.0, 0.0};
}

// One step of a path from the site n + at: U_mu(n + at) or U_mu(n + at - mu)^dagger.
__device__ __forceinline__ M3<double> path_step(const Geom& g, const double2* __restrict__ U64, const SiteCoord& s,
                                                const int at[4], int mu, int sg) {
  int q[4] = {at[0], at[1], at[2], at[3]};
  if (sg < 0) q[mu] -= 1;
  const M3<double> u = load_soa(U64 + (int64_t)mu * 9 * g.V, g.V, displaced(g, s, q[0], q[1], q[2], q[3]));
  return sg > 0 ? u : adj(u);
}

// The stored one-hop links W_{-mu}(n) = U_mu(n - mu)^dagger (offset lists hold
// the stored offsets of one level).
__global__ void stored1_kernel(Geom g, const double2* __restrict__ U64, double2* W64, float2* W32, __nv_bfloat162* W16) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  const SiteCoord s = coords(g, n);
  const int mu = blockIdx.y;
  const int zero[4] = {0, 0, 0, 0};
  int e[4] = {0, 0, 0, 0};
  e[mu] = -1;
  store_link(W64, W32, W16, g.V, n, nu_of(e[0], e[1], e[2], e[3]), path_step(g, U64, s, zero, mu, -1));
}

// Stored k-hop links from the (k-1)-hop ones, one thread per site and offset.
// With AB (two-hop level, clover wanted) the two paths of the offset d =
// s1 e_mu + s2 e_nu, mu < nu, go to AB[2 * entry][9][V] (mu first) and
// AB[2 * entry + 1] (nu first).
__global__ void __launch_bounds__(128) storedk_kernel(Geom g, const double2* __restrict__ U64, double2* W64, float2* W32,
                                                      __nv_bfloat162* W16, LevelList lst, int k, double2* AB) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  const int which = blockIdx.y, nu = lst.nu[which];
  const int d[4] = {nu % 3 - 1, (nu / 3) % 3 - 1, (nu / 9) % 3 - 1, (nu / 27) % 3 - 1};
  const SiteCoord s = coords(g, n);
  M3<double> acc;
  mzero(acc);
  int path = 0;
#pragma unroll 1
  for (int mu = 3; mu >= 0; --mu) {  // last hop; two hops: last hop nu (mu first) comes first
    if (d[mu] == 0) continue;
    int dp[4] = {d[0], d[1], d[2], d[3]};
    dp[mu] = 0;
    const int at = nu_of(dp[0], dp[1], dp[2], dp[3]);
    const int64_t m = at < 40 ? n : displaced(g, s, dp[0], dp[1], dp[2], dp[3]);
    M3<double> w = load_soa(W64 + (int64_t)(at < 40 ? at : 80 - at) * 9 * g.V, g.V, m);
    if (at > 40) w = adj(w);
    const M3<double> u = path_step(g, U64, s, dp, mu, d[mu]);
    if (AB) {
      M3<double> p;
      mzero(p);
      mmac(p, w, u);
      store_soa(AB + (int64_t)(2 * which + path) * 9 * g.V, g.V, n, p);
      madd(acc, p);
      ++path;
    } else {
      mmac(acc, w, u);
    }
  }
  const double inv = 1.0 / k;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) acc.m[i][j] = inv * acc.m[i][j];
  store_link(W64, W32, W16, g.V, n, nu, acc);
}

// ------------------------------------------------------------------ clover
// F_{mu nu}(n), mu < nu: traceless part of (Q - Q^dagger)/(8i), Q the sum of the
// four counter-clockwise plaquette leaves around n in the (mu, nu) plane.  With
// A_d, B_d the two paths of a stored offset (mu first, nu first):
//   Q = A_-(n) B_-(n)^+ + B_-(m)^+ A_-(m) + B_+(n) A_+(n)^+ + A_+(p)^+ B_+(p),
// d_- = (-mu, -nu), m = n + mu + nu, d_+ = (+mu, -nu), p = n + nu - mu.
__device__ __forceinline__ M3<double> field_strength(const Geom& g, const double2* __restrict__ AB, const LevelList& two,
                                                     const SiteCoord& s, int64_t n, int mu, int nu) {
  int em[4] = {0, 0, 0, 0}, ep[4] = {0, 0, 0, 0}, tm[4] = {0, 0, 0, 0}, tp[4] = {0, 0, 0, 0};
  em[mu] = -1; em[nu] = -1; ep[mu] = 1; ep[nu] = -1;
  tm[mu] = 1; tm[nu] = 1; tp[mu] = -1; tp[nu] = 1;
  const int im = nu_of(em[0], em[1], em[2], em[3]), ip = nu_of(ep[0], ep[1], ep[2], ep[3]);
  int km = 0, kp = 0;
  for (int i = 0; i < two.count; ++i) {
    if (two.nu[i] == im) km = i;
    if (two.nu[i] == ip) kp = i;
  }
  auto ld = [&](int entry, int path, int64_t m) { return load_soa(AB + (int64_t)(2 * entry + path) * 9 * g.V, g.V, m); };
  M3<double> q;
  mzero(q);
  mmac(q, ld(km, 0, n), adj(ld(km, 1, n)));
  const int64_t m = displaced(g, s, tm[0], tm[1], tm[2], tm[3]);
  mmac(q, adj(ld(km, 1, m)), ld(km, 0, m));
  mmac(q, ld(kp, 1, n), adj(ld(kp, 0, n)));
  const int64_t p = displaced(g, s, tp[0], tp[1], tp[2], tp[3]);
  mmac(q, adj(ld(kp, 0, p)), ld(kp, 1, p));
  M3<double> f;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // (Q - Q^+)_{ij} / (8i) = -i (Q_ij - conj(Q_ji)) / 8
      const C<double> a = q.m[i][j] - conj(q.m[j][i]);
      f.m[i][j] = C<double>{a.im / 8.0, -a.re / 8.0};
    }
  const C<double> tr = f.m[0][0] + f.m[1][1] + f.m[2][2];
#pragma unroll
  for (int i = 0; i < 3; ++i) f.m[i][i] = f.m[i][i] - (1.0 / 3.0) * tr;
  return f;
}

// Chiral basis: sigma_{jk} = -eps_{jkl} diag(s_l, s_l), sigma_{j4} = diag(s_j, -s_j)
// (s = Pauli, sigma_{mu nu} = (i/2)[gamma_mu, gamma_nu]).  Hence the upper
// (lower) 6x6 block of sum_{mu<nu} sigma_{mu nu} F_{mu nu} is sum_l s_l (x) X_l with
//   X_1 = -F_23 +- F_14,  X_2 = F_13 +- F_24,  X_3 = -F_12 +- F_34:
// [[X_3, X_1 - i X_2], [h.c., -X_3]].  blockIdx.y = 0: the X_3 entries of both
// blocks, 1: the spin-off-diagonal ones.
__global__ void __launch_bounds__(64) clover_kernel(Geom g, const double2* __restrict__ AB, LevelList two, double c_sw,
                                                    double* C64, float* C32) {
  const int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (n >= g.V) return;
  const SiteCoord s = coords(g, n);
  const double pre = -0.5 * c_sw;
  auto put = [&](int blk, int k, double v) {
    C64[((int64_t)blk * 36 + k) * g.V + n] = v;
    C32[clover_at32(n, blk, k)] = (float)v;
  };
  auto at = [](int i, int j) { return 6 + 2 * (i * 5 - i * (i - 1) / 2 + j - i - 1); };  // entry (i, j), i < j
  // S and D: the two blocks' values are S + D and S - D
  M3<double> S, D;
  if (blockIdx.y == 0) {
    S = field_strength(g, AB, two, s, n, 0, 1);  // X_3 = -F_12 +- F_34
    D = field_strength(g, AB, two, s, n, 2, 3);
#pragma unroll
    for (int blk = 0; blk < 2; ++blk)
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b) {
          const double sg = blk == 0 ? 1.0 : -1.0;
          const double re = pre * (sg * D.m[a][b].re - S.m[a][b].re), im = pre * (sg * D.m[a][b].im - S.m[a][b].im);
          if (a == b) {
            put(blk, a, re);
            put(blk, 3 + a, -re);
          } else {
            put(blk, at(a, b), re);
            put(blk, at(a, b) + 1, im);
            put(blk, at(3 + a, 3 + b), -re);
            put(blk, at(3 + a, 3 + b) + 1, -im);
          }
        }
  } else {
    // X_1 - i X_2 = (-F_23 - i F_13) +- (F_14 - i F_24)
    S = field_strength(g, AB, two, s, n, 1, 2);
    M3<double> f = field_strength(g, AB, two, s, n, 0, 2);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) S.m[a][b] = C<double>{-S.m[a][b].re + f.m[a][b].im, -S.m[a][b].im - f.m[a][b].re};
    D = field_strength(g, AB, two, s, n, 0, 3);
    f = field_strength(g, AB, two, s, n, 1, 3);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) D.m[a][b] = C<double>{D.m[a][b].re + f.m[a][b].im, D.m[a][b].im - f.m[a][b].re};
#pragma unroll
    for (int blk = 0; blk < 2; ++blk)
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const double sg = blk == 0 ? 1.0 : -1.0;
          put(blk, at(a, 3 + b), pre * (S.m[a][b].re + sg * D.m[a][b].re));
          put(blk, at(a, 3 + b) + 1, pre * (S.m[a][b].im + sg * D.m[a][b].im));
        }
  }
}

// Caller layout [V][40][3][3] from the element planes, 32 sites x 40 elements at
// a time through shared memory so that both sides are contiguous.
__global__ void __launch_bounds__(256) export_links_kernel(Geom g, const double2* __restrict__ W64, double2* out) {
  __shared__ double2 t[40][33];
  const int64_t n0 = blockIdx.x * (int64_t)32;
  const int k0 = blockIdx.y * 40;
  const int m = (int)min((int64_t)32, g.V - n0);
  for (int i = threadIdx.x; i < 40 * 32; i += 256) {
    const int k = i / 32, l = i % 32;
    if (l < m) t[k][l] = W64[(int64_t)(k0 + k) * g.V + n0 + l];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 40 * m; i += 256) {
    const int l = i / 40, k = i - 40 * l;
    out[(n0 + l) * 360 + k0 + k] = t[k][l];
  }
}

}  // namespace

int build_transporters(bri_ctx* c, double2* T) {
  const Geom& g = c->g;
  const int64_t V = g.V;
  cudaStream_t st = c->stream;
  const int th = 128;
  level1_kernel<<<blocks_for(V, th), th, 0, st>>>(g, c->U64, T); note_launch();
  for (int k = 2; k <= 4; ++k) {
    LevelList lst = level_list(k);
    dim3 grid(blocks_for(V, th), lst.count);
    levelk_kernel<<<grid, th, 0, st>>>(g, c->U64, T, lst, k); note_launch();
  }
  BRI_LAUNCH_CHECK("link construction kernels");
  return BRI_OK;
}

int launch_build_links(bri_ctx* c, const double* U, double c_sw) {
  const Geom& g = c->g;
  const int64_t V = g.V;
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
  // Everything is allocated before the first write: without memory for a rebuild the
  // links and clover of the last one stay as they were.
  int rc;
  if ((rc = alloc((void**)&c->W64, sizeof(double2) * 360 * V))) return rc;
  if ((rc = alloc((void**)&c->W32, kLinkBytes32 * kLinkBlock * 40 * link_blocks(V)))) return rc;
  if ((rc = alloc((void**)&c->W16, kLinkBytes16 * kLinkBlock * 40 * link_blocks(V)))) return rc;
  if ((rc = alloc((void**)&c->U64, sizeof(double2) * 36 * V))) return rc;
  if ((rc = alloc((void**)&c->U32, kLinkBytes32 * kLinkBlock * 4 * link_blocks(V)))) return rc;
  // the two paths of every stored two-hop offset, kept for the clover leaves
  LevelList two = stored_level(2);
  double2* AB = nullptr;
  if (c_sw != 0.0) {
    if ((rc = alloc((void**)&c->C64, sizeof(double) * 72 * V))) return rc;
    if ((rc = alloc((void**)&c->C32, sizeof(float4) * clover_words32(V)))) return rc;
    const cudaError_t e = scratch_alloc((void**)&AB, sizeof(double2) * 9 * 2 * two.count * V, st);
    if (e != cudaSuccess) return cuda_fail(e, "bri_build_links: cudaMallocAsync");
  }
  // no operator runs on what a failure from here on leaves behind
  c->have_links = false;
  c->have_clover = false;
  c->dw_valid = false;
  c->c_sw = c_sw;
  const int th = 128;
  thin_links_kernel<<<blocks_for(V, th), th, 0, st>>>(g, (const double2*)U, c->U64, c->U32,
                                                       (c->flags & BRI_ANTIPERIODIC_T) ? 1 : 0); note_launch();
  stored1_kernel<<<dim3(blocks_for(V, th), 4), th, 0, st>>>(g, c->U64, c->W64, c->W32, c->W16); note_launch();
  for (int k = 2; k <= 4; ++k) {
    const LevelList lst = stored_level(k);
    storedk_kernel<<<dim3(blocks_for(V, th), lst.count), th, 0, st>>>(g, c->U64, c->W64, c->W32, c->W16, lst, k,
                                                                     k == 2 ? AB : nullptr);
    note_launch();
  }
  if (AB) {
    clover_kernel<<<dim3(blocks_for(V, 64), 2), 64, 0, st>>>(g, AB, two, c_sw, c->C64, c->C32); note_launch();
    cudaFreeAsync(AB, st);
    c->have_clover = true;
  }
  BRI_LAUNCH_CHECK("link construction kernels");
  BRI_CUDA(cudaStreamSynchronize(st));
  c->have_links = true;
  return BRI_OK;
}

int launch_export_links(bri_ctx* c, double* W) {
  export_links_kernel<<<dim3(blocks_for(c->g.V, 32), 9), 256, 0, c->stream>>>(c->g, c->W64, (double2*)W); note_launch();
  BRI_LAUNCH_CHECK("export_links_kernel");
  return BRI_OK;
}

}  // namespace bri
