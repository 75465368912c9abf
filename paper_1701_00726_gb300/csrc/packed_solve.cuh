// Multi-shift CG on packed FP32 vectors (included by mscg.cu): one or several
// lattices' systems, each a packed vector of one right-hand side (bri_pair.cuh;
// as pairs the two stencils of an iteration took 381 + 363 us for 4 systems of
// 16^3 x 32 where single ones take 349 + 351).  Base direction p_0, t = D p_0,
// q = (A + sigma) p_0 and the residuals live in the stencil's layout; per iteration
//   t = D p, q = D^dagger t + sigma p with the partials of <p, q>,   (stencil)
//   alpha; r_{j+1} = r_j - alpha q_j with the partials of ||r||^2;   (3 vectors)
//   beta; p = r + beta p, and for a single shift x += alpha p first. (3 or 5)
// With several shifts the residuals of eight iterations stay in a ring, and
// every DW = 4 iterations kp_flush advances all shifted directions (the base
// shift's is a lagging copy) and the FP64 solutions from it, in the order and
// with the operations of the per-iteration form.
#pragma once

constexpr int kRing = 8;  // residual slots; also the iterations of one graph block

// One system of the problem, on lattice lat.
struct PackedSys {
  int lat;
  int64_t V;
  int64_t poff;        // offset in the packed vectors, 16-byte words
  int64_t offn, kstr;  // complex offset of its shift 0 in p and x, and from shift to shift
};

__global__ void __launch_bounds__(256) kp_norm(const PackedSys* __restrict__ gd, const float4* __restrict__ r, double* part) {
  const PackedSys g = gd[blockIdx.y];
  const int64_t nw = packed_words(g.V, 6);
  const float4* v = r + g.poff;
  double a = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 x = v[i];
    a += (double)x.x * x.x + (double)x.y * x.y + (double)x.z * x.z + (double)x.w * x.w;
  }
  const double t = block_sum(a);
  if (threadIdx.x == 0) part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
}

// rout = rin - alpha q, partials of ||rout||^2 (rin may be rout).  The squares of four words are summed in
// three FP32 words (sum3.cuh, scaled by the residual's norm so far) and those sums in FP64.  Bound by HBM: 174 us
// on average in the 24^3 x 48 solves of 4 rhs, 91 % of the copy rate.  FP64 squares bound it instead (102 us on
// average in the 16^3 x 32 solves against 43 with two FP32 words, which kept only 2^-47 and FP32's range); the third
// word costs the whole solve 0.4 %.
__global__ void __launch_bounds__(256) kp_update_r(const PackedSys* __restrict__ gd, const MsState* __restrict__ st,
                                                   const float4* __restrict__ q, const float4* rin, float4* rout, double* part) {
  const PackedSys g = gd[blockIdx.y];
  if (st[blockIdx.y].done) return;
  const float2 f = pr_bc(-(float)st[blockIdx.y].alpha);
  const int k2 = unit_exponent(st[blockIdx.y].rr);
  const float2 sc = pr_bc(exp2_float(k2));
  const int64_t nw = packed_words(g.V, 6), stride = (int64_t)gridDim.x * blockDim.x;
  const float4 *qv = q + g.poff, *ri = rin + g.poff;
  float4* ro = rout + g.poff;
  double a = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += 4 * stride) {
    float4 x[4], v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * stride < nw) {
        x[k] = __ldg(qv + i + k * stride);
        v[k] = ri[i + k * stride];
      }
    Sum3 sum = sum3_zero();
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * stride < nw) {
        const float2 re = __ffma2_rn(f, make_float2(x[k].x, x[k].y), make_float2(v[k].x, v[k].y));
        const float2 im = __ffma2_rn(f, make_float2(x[k].z, x[k].w), make_float2(v[k].z, v[k].w));
        ro[i + k * stride] = make_float4(re.x, re.y, im.x, im.y);
        const float2 u = __fmul2_rn(re, sc), v = __fmul2_rn(im, sc);
        sum3_add(sum, u, u);
        sum3_add(sum, v, v);
      }
    a += sum3_total(sum);
  }
  const double t = block_sum(a);
  if (threadIdx.x == 0) part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = t * exp2_square(k2);
}

// x += alpha p (XUP: single-shift solves, also in the iteration that converged),
// p = r + beta p.
template <bool XUP>
__global__ void __launch_bounds__(256) kp_update_p(const PackedSys* __restrict__ gd, const MsState* __restrict__ st,
                                                   const float4* __restrict__ r, float4* p, float4* x) {
  const PackedSys g = gd[blockIdx.y];
  const MsState& A = st[blockIdx.y];
  const bool up = !A.done, xup = XUP && A.pend;
  if (!(up || xup)) return;
  const float b = (float)A.b_s[0], a = xup ? (float)A.a_s[0] : 0.f;
  const int64_t nw = packed_words(g.V, 6);
  const float4* rv = r + g.poff;
  float4 *pv = p + g.poff, *xv = x + g.poff;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = pv[i];
    if constexpr (XUP) {
      const float4 s = xv[i];
      xv[i] = make_float4(fmaf(a, v.x, s.x), fmaf(a, v.y, s.y), fmaf(a, v.z, s.z), fmaf(a, v.w, s.w));
    }
    if (up) {
      const float4 w = rv[i];
      pv[i] = make_float4(fmaf(b, v.x, w.x), fmaf(b, v.y, w.y), fmaf(b, v.z, w.z), fmaf(b, v.w, w.w));
    }
  }
}

// The coefficients of a window, staged per system in shared memory: the shifts
// that took part (compacted) and their steps.
struct FlushCoef {
  float z[DW][NS], b[DW][NS];
  double a[DW][NS];
  unsigned char act[DW][NS];
  int k[NS], first[DW], nk, n;
};
__device__ __forceinline__ void load_flush_coef(FlushCoef& c, const ShiftHist& h) {
  // one thread per shift: position = number of participating shifts below it
  const int k = threadIdx.x;
  if (k < 32) {
    int any = 0;
    for (int m = 0; m < h.n; ++m) any |= h.act[m][k];
    const unsigned mask = __ballot_sync(0xffffffffu, any);
    const int at = __popc(mask & ((1u << k) - 1));
    if (any) {
      c.k[at] = k;
      for (int m = 0; m < h.n; ++m) {
        c.z[m][at] = h.z[m][k];
        c.b[m][at] = h.b[m][k];
        c.a[m][at] = h.a[m][k];
        c.act[m][at] = h.act[m][k];
      }
    }
    if (k == 0) {
      c.nk = __popc(mask);
      c.n = h.n;
      for (int m = 0; m < h.n; ++m) c.first[m] = h.first[m];
    }
  }
}

// The recorded steps of one system for two of its complex numbers (p and x at
// complex offset o + k kstr and o1 beyond), residuals r[m].
__device__ __forceinline__ void flush_system(const FlushCoef& c, const float2 (&ra)[DW], const float2 (&rb)[DW], float2* p,
                                             double2* x, int64_t o, int64_t o1, int64_t kstr) {
  const bool first = c.first[0];  // p_i = b = r_0 before the first step
  float2 na = ra[0], nb = rb[0];
  double2 nxa, nxb;
  auto fetch = [&](int j) {
    const int64_t at = o + c.k[j] * kstr, bt = at + o1;
    if (!first) {
      na = p[at];
      nb = p[bt];
    }
    nxa = x[at];
    nxb = x[bt];
  };
  if (c.nk > 0) fetch(0);
  for (int j = 0; j < c.nk; ++j) {
    const int64_t at = o + c.k[j] * kstr, bt = at + o1;
    float2 pa = na, pb = nb;
    double2 xa = nxa, xb = nxb;
    if (j + 1 < c.nk) fetch(j + 1);  // the next shift's vectors are under way during this one's arithmetic
#pragma unroll
    for (int m = 0; m < DW; ++m) {
      if (m >= c.n || !c.act[m][j]) continue;
      if (!c.first[m]) {
        const float z = c.z[m][j], b = c.b[m][j];
        pa.x = fmaf(b, pa.x, z * ra[m].x);
        pa.y = fmaf(b, pa.y, z * ra[m].y);
        pb.x = fmaf(b, pb.x, z * rb[m].x);
        pb.y = fmaf(b, pb.y, z * rb[m].y);
      }
      const double a = c.a[m][j];
      xa.x = fma(a, (double)pa.x, xa.x);
      xa.y = fma(a, (double)pa.y, xa.y);
      xb.x = fma(a, (double)pb.x, xb.x);
      xb.y = fma(a, (double)pb.y, xb.y);
    }
    p[at] = pa;
    p[bt] = pb;
    x[at] = xa;
    x[bt] = xb;
  }
}

// Every shift's recorded steps (ring slots base, base + 1, ...), in order:
// p_i = zeta_i r_m + beta_i p_i (not on the first iteration), x_i += alpha_i p_i.
// Runs while a system may already be done (its last steps still pending).  One
// thread per site and packed word (two spins), neighbouring threads on one site,
// so that p and x stream; the ring is read in rows of five to six sites.
__global__ void __launch_bounds__(256) kp_flush(const PackedSys* __restrict__ gd, const ShiftHist* __restrict__ hist,
                                                const float4* __restrict__ ring, int64_t rstride, int base, float2* p,
                                                double2* x) {
  const PackedSys g = gd[blockIdx.y];
  __shared__ FlushCoef c;
  load_flush_coef(c, hist[blockIdx.y]);
  __syncthreads();
  const int nm = c.n;
  if (nm == 0) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.V * 6; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = i / 6;
    const int q = (int)(i - n * 6);
    float2 a0[DW], a1[DW];
    const float4* rr = ring + g.poff + packed_at<6>((int)n) + q * kPackBlock;
#pragma unroll
    for (int m = 0; m < DW; ++m)
      if (m < nm) {
        const float4 u = __ldg(rr + (int64_t)((base + m) % kRing) * rstride);
        a0[m] = make_float2(u.x, u.z);
        a1[m] = make_float2(u.y, u.w);
      }
    flush_system(c, a0, a1, p, x, g.offn + n * 12 + q + 3 * (q / 3), 3, g.kstr);
  }
}

// Stencil on the systems of one lattice, the systems of a site block next to each
// other (stencil_grid); converged systems are skipped, not only the trailing ones
// that the host has dropped at its last look.
template <typename LS, bool EPI, int KS>
__global__ void __launch_bounds__(128, 4)
    kp_stencil(Geom g, const MsState* __restrict__ st, float4* __restrict__ Y, const float4* __restrict__ X,
               const LS* __restrict__ W, const float* __restrict__ cl, float diag, int gfirst,
               const __grid_constant__ PairHops<float> H, PackedDot sd) {
  const int s = gfirst ? blockIdx.x : blockIdx.y, blk = gfirst ? blockIdx.y : blockIdx.x;
  if (st[s].done) return;
  const int64_t o = s * packed_words(g.V, 6);
  pr_block<2, LS, 1, EPI ? 1 : 0, KS>(g, blk, nullptr, Y + o, X + o, W, cl, diag, H, sd, o, s, gfirst ? gridDim.y : gridDim.x);
}

// Stencil on the work list of several lattices: item (system, block of 128 / KS
// sites); converged systems are skipped.
template <typename LS, bool EPI, int KS>
__global__ void __launch_bounds__(128, 4)
    kb_pair(const __grid_constant__ BatchTab T, const PackedSys* __restrict__ gd, const int2* __restrict__ items,
            const MsState* __restrict__ st, float4* __restrict__ Y, const float4* __restrict__ X,
            const __grid_constant__ PairHops<float> H, PackedDot sd, int nb) {
  const int2 it = items[blockIdx.x];
  const PackedSys gr = gd[it.x];
  if (st[it.x].done) return;
  const BatchLat& L = T.lat[gr.lat];
  pr_block<2, LS, 1, EPI ? 2 : 0, KS>(L.g, it.y, nullptr, Y + gr.poff, X + gr.poff, (const LS*)L.W, (const float*)L.C, (float)L.diag,
                                     H, sd, gr.poff, it.x, nb, EPI ? unit_exponent(st[it.x].rr) : 0);
}

// A problem on packed vectors: `words` 16-byte words per packed vector.
struct PackedProblem {
  std::vector<PackedSys> sys;
  int nsys = 0, nshift = 0, maxiter = 0;
  int64_t words = 0;
  std::vector<double> sig;  // [nsys][nshift], increasing within a system
  std::vector<double> tol;  // [nsys]
};

// Solves (A + sig[s][k]) x[k][s] = b[s].  pack(dst) writes the packed right-hand
// sides; apply(dagger, X, Y, P, na) enqueues Y = D X (P null) or Y = D^dagger X +
// sigma P with partials [na][blocks(na)] in sdpart, for the first na systems.
// Several shifts: solutions in x64 (zeroed here).  One shift: packed in xp.
// whole: all iterations in one WHILE-node graph (no host polling), else host
// polling every kRing iterations and a shrinking prefix of systems.  all_iters: the
// systems' iterations in all.
template <typename Pack, typename Apply, typename Blocks>
int packed_solve(cudaStream_t st, const PackedProblem& pb, Pack&& pack, Apply&& apply, double* sdpart, Blocks&& blocks,
                 double2* x64, size_t x64_bytes, float4* xp, bool whole, bool graphs, int* hdone,
                 int* iters_out, Counters* cnt, double* lam_out, const MsState** state_out = nullptr,
                 int64_t* all_iters = nullptr) {
  const int nsys = pb.nsys, nshift = pb.nshift;
  const bool defer = x64 != nullptr;
  const size_t vb = sizeof(float4) * (size_t)pb.words;
  int64_t maxw = 0, n2all = 0;
  for (const PackedSys& g : pb.sys) {
    maxw = std::max(maxw, packed_words(g.V, 6));
    n2all += g.V * 12;
  }
  // Reductions: four words per thread in flight (kp_update_r), but two blocks per SM
  // as long as there is a word for every thread; partials as everywhere.  8^3 x 16,
  // 12 systems: 24 us with 170 blocks per system, 12 with 48.
  const int64_t one = (maxw + 255) / 256, four = (maxw + 1023) / 1024;
  const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>(std::max(four, std::min<int64_t>(one, 304 / nsys)),
                                                               std::max(1, kMaxPartials / nsys)));
  // the other vector kernels: a word per thread, so that no block has a round more than the next
  const int nvec = (int)std::min<int64_t>(one, 65536);
  DevBuf bgd, bst, bpart, bring, bP, bT, bQ, bpk, bhist, bflags;
  int rc;
  if ((rc = bgd.alloc(sizeof(PackedSys) * nsys, st))) return rc;
  if ((rc = bst.alloc(sizeof(MsState) * nsys, st))) return rc;
  if ((rc = bpart.alloc(sizeof(double) * nblk * nsys, st))) return rc;
  if ((rc = bring.alloc(vb * (defer ? kRing : 1), st))) return rc;
  if ((rc = bP.alloc(vb, st))) return rc;
  if ((rc = bT.alloc(vb, st))) return rc;
  if ((rc = bQ.alloc(vb, st))) return rc;
  if (defer && (rc = bpk.alloc(sizeof(float2) * n2all * nshift, st))) return rc;
  if (defer && (rc = bhist.alloc(sizeof(ShiftHist) * nsys, st))) return rc;
  if ((rc = bflags.alloc(sizeof(int) * nsys, st))) return rc;
  const PackedSys* gd = bgd.as<PackedSys>();
  MsState* S = bst.as<MsState>();
  ShiftHist* hist = defer ? bhist.as<ShiftHist>() : nullptr;
  double* part = bpart.as<double>();
  if (state_out) *state_out = S;
  float4 *ring = bring.as<float4>(), *P = bP.as<float4>(), *T = bT.as<float4>(), *Q = bQ.as<float4>();
  std::vector<MsState> hs(nsys);
  for (int s = 0; s < nsys; ++s) {
    MsState& h = hs[s];
    memset(&h, 0, sizeof(h));
    h.nshift = nshift;
    h.sig_base = pb.sig[(size_t)s * nshift];
    for (int k = 0; k < nshift; ++k) h.delta[k] = pb.sig[(size_t)s * nshift + k] - h.sig_base;
    h.tol2 = pb.tol[s] * pb.tol[s];
    h.maxiter = pb.maxiter;
  }
  BRI_CUDA(cudaMemcpyAsync(bgd.p, pb.sys.data(), sizeof(PackedSys) * nsys, cudaMemcpyHostToDevice, st));
  BRI_CUDA(cudaMemcpyAsync(S, hs.data(), sizeof(MsState) * nsys, cudaMemcpyHostToDevice, st));
  // rows of the sites that pad a volume to whole blocks stay zero in every vector
  for (float4* v : {ring, P, T, Q}) BRI_CUDA(cudaMemsetAsync(v, 0, v == ring ? vb * (defer ? kRing : 1) : vb, st));
  if (defer) {
    BRI_CUDA(cudaMemsetAsync(hist, 0, sizeof(ShiftHist) * nsys, st));
    BRI_CUDA(cudaMemsetAsync(x64, 0, x64_bytes, st));
  } else {
    BRI_CUDA(cudaMemsetAsync(xp, 0, vb, st));
  }
  if ((rc = pack(ring))) return rc;
  BRI_CUDA(cudaMemcpyAsync(P, ring, vb, cudaMemcpyDeviceToDevice, st));
  kp_norm<<<dim3(nblk, nsys), 256, 0, st>>>(gd, ring, part); note_launch();
  k_scalar_init<<<nsys, RED_THREADS, 0, st>>>(S, part, nblk); note_launch();
  BRI_LAUNCH_CHECK("packed multi-shift init");

  // `count` iterations from ring slot 0 on (every block of iterations starts there)
  auto enqueue = [&](int na, int count) -> int {
    int q;
    for (int j = 0; j < count; ++j) {
      if ((q = apply(0, P, T, (const float4*)nullptr, na))) return q;
      if ((q = apply(1, T, Q, (const float4*)P, na))) return q;
      k_scalar_alpha<<<na, RED_THREADS, 0, st>>>(S, sdpart, blocks(na), hist, defer && j % DW == 0, 1); note_launch();
      float4 *rin = defer ? ring + (j % kRing) * pb.words : ring, *rout = defer ? ring + ((j + 1) % kRing) * pb.words : ring;
      kp_update_r<<<dim3(nblk, na), 256, 0, st>>>(gd, S, Q, rin, rout, part); note_launch();
      k_scalar_beta<<<na, RED_THREADS, 0, st>>>(S, part, nblk); note_launch();
      if (defer) kp_update_p<false><<<dim3(nvec, na), 256, 0, st>>>(gd, S, rout, P, nullptr);
      else kp_update_p<true><<<dim3(nvec, na), 256, 0, st>>>(gd, S, rout, P, xp);
      note_launch();
      if (defer && ((j + 1) % DW == 0 || j == count - 1)) {
        kp_flush<<<dim3(nvec, na), 256, 0, st>>>(gd, hist, ring, pb.words, j / DW * DW, bpk.as<float2>(), x64);
        note_launch();
      }
    }
    return BRI_OK;
  };

  if (whole) {
    cudaGraph_t graph = nullptr;
    BRI_CUDA(cudaGraphCreate(&graph, 0));
    cudaGraphExec_t gexec = nullptr;
    auto fail = [&](cudaError_t e, const char* where) {
      if (gexec) cudaGraphExecDestroy(gexec);
      cudaGraphDestroy(graph);
      return cuda_fail(e, where);
    };
    cudaGraphConditionalHandle handle;
    cudaError_t e = cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return fail(e, "packed multi-shift: conditional handle");
    // (the parameter union has no default constructor: zeroed storage instead)
    alignas(cudaGraphNodeParams) unsigned char cp_raw[sizeof(cudaGraphNodeParams)];
    memset(cp_raw, 0, sizeof(cp_raw));
    cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(cp_raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = handle;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp);
    if (e != cudaSuccess) return fail(e, "packed multi-shift: conditional node");
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    const long long l0 = bri_kernel_launches();
    e = cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return fail(e, "packed multi-shift: capture");
    const int erc = enqueue(nsys, kRing);
    kb_while<<<1, 32, 0, st>>>(handle, S, nsys); note_launch();
    e = cudaStreamEndCapture(st, &body);
    const long long per_body = bri_kernel_launches() - l0;
    if (erc) {
      cudaGraphDestroy(graph);
      return erc;
    }
    if (e != cudaSuccess) return fail(e, "packed multi-shift: end capture");
    e = cudaGraphInstantiate(&gexec, graph, 0);
    if (e != cudaSuccess) return fail(e, "packed multi-shift: instantiate");
    e = cudaGraphLaunch(gexec, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), S, sizeof(MsState) * nsys, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaGraphExecDestroy(gexec);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return cuda_fail(e, "packed multi-shift: graph run");
    int maxit = 0;
    for (const MsState& h : hs) maxit = std::max(maxit, h.iters);
    note_launches(per_body * (std::max(1, (maxit + kRing - 1) / kRing) - 1));
    cnt->matvecs += 2 * maxit;
  } else {
    int it = 0, nact = nsys, g_nact = -1;
    cudaGraphExec_t gexec = nullptr;
    struct ExecGuard {
      cudaGraphExec_t& e;
      ~ExecGuard() {
        if (e) cudaGraphExecDestroy(e);
      }
    } guard{gexec};
    long long g_launches = 0;
    while (nact > 0 && it < pb.maxiter) {
      const int count = std::min(kRing, pb.maxiter - it);
      if (graphs && it > 0 && count == kRing) {
        if (g_nact != nact) {
          if (gexec) cudaGraphExecDestroy(gexec);
          gexec = nullptr;
          cudaGraph_t graph = nullptr;
          const long long l0 = bri_kernel_launches();
          BRI_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
          const int erc = enqueue(nact, count);
          const cudaError_t ce = cudaStreamEndCapture(st, &graph);
          g_launches = bri_kernel_launches() - l0;
          if (erc) {
            if (graph) cudaGraphDestroy(graph);
            return erc;
          }
          if (ce != cudaSuccess) return cuda_fail(ce, "packed multi-shift: graph capture");
          const cudaError_t ie = cudaGraphInstantiate(&gexec, graph, 0);
          cudaGraphDestroy(graph);
          if (ie != cudaSuccess) return cuda_fail(ie, "packed multi-shift: graph instantiate");
          g_nact = nact;
        } else {
          note_launches(g_launches);
        }
        BRI_CUDA(cudaGraphLaunch(gexec, st));
      } else if ((rc = enqueue(nact, count))) {
        return rc;
      }
      cnt->matvecs += 2 * count;
      it += count;
      BRI_LAUNCH_CHECK("packed multi-shift iteration");
      k_gather_done<<<1, 256, 0, st>>>(S, nsys, bflags.as<int>()); note_launch();
      BRI_CUDA(cudaMemcpyAsync(hdone, bflags.as<int>(), sizeof(int) * nsys, cudaMemcpyDeviceToHost, st));
      BRI_CUDA(cudaStreamSynchronize(st));
      while (nact > 0 && hdone[nact - 1]) --nact;
    }
    BRI_CUDA(cudaMemcpyAsync(hs.data(), S, sizeof(MsState) * nsys, cudaMemcpyDeviceToHost, st));
    BRI_CUDA(cudaStreamSynchronize(st));
  }
  int maxit = 0, err = 0, notconv = 0;
  double lm = 0.0;
  for (const MsState& h : hs) {
    maxit = std::max(maxit, h.iters);
    err |= h.error;
    if (h.active[0] && !h.error) notconv = 1;
    lm = std::max(lm, h.lam_max - h.sig_base);
  }
  *iters_out = maxit;
  if (all_iters) {
    *all_iters = 0;
    for (const MsState& h : hs) *all_iters += h.iters;
  }
  if (lam_out) *lam_out = lm;
  if (err) {
    set_error("multi-shift CG: non-finite or non-positive curvature in a reduction");
    return BRI_ERR_NONFINITE;
  }
  return notconv ? BRI_NOT_CONVERGED : BRI_OK;
}
