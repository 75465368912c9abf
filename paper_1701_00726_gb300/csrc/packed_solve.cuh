// Multi-shift CG on packed FP32 vectors (included by mscg.cu): one or several
// lattices as groups of packed systems (bri_pair.cuh).  Base direction p_0,
// t = D p_0, q = (A + sigma) p_0 and the residuals live in the stencil's layout;
// per iteration
//   t = D p, q = D^dagger t + sigma p with the partials of <p, q>,   (stencil)
//   alpha; r_{j+1} = r_j - alpha q_j with the partials of ||r||^2;   (3 vectors)
//   beta; p = r + beta p, and for a single shift x += alpha p first. (3 or 5)
// With several shifts the residuals of eight iterations stay in a ring, and
// every DW = 4 iterations kp_flush advances all shifted directions (the base
// shift's is a lagging copy) and the FP64 solutions from it, in the order and
// with the operations of the per-iteration form.
#pragma once

constexpr int kRing = 8;  // residual slots; also the iterations of one graph block

// One group of the problem: systems s0 (and s0 + 1 when two), lattice lat.
struct GroupDesc {
  int s0, two, lat, pad;
  int64_t V;
  int64_t poff;        // offset of the group in the packed vectors, 16-byte words
  int64_t offn, kstr;  // complex offset of system s0's shift 0 in p and x, and from shift to shift
};

__device__ __forceinline__ int64_t group_words(const GroupDesc& g) { return packed_words(g.V, g.two ? 12 : 6); }

// partial sums of the two components of a group's words (a pair: one system
// each, a single right-hand side: both its own)
__device__ __forceinline__ void group_partials(const GroupDesc& g, double* part, double a, double b) {
  const double t = block_sum(g.two ? a : a + b);
  if (threadIdx.x == 0) part[(int64_t)g.s0 * gridDim.x + blockIdx.x] = t;
  if (g.two) {
    __syncthreads();
    const double u = block_sum(b);
    if (threadIdx.x == 0) part[(int64_t)(g.s0 + 1) * gridDim.x + blockIdx.x] = u;
  }
}

__global__ void __launch_bounds__(256) kp_norm(const GroupDesc* __restrict__ gd, const float4* __restrict__ r, double* part) {
  const GroupDesc g = gd[blockIdx.y];
  const int64_t nw = group_words(g);
  const float4* v = r + g.poff;
  double a = 0.0, b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 x = v[i];
    a += (double)x.x * x.x + (double)x.z * x.z;
    b += (double)x.y * x.y + (double)x.w * x.w;
  }
  group_partials(g, part, a, b);
}

// (h, l) += v^2 on two components: exact square and sum by TwoProduct and TwoSum
// (bri_dw.cu), their errors collected in l.
__device__ __forceinline__ void add_square(float2& h, float2& l, float2 v) {
  const float2 p = __fmul2_rn(v, v);
  const float2 e = __ffma2_rn(v, v, pr_neg(p));
  const float2 s = __fadd2_rn(h, p);
  const float2 bb = __fadd2_rn(s, pr_neg(h));
  const float2 t = __fadd2_rn(__fadd2_rn(h, pr_neg(__fadd2_rn(s, pr_neg(bb)))), __fadd2_rn(p, pr_neg(bb)));
  h = s;
  l = __fadd2_rn(l, __fadd2_rn(t, e));
}

// rout = rin - alpha q, partials of ||rout||^2 (rin may be rout).  A converged
// system of a pair keeps its residual.  The squares of four words are summed in
// double-word FP32 (48 bits), those sums in FP64: one FP64 addition per eight
// squares instead of eight, which bound the kernel (102 -> 43 us on average in the
// 16^3 x 32 solves; the random 2^-47 of a chunk vanish below 2^-53 in the sum).
__global__ void __launch_bounds__(256) kp_update_r(const GroupDesc* __restrict__ gd, const MsState* __restrict__ st,
                                                   const float4* __restrict__ q, const float4* rin, float4* rout, double* part) {
  const GroupDesc g = gd[blockIdx.y];
  const int sb = g.two ? g.s0 + 1 : g.s0;
  if (st[g.s0].done && st[sb].done) return;
  const float2 f = make_float2(st[g.s0].done ? 0.f : -(float)st[g.s0].alpha, st[sb].done ? 0.f : -(float)st[sb].alpha);
  const int64_t nw = group_words(g), stride = (int64_t)gridDim.x * blockDim.x;
  const float4 *qv = q + g.poff, *ri = rin + g.poff;
  float4* ro = rout + g.poff;
  double a = 0.0, b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += 4 * stride) {
    float4 x[4], v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * stride < nw) {
        x[k] = __ldg(qv + i + k * stride);
        v[k] = ri[i + k * stride];
      }
    float2 h = make_float2(0.f, 0.f), l = h;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * stride < nw) {
        const float2 re = __ffma2_rn(f, make_float2(x[k].x, x[k].y), make_float2(v[k].x, v[k].y));
        const float2 im = __ffma2_rn(f, make_float2(x[k].z, x[k].w), make_float2(v[k].z, v[k].w));
        ro[i + k * stride] = make_float4(re.x, re.y, im.x, im.y);
        add_square(h, l, re);
        add_square(h, l, im);
      }
    a += (double)h.x + (double)l.x;
    b += (double)h.y + (double)l.y;
  }
  group_partials(g, part, a, b);
}

// x += alpha p (XUP: single-shift solves, also in the iteration that converged),
// p = r + beta p.
template <bool XUP>
__global__ void __launch_bounds__(256) kp_update_p(const GroupDesc* __restrict__ gd, const MsState* __restrict__ st,
                                                   const float4* __restrict__ r, float4* p, float4* x) {
  const GroupDesc g = gd[blockIdx.y];
  const MsState &A = st[g.s0], &B = st[g.two ? g.s0 + 1 : g.s0];
  const bool ua = !A.done, ub = !B.done, xa = XUP && A.pend, xb = XUP && B.pend;
  if (!(ua || ub || xa || xb)) return;
  const float ba = (float)A.b_s[0], bb = (float)B.b_s[0];
  const float aa = xa ? (float)A.a_s[0] : 0.f, ab = xb ? (float)B.a_s[0] : 0.f;
  const int64_t nw = group_words(g);
  const float4* rv = r + g.poff;
  float4 *pv = p + g.poff, *xv = x + g.poff;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x) {
    float4 v = pv[i];
    if constexpr (XUP) {
      float4 s = xv[i];
      s.x = fmaf(aa, v.x, s.x);
      s.y = fmaf(ab, v.y, s.y);
      s.z = fmaf(aa, v.z, s.z);
      s.w = fmaf(ab, v.w, s.w);
      xv[i] = s;
    }
    const float4 w = rv[i];
    if (ua) {
      v.x = fmaf(ba, v.x, w.x);
      v.z = fmaf(ba, v.z, w.z);
    }
    if (ub) {
      v.y = fmaf(bb, v.y, w.y);
      v.w = fmaf(bb, v.w, w.w);
    }
    pv[i] = v;
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
// thread per site and 16-byte word of the spinors' own layout, so that p and x
// stream; the ring is read in rows of five to six sites.
__global__ void __launch_bounds__(256) kp_flush(const GroupDesc* __restrict__ gd, const ShiftHist* __restrict__ hist,
                                                const float4* __restrict__ ring, int64_t rstride, int base, float2* p,
                                                double2* x) {
  const GroupDesc g = gd[blockIdx.y];
  __shared__ FlushCoef ca, cb;
  load_flush_coef(ca, hist[g.s0]);
  if (g.two) load_flush_coef(cb, hist[g.s0 + 1]);
  __syncthreads();
  const int na = ca.n, nb = g.two ? cb.n : 0, nmax = max(na, nb);
  if (nmax == 0) return;
  const int64_t n2 = g.V * 12;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < g.V * 6; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = i / 6;
    const int q = (int)(i - n * 6);
    float2 a0[DW], a1[DW], b0[DW], b1[DW];
    if (g.two) {
      const float4* rr = ring + g.poff + packed_at<12>((int)n) + 2 * q * kPackBlock;
#pragma unroll
      for (int m = 0; m < DW; ++m)
        if (m < nmax) {
          const float4* rs = rr + (int64_t)((base + m) % kRing) * rstride;
          const float4 u = __ldg(rs), v = __ldg(rs + kPackBlock);
          a0[m] = make_float2(u.x, u.z);
          b0[m] = make_float2(u.y, u.w);
          a1[m] = make_float2(v.x, v.z);
          b1[m] = make_float2(v.y, v.w);
        }
      const int64_t o = g.offn + 2 * i;
      flush_system(ca, a0, a1, p, x, o, 1, g.kstr);
      flush_system(cb, b0, b1, p, x, o + n2, 1, g.kstr);
    } else {
      const float4* rr = ring + g.poff + packed_at<6>((int)n) + q * kPackBlock;
#pragma unroll
      for (int m = 0; m < DW; ++m)
        if (m < nmax) {
          const float4 u = __ldg(rr + (int64_t)((base + m) % kRing) * rstride);
          a0[m] = make_float2(u.x, u.z);
          a1[m] = make_float2(u.y, u.w);
        }
      flush_system(ca, a0, a1, p, x, g.offn + n * 12 + q + 3 * (q / 3), 3, g.kstr);
    }
  }
}

// Stencil on the work list of several lattices: item (group, 128-site block);
// groups whose systems have all converged are skipped.
template <int R, typename LS, bool EPI>
__global__ void __launch_bounds__(128, R == 4 ? 3 : 4)
    kb_pair(const __grid_constant__ BatchTab T, const GroupDesc* __restrict__ gd, const int2* __restrict__ items,
            const MsState* __restrict__ st, float4* __restrict__ Y, const float4* __restrict__ X,
            const __grid_constant__ PairHops H, PackedDot sd, int nb) {
  const int2 it = items[blockIdx.x];
  const GroupDesc gr = gd[it.x];
  if (st[gr.s0].done && (R == 2 || st[gr.s0 + 1].done)) return;
  const BatchLat& L = T.lat[gr.lat];
  const int n0 = it.y * 128 + threadIdx.x;
  const bool valid = n0 < L.g.V;
  float dA = 0.f, dB = 0.f, sA = 0.f, sB = 0.f;
  if constexpr (EPI) {
    sA = (float)sd.sig[gr.s0];
    sB = R == 4 ? (float)sd.sig[gr.s0 + 1] : sA;
  }
  pr_site<R, LS, 1, EPI>(L.g, valid ? n0 : 0, valid, nullptr, 0, Y + gr.poff, X + gr.poff, (const LS*)L.W, (const float*)L.C,
                         (float)L.diag, H, EPI ? sd.p + gr.poff : nullptr, sA, sB, dA, dB);
  if constexpr (EPI) pr_partials<R>(sd.part, gr.s0, nb, it.y, valid, dA, dB);
}

// A problem on packed vectors: groups in the order of their systems (pairs of a
// lattice first, then its odd one), `words` 16-byte words per packed vector.
struct PackedProblem {
  std::vector<GroupDesc> grp;
  int nsys = 0, nshift = 0, maxiter = 0;
  int64_t words = 0;
  std::vector<double> sig;  // [nsys][nshift], increasing within a system
  std::vector<double> tol;  // [nsys]
};

// Solves (A + sig[s][k]) x[k][s] = b[s].  pack(dst) writes the packed right-hand
// sides; apply(dagger, X, Y, P, na) enqueues Y = D X (P null) or Y = D^dagger X +
// sigma P with partials [nsys][nb] in sdpart, for at least the first na systems.
// Several shifts: solutions in x64 (zeroed here).  One shift: packed in xp.
// whole: all iterations in one WHILE-node graph (no host polling), else host
// polling every kRing iterations and a shrinking prefix of systems.
template <typename Pack, typename Apply>
int packed_solve(cudaStream_t st, const PackedProblem& pb, Pack&& pack, Apply&& apply, double* sdpart, int nb,
                 double2* x64, size_t x64_bytes, float4* xp, bool whole, bool graphs, int* hdone,
                 int* iters_out, Counters* cnt, double* lam_out, const MsState** state_out = nullptr) {
  const int nsys = pb.nsys, nshift = pb.nshift, ngrp = (int)pb.grp.size();
  const bool defer = x64 != nullptr;
  const size_t vb = sizeof(float4) * (size_t)pb.words;
  int64_t maxw = 0, n2all = 0;
  for (const GroupDesc& g : pb.grp) {
    maxw = std::max(maxw, packed_words(g.V, g.two ? 12 : 6));
    n2all += g.V * 12 * (g.two ? 2 : 1);
  }
  const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>((maxw + 255) / 256, std::max(1, kMaxPartials / ngrp)));
  DevBuf bgd, bst, bpart, bring, bP, bT, bQ, bpk, bhist, bflags;
  int rc;
  if ((rc = bgd.alloc(sizeof(GroupDesc) * ngrp, st))) return rc;
  if ((rc = bst.alloc(sizeof(MsState) * nsys, st))) return rc;
  if ((rc = bpart.alloc(sizeof(double) * nblk * nsys, st))) return rc;
  if ((rc = bring.alloc(vb * (defer ? kRing : 1), st))) return rc;
  if ((rc = bP.alloc(vb, st))) return rc;
  if ((rc = bT.alloc(vb, st))) return rc;
  if ((rc = bQ.alloc(vb, st))) return rc;
  if (defer && (rc = bpk.alloc(sizeof(float2) * n2all * nshift, st))) return rc;
  if (defer && (rc = bhist.alloc(sizeof(ShiftHist) * nsys, st))) return rc;
  if ((rc = bflags.alloc(sizeof(int) * nsys, st))) return rc;
  const GroupDesc* gd = bgd.as<GroupDesc>();
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
  BRI_CUDA(cudaMemcpyAsync(bgd.p, pb.grp.data(), sizeof(GroupDesc) * ngrp, cudaMemcpyHostToDevice, st));
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
  kp_norm<<<dim3(nblk, ngrp), 256, 0, st>>>(gd, ring, part); note_launch();
  k_scalar_init<<<nsys, RED_THREADS, 0, st>>>(S, part, nblk); note_launch();
  BRI_LAUNCH_CHECK("packed multi-shift init");

  // systems and groups of the active prefix (a pair counts whole)
  auto prefix = [&](int na, int* ns, int* ng) {
    *ns = 0;
    *ng = 0;
    while (*ns < na && *ng < ngrp) *ns += pb.grp[(*ng)++].two ? 2 : 1;
  };
  // `count` iterations from ring slot 0 on (every block of iterations starts there)
  auto enqueue = [&](int na, int count) -> int {
    int ns, ng, q;
    prefix(na, &ns, &ng);
    for (int j = 0; j < count; ++j) {
      if ((q = apply(0, P, T, (const float4*)nullptr, na))) return q;
      if ((q = apply(1, T, Q, (const float4*)P, na))) return q;
      k_scalar_alpha<<<ns, RED_THREADS, 0, st>>>(S, sdpart, nb, hist, defer && j % DW == 0, 1); note_launch();
      float4 *rin = defer ? ring + (j % kRing) * pb.words : ring, *rout = defer ? ring + ((j + 1) % kRing) * pb.words : ring;
      kp_update_r<<<dim3(nblk, ng), 256, 0, st>>>(gd, S, Q, rin, rout, part); note_launch();
      k_scalar_beta<<<ns, RED_THREADS, 0, st>>>(S, part, nblk); note_launch();
      if (defer) kp_update_p<false><<<dim3(nblk, ng), 256, 0, st>>>(gd, S, rout, P, nullptr);
      else kp_update_p<true><<<dim3(nblk, ng), 256, 0, st>>>(gd, S, rout, P, xp);
      note_launch();
      if (defer && ((j + 1) % DW == 0 || j == count - 1)) {
        kp_flush<<<dim3(nblk, ng), 256, 0, st>>>(gd, hist, ring, pb.words, j / DW * DW, bpk.as<float2>(), x64);
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
  if (lam_out) *lam_out = lm;
  if (err) {
    set_error("multi-shift CG: non-finite or non-positive curvature in a reduction");
    return BRI_ERR_NONFINITE;
  }
  return notconv ? BRI_NOT_CONVERGED : BRI_OK;
}
