"""Forms of the kernels that the public calls take rarely, at the sizes where they can go wrong: against the FP64 oracle
or against the common form, with the tolerances of the parity tests (FP32 1e-5 and BF16 links 1e-2 of the largest
element, FP64 1e-12, mixed solves 1e-10).
"""
import ctypes
import functools
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

import synthetic_fields as sf
from oracle import dirac
from paper_1701_00726_gb300 import PREC_F32, PREC_F64, Lattice, build, overlap_apply_batch

pytestmark = pytest.mark.gpu

LARGE = (9, 8, 7, 17)  # 8568 sites: 267 blocks of 32 and 24 sites


@functools.lru_cache(maxsize=None)
def _operator(dims):
    u = sf.gauge_field(dims, 31)
    return u, dirac.DiracOperator(u, "bri", m0=-1.0, c_sw=1.0, antiperiodic_t=True)


def _lattice(dims, c_sw=1.0, **kw):
    lat = Lattice(dims, antiperiodic_t=True, **kw)
    lat.build_links(torch.from_numpy(_operator(dims)[0]).cuda(), c_sw)
    return lat


def relerr(got, want):
    return float(np.abs(got - want).max() / np.abs(want).max())


@pytest.mark.parametrize("dims,nrhs", [(LARGE, 1), (LARGE, 3), ((8, 6, 7, 10), 40), ((16, 15, 17, 19), 7), ((16, 15, 17, 19), 11)])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("dagger", [False, True])
def test_captured_application(dims, nrhs, bf16, dagger):
    """Captured into a graph, a large FP32 application reads the spinors in their own layout (four, two and one thread
    groups per site): the oracle's result, and the eager call's to FP32 rounding, on every replay."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        lat = _lattice(dims, stream=stream)
        x = torch.from_numpy(sf.gaussian_source(dims, nrhs, 1041)).to(torch.complex64).cuda()
        eager = lat.bri_apply(x, -1.0, dagger=dagger, bf16_links=bf16)
        y = torch.empty_like(x)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lat.bri_apply(x, -1.0, dagger=dagger, bf16_links=bf16, out=y)
        for _ in range(2):
            y.zero_()
            graph.replay()
        stream.synchronize()
        some = [0, nrhs - 1] if lat.volume < 20000 else [nrhs - 1]
        xs = x[some].cpu().numpy().astype(np.complex128)
        op = _operator(dims)[1]
        want = op.apply_dagger(xs) if dagger else op.apply(xs)
        assert relerr(y[some].cpu().numpy(), want) < (1e-2 if bf16 else 1e-5)
        assert relerr(y.cpu().numpy(), eager.cpu().numpy()) < 1e-6  # the same operands, a few roundings apart


SUM3 = r"""
#include "sum3.cuh"
using namespace bri;
__global__ void k(int n, const float2* x, const float2* y, double n2, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, e = unit_exponent(n2);
  const float2 f = make_float2(exp2_float(e), exp2_float(e));
  Sum3 s = sum3_zero();
  for (int i = 0; i < n; ++i) sum3_add(s, __fmul2_rn(x[t * n + i], f), __fmul2_rn(y[t * n + i], f));
  out[t] = sum3_total(s) * exp2_square(e);
}
extern "C" int run(int threads, int n, const float2* x, const float2* y, double n2, double* out) {
  k<<<threads / 64, 64>>>(n, x, y, n2, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def sum3(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum3")
    (d / "t.cu").write_text(SUM3)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-o",
                    str(d / "t.so"), str(d / "t.cu")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("n", [1, 8, 24])
@pytest.mark.parametrize("scale", [-120, -65, 0, 62, 110])
@pytest.mark.parametrize("square", [True, False])
def test_fp32_sums_of_products_to_fp64_accuracy(sum3, n, scale, square):
    """The reductions of the packed solver, at element scales whose FP32 squares under- and overflow: two FP64 roundings
    of the absolute sum (2^-52; the rounding of the third word adds 2^-54 for 24 products), where FP64 multiply-adds
    may err by one rounding per product and a double-word sum by 2^-48 for each."""
    rng = np.random.default_rng(31 + n)
    threads = 128
    x = (rng.standard_normal((threads, n, 2)) * 10.0 ** rng.uniform(-5, 0, (threads, n, 2))).astype(np.float32)
    y = x if square else rng.standard_normal(x.shape).astype(np.float32)
    f = 2.0 ** scale
    xt, yt = (torch.from_numpy((v.astype(np.float64) * f).astype(np.float32)).cuda() for v in (x, y))
    out = torch.zeros(threads, dtype=torch.float64, device="cuda")
    assert sum3.run(threads, n, *(ctypes.c_void_p(v.data_ptr()) for v in (xt, yt)), ctypes.c_double(f * f),
                    ctypes.c_void_p(out.data_ptr())) == 0
    xs, ys = xt.cpu().tolist(), yt.cpu().tolist()  # (at 2^-120 the small ones were rounded to FP32 subnormals)
    for t, got in enumerate(out.cpu().tolist()):
        prods = [Fraction(a) * Fraction(b) for i in range(n) for a, b in zip(xs[t][i], ys[t][i])]
        assert abs(Fraction(got) - sum(prods)) <= Fraction(5, 4) * Fraction(2) ** -52 * sum(map(abs, prods))


@pytest.mark.parametrize("scale", [-65, 66])
def test_batch_of_small_and_large_sources(scale):
    """Sources whose elements' squares leave FP32's range: the batched solve takes its inner products to FP64 range, so
    that a source scaled by a power of two gives the scaled result bit by bit (at 1e-3 the first phase is all there is;
    the FP32 corrections' own inner products are in FP32)."""
    dims = [LARGE, (6, 5, 4, 3)]
    lats = [_lattice(d) for d in dims]
    xs = [torch.from_numpy(sf.gaussian_source(d, r, 1042)).cuda() for d, r in zip(dims, (2, 3))]
    want, _ = overlap_apply_batch(lats, xs, n=4, tol=1e-3, prec=PREC_F32)
    got, st = overlap_apply_batch(lats, [x * 2.0 ** scale for x in xs], n=4, tol=1e-3, prec=PREC_F32)
    assert all(s["refinements"] == 0 for s in st)
    for g, w in zip(got, want):
        assert torch.equal(g, w * 2.0 ** scale)


@pytest.mark.parametrize("dagger", [False, True])
def test_fp64_sixteen_sites_per_block(dagger):
    """FP64 split kernel between 9728 and 19455 sites x right-hand sides (17136), against the oracle."""
    x = sf.gaussian_source(LARGE, 2, 1043)
    op = _operator(LARGE)[1]
    y = _lattice(LARGE).bri_apply(torch.from_numpy(x).cuda(), -1.0, dagger=dagger).cpu().numpy()
    assert relerr(y, op.apply_dagger(x) if dagger else op.apply(x)) < 1e-12


@pytest.mark.parametrize("dims,nrhs", [(LARGE, 17), ((16, 15, 17, 19), 7), ((16, 15, 17, 19), 15)])
def test_bf16_links_in_the_packed_forms(dims, nrhs):
    """BF16 links with two thread groups per site and a rest of one right-hand side, with one group, and in pairs: the
    oracle's result to the links' 8 bits."""
    x = torch.from_numpy(sf.gaussian_source(dims, nrhs, 1044)).to(torch.complex64).cuda()
    y = _lattice(dims).bri_apply(x, -1.0, bf16_links=True)
    some = [0, nrhs - 1] if nrhs == 17 else [nrhs - 1]
    want = _operator(dims)[1].apply(x[some].cpu().numpy().astype(np.complex128))
    assert relerr(y[some].cpu().numpy(), want) < 1e-2


@pytest.mark.parametrize("nrhs,prec", [((1, 4), PREC_F64), ((2, 8), PREC_F64), ((9, 24), PREC_F32), ((40, 60), PREC_F32)])
def test_batch_of_uneven_volumes(nrhs, prec):
    """Batches of two volumes: FP64 with 16 (12768 sites x systems) and 32 (25536) sites per block, mixed with two (102312)
    and one (405720) thread groups per site: each lattice's own FP64 result."""
    dims = [LARGE, (7, 5, 6, 5)]
    lats = [_lattice(d) for d in dims]
    xs = [torch.from_numpy(sf.gaussian_source(d, r, 1045)).cuda() for d, r in zip(dims, nrhs)]
    ys, _ = overlap_apply_batch(lats, xs, n=4, tol=1e-13 if prec == PREC_F64 else 1e-11, prec=prec)
    for lat, x, y in zip(lats, xs, ys):
        want, _ = lat.overlap_apply(x, n=4, tol=1e-13, prec=PREC_F64)
        assert relerr(y.cpu().numpy(), want.cpu().numpy()) < 1e-10
