"""Forms of the kernels that the public calls take rarely, at the sizes where they can go wrong: against the FP64 oracle
or against the common form, with the tolerances of the parity tests (FP32 1e-5 and BF16 links 1e-2 of the largest
element, FP64 1e-12, mixed solves 1e-10).
"""
import functools

import numpy as np
import pytest
import torch

import synthetic_fields as sf
from oracle import dirac
from paper_1701_00726_gb300 import Lattice

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
