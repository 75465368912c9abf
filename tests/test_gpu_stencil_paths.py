"""Every kernel the Brillouin stencil's dispatch can take, at the sizes where it can go wrong, against
the FP64 oracle: both sides of the line between the split and the packed FP32 kernels (24576 sites x
right-hand sides), 8, 16 and 32 sites per block of the split kernel, an odd right-hand side behind the
packed pairs, volumes that are no multiple of a link chunk (32 sites) or a block, extents of two.

Tolerances are those of the parity tests: FP32 1e-5 and BF16 links 1e-2 of the largest element (a few
hundred roundings of 2^-24 per element, 2^-9 per BF16 link element), FP64 1e-12, mixed solves 1e-10.
"""
import functools

import numpy as np
import pytest
import torch

import synthetic_fields as sf
from oracle import dirac
from paper_1701_00726_gb300 import PREC_F32, PREC_F32_BF16, PREC_F64, Lattice

pytestmark = pytest.mark.gpu

LARGE = (9, 8, 7, 17)  # 8568 sites: 2 right-hand sides split, 3 and more packed; 267 full chunks and 24 sites


@functools.lru_cache(maxsize=None)
def _operator(dims, anti):
    u = sf.gauge_field(dims, 31)
    return u, dirac.DiracOperator(u, "bri", m0=-1.0, c_sw=1.0, antiperiodic_t=anti)


def _lattice(dims, anti=False):
    lat = Lattice(dims, antiperiodic_t=anti)
    lat.build_links(torch.from_numpy(_operator(dims, anti)[0]).cuda(), 1.0)
    return lat


@functools.lru_cache(maxsize=None)
def _want(dims, nrhs, dagger, anti):
    x = sf.gaussian_source(dims, nrhs, 1031)
    op = _operator(dims, anti)[1]
    return x, op.apply_dagger(x) if dagger else op.apply(x)


def relerr(got, want):
    return float(np.abs(got - want).max() / np.abs(want).max())


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 2, 5, 2), 3), ((6, 5, 4, 3), 1), ((7, 5, 6, 5), 9),
                                       (LARGE, 2), (LARGE, 3), (LARGE, 4)])
@pytest.mark.parametrize("dagger", [False, True])
def test_bri_apply_every_path(dims, nrhs, dagger):
    x, want = _want(dims, nrhs, dagger, True)
    lat = _lattice(dims, anti=True)
    xt = torch.from_numpy(x).cuda()
    assert relerr(lat.bri_apply(xt, -1.0, dagger=dagger).cpu().numpy(), want) < 1e-12
    x32 = xt.to(torch.complex64)
    for bf16, bound in ((False, 1e-5), (True, 1e-2)):
        assert relerr(lat.bri_apply(x32, -1.0, dagger=dagger, bf16_links=bf16).cpu().numpy(), want) < bound


def test_packed_launch_in_chunks():
    """More right-hand sides than one packed buffer holds (16) and an odd count: each equals its own launch."""
    dims = (8, 6, 7, 10)  # 3360 sites x 19 right-hand sides: packed, in two chunks, the second with an odd one
    lat = _lattice(dims)
    x = torch.from_numpy(sf.gaussian_source(dims, 19, 1032)).to(torch.complex64).cuda()
    y = lat.bri_apply(x, -1.0)
    want = _operator(dims, False)[1].apply(x[[0, 15, 16, 18]].cpu().numpy().astype(np.complex128))
    assert relerr(y[[0, 15, 16, 18]].cpu().numpy(), want) < 1e-5
    y64 = lat.bri_apply(x.to(torch.complex128), -1.0)
    assert relerr(y.cpu().numpy(), y64.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("nrhs", [2, 3, 4])
@pytest.mark.parametrize("prec", [PREC_F32, PREC_F32_BF16])
def test_mixed_solve_packed_and_split(nrhs, prec):
    """The mixed sign function with the solver's vectors packed (3: a pair and an odd system, 4: two
    pairs) and with the split kernel (2), a zero source among them: the FP64 path's result."""
    lat = _lattice(LARGE)
    x = torch.from_numpy(sf.gaussian_source(LARGE, nrhs, 1033)).cuda()
    x[nrhs - 1] = 0.0
    y64, _ = lat.sign_apply(x, 4, tol=1e-13, prec=PREC_F64)
    y, st = lat.sign_apply(x, 4, tol=1e-11, prec=prec, want_true_residual=True)
    assert st["converged"] and st["max_true_residual"] <= 1e-11
    assert relerr(y.cpu().numpy(), y64.cpu().numpy()) < 1e-10
    assert float(y[nrhs - 1].abs().max()) == 0.0
