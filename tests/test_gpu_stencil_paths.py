"""Every kernel the Brillouin stencil's dispatch can take, at the sizes where it can go wrong, against
the FP64 oracle: both sides of the line between the split and the packed FP32 kernels (8192 sites x
right-hand sides) and of those between the packed forms (98304: four or two thread groups per site,
393216: one, 786432: pairs of right-hand sides), 8, 16 and 32 sites per block of the split kernel, an odd right-hand
side behind the packed pairs, volumes that are no multiple of a link chunk (32 sites) or a block, extents of two.

Tolerances are those of the parity tests: FP32 1e-5 and BF16 links 1e-2 of the largest element (a few
hundred roundings of 2^-24 per element, 2^-9 per BF16 link element), FP64 1e-12, mixed solves 1e-10.
"""
import functools

import numpy as np
import pytest
import torch

import synthetic_fields as sf
from oracle import dirac
from paper_1701_00726_gb300 import PREC_F32, PREC_F32_BF16, PREC_F64, Lattice, overlap_apply_batch

pytestmark = pytest.mark.gpu

LARGE = (9, 8, 7, 17)  # 8568 sites: 267 full chunks and 24 sites


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


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 2, 5, 2), 3), ((6, 5, 4, 3), 1), ((7, 5, 6, 5), 7),
                                       ((7, 5, 6, 5), 8), (LARGE, 1), (LARGE, 3), (LARGE, 4)])
@pytest.mark.parametrize("dagger", [False, True])
def test_bri_apply_every_path(dims, nrhs, dagger):
    x, want = _want(dims, nrhs, dagger, True)
    lat = _lattice(dims, anti=True)
    xt = torch.from_numpy(x).cuda()
    assert relerr(lat.bri_apply(xt, -1.0, dagger=dagger).cpu().numpy(), want) < 1e-12
    x32 = xt.to(torch.complex64)
    for bf16, bound in ((False, 1e-5), (True, 1e-2)):
        assert relerr(lat.bri_apply(x32, -1.0, dagger=dagger, bf16_links=bf16).cpu().numpy(), want) < bound


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((5, 4, 6, 3), 3), ((7, 5, 6, 5), 2), ((4, 4, 4, 5), 5)])
@pytest.mark.parametrize("dagger", [False, True])
def test_wils_apply_blocks(dims, nrhs, dagger):
    """The FP32 Wilson kernel's blocks of 64 sites x 2 right-hand sides and 128 x 1 (the odd one), full
    (320 sites) and with a partial last block: 1e-5 of the largest element."""
    x = sf.gaussian_source(dims, nrhs, 1036)
    op = dirac.DiracOperator(sf.gauge_field(dims, 31), "wil", m0=-1.0, c_sw=1.0, antiperiodic_t=True)
    y = _lattice(dims, anti=True).wils_apply(torch.from_numpy(x).to(torch.complex64).cuda(), -1.0, dagger=dagger)
    assert relerr(y.cpu().numpy(), op.apply_dagger(x) if dagger else op.apply(x)) < 1e-5


@pytest.mark.parametrize("dims,nrhs", [((2, 2, 2, 2), 1), ((3, 2, 5, 2), 3), (LARGE, 2), (LARGE, 46)])
@pytest.mark.parametrize("dagger", [False, True])
def test_double_word_forms(dims, nrhs, dagger):
    """Double-word stencil with four groups of threads per site and (394128 sites x rhs) with one: 1e-13 of
    the largest element, as in the parity tests (48-bit operands, a few hundred roundings)."""
    some = [0, nrhs - 1] if nrhs > 4 else list(range(nrhs))
    x = sf.gaussian_source(dims, nrhs, 1035)
    op = _operator(dims, True)[1]
    want = op.apply_dagger(x[some]) if dagger else op.apply(x[some])
    y = _lattice(dims, anti=True).bri_apply(torch.from_numpy(x).cuda(), -1.0, dagger=dagger, double_word=True)
    assert relerr(y[some].cpu().numpy(), want) < 1e-13


@pytest.mark.parametrize("dims,nrhs", [((8, 6, 7, 10), 19), (LARGE, 17), ((16, 15, 17, 19), 7), ((16, 15, 17, 19), 15)])
def test_packed_forms_and_chunks(dims, nrhs):
    """Chunks of 16 right-hand sides (the packed buffer's size) and what is left, in every packed form:
    four groups per site; two (137088 sites x rhs) and four; one (542640); pairs and an odd one."""
    lat = _lattice(dims)
    x = torch.from_numpy(sf.gaussian_source(dims, nrhs, 1032)).to(torch.complex64).cuda()
    y = lat.bri_apply(x, -1.0)
    some = sorted({0, min(15, nrhs - 1), nrhs - 1})[:3 if lat.volume < 20000 else 1]
    want = _operator(dims, False)[1].apply(x[some].cpu().numpy().astype(np.complex128))
    assert relerr(y[some].cpu().numpy(), want) < 1e-5
    y64 = lat.bri_apply(x.to(torch.complex128), -1.0)
    assert relerr(y.cpu().numpy(), y64.cpu().numpy()) < 1e-5


@pytest.mark.parametrize("dims,nrhs", [((7, 5, 6, 5), 7), (LARGE, 1), (LARGE, 4), (LARGE, 16), (LARGE, 48)])
@pytest.mark.parametrize("prec", [PREC_F32, PREC_F32_BF16])
def test_mixed_solve_packed_and_split(dims, nrhs, prec):
    """The mixed sign function with the split kernel (7350 sites x systems) and with the solver's vectors
    packed (four groups per site: 1 and 4, two: 16, one: 48), a zero source among
    them: the FP64 path's result."""
    lat = _lattice(dims)
    x = torch.from_numpy(sf.gaussian_source(dims, nrhs, 1033)).cuda()
    if nrhs > 1:
        x[nrhs - 1] = 0.0
    y64, _ = lat.sign_apply(x, 4, tol=1e-13, prec=PREC_F64)
    y, st = lat.sign_apply(x, 4, tol=1e-11, prec=prec, want_true_residual=True)
    assert st["converged"] and st["max_true_residual"] <= 1e-11
    assert relerr(y.cpu().numpy(), y64.cpu().numpy()) < 1e-10
    if nrhs > 1:
        assert float(y[nrhs - 1].abs().max()) == 0.0


@pytest.mark.parametrize("nrhs", [(3, 4), (9, 8), (24, 23)])
def test_batch_packed_forms(nrhs):
    """Two lattices in one batch with four, two and one (402696 sites x systems) groups per site: the
    lattices' own FP64 results."""
    lats = [_lattice(LARGE), _lattice(LARGE, anti=True)]
    xs = [torch.from_numpy(sf.gaussian_source(LARGE, r, 1034 + i)).cuda() for i, r in enumerate(nrhs)]
    ys, _ = overlap_apply_batch(lats, xs, n=4, tol=1e-11, prec=PREC_F32)
    for lat, x, y in zip(lats, xs, ys):
        want, _ = lat.overlap_apply(x, n=4, tol=1e-13, prec=PREC_F64)
        assert relerr(y.cpu().numpy(), want.cpu().numpy()) < 1e-10
