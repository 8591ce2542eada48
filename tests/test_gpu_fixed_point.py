"""The stored-basis solves in fixed point against the FP64 regeneration form (GPU).

OV_MODE_FP64_2PASS and OV_MODE_F32X2 run their Lanczos vectors as integers of one scale per
vector when the links are unitary and |4 - m0| <= 4, else in FP64 and double-float.
OV_MODE_FP64_REGEN computes the same iterates in FP64 throughout.  Both forms stop at a node
residual of tol ||b||, so that each differs from the quadrature sum by at most
sum_j |c_j| tol / |Im z_j|; the nodes below have sum_j |c_j / Im z_j| < 4, which bounds the
difference of two results by 8 tol ||b|| = 8e-12 in norm.
"""
import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import make_ctx, rel, sgn_gpu, to_dev

pytestmark = pytest.mark.gpu

Z = np.array([0.3 + 0.9j, 0.3 - 0.9j, -1.5 + 1.1j, -1.5 - 1.1j, 4.0 + 2.0j])
C = np.array([0.4 - 0.3j, 0.4 + 0.3j, -0.7 + 0.2j, -0.7 - 0.2j, 0.5 + 0.1j])
TOL = 1e-12


def _agree(ctx, b, nrhs, modes=("fp64_2pass", "f32x2")):
    ctx.set_contour(Z, C, 0.2)
    want, _ = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64_regen")
    for mode in modes:
        got, st = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode=mode)
        assert st["converged"] == 1
        for k in range(nrhs):
            w = want[k] if b.ndim == 7 else want
            g = got[k] if b.ndim == 7 else got
            assert np.linalg.norm(g - w) <= 8 * TOL * np.linalg.norm(b[k] if b.ndim == 7 else b), (mode, k)


@pytest.mark.parametrize("bc_t", [-1, 1])
@pytest.mark.parametrize("dims,nrhs", [((3, 5, 4, 6), 5), ((2, 2, 2, 3), 1), ((1, 7, 5, 9), 3), ((8, 4, 4, 5), 13),
                                       ((33, 1, 2, 2), 2)],
                         ids=["3x5x4x6-5", "2x2x2x3-1", "1x7x5x9-3", "8x4x4x5-13", "33x1x2x2-2"])
def test_lattices_and_source_counts(gpu_lib, dims, nrhs, bc_t):
    """Padded last tiles, extents 1 and 2, more sources than one block takes in turn."""
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 3101, bc_t=bc_t)
    _agree(ctx, S.gaussian_spinor(dims, 3102, n=nrhs), nrhs)


@pytest.mark.parametrize("scale", [1e-120, 2.0**-3, 1.0, 1e120])
def test_source_scales(gpu_lib, scale):
    dims = (4, 4, 4, 6)
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 3111)
    b = S.gaussian_spinor(dims, 3112, n=2)
    b[1] *= 1e-8  # each source has its own scale
    _agree(ctx, scale * b, 2)


def test_point_sources(gpu_lib):
    """The first vectors of a point source spread from one site over the lattice (the shift
    of w against its successor), and most of their components are zero."""
    dims = (8, 8, 8, 8)
    ctx, _ = make_ctx(gpu_lib, dims, 0.4, 3121)
    _agree(ctx, S.point_sources(dims, site=(7, 0, 3, 7)), 12)


@pytest.mark.parametrize("factor,m0", [(1.0, 0.0), (1.0, 8.0), (1.0, -0.5), (1.0, 1.0), (0.7, 1.6), (1.4, 1.6)])
def test_links_and_masses_on_both_sides_of_the_rule(gpu_lib, factor, m0):
    """Masses at and beyond |4 - m0| = 4, links shorter than unitary (still within the
    bounds) and longer (FP64 and double-float kernels)."""
    dims = (4, 4, 6, 4)
    U = factor * S.su3_links(dims, 0.5, 3131)
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=m0)
    ctx.set_gauge(to_dev(U))
    _agree(ctx, S.gaussian_spinor(dims, 3132, n=2), 2)


def test_gauge_reload_refreshes_the_links(gpu_lib):
    dims = (4, 4, 4, 4)
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 3141)
    b = S.gaussian_spinor(dims, 3142)
    _agree(ctx, b, 1)
    first, _ = sgn_gpu(ctx, b, tol=TOL, mode="fp64_2pass")
    ctx.set_gauge(to_dev(S.su3_links(dims, 0.5, 3143)))
    _agree(ctx, b, 1)
    second, _ = sgn_gpu(ctx, b, tol=TOL, mode="fp64_2pass")
    assert rel(second, first) > 1e-2


@pytest.mark.parametrize("mode", ["fp64_2pass", "f32x2"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_link_breaks_down(gpu_lib, mode, bad):
    dims = (4, 4, 4, 4)
    U = S.su3_links(dims, 0.5, 3151)
    U[2, 1, 0, 3, 2, 0, 1] = bad
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=1.6)
    ctx.set_gauge(to_dev(U))
    ctx.set_contour(Z, C, 0.2)
    with pytest.raises(gpu_lib.OvError) as e:
        sgn_gpu(ctx, S.gaussian_spinor(dims, 3152), mode=mode)
    assert e.value.code == gpu_lib.OV_ERR_BREAKDOWN


@pytest.mark.parametrize("imag", [0.9, 0.22, 0.12])
def test_coefficients_of_short_and_long_recurrences(gpu_lib, imag):
    """Nodes that stop early beside one at distance `imag`, which decides the count: within
    one pass of the coefficient recurrence (512 rows), and beyond it.  Both forms stop at
    residual tol ||b||: at most 2 sum_j |c_j / Im z_j| tol ||b|| apart."""
    dims = (4, 4, 4, 6)
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 3181)
    z = np.array([0.3 + 1j * imag, -2.0 + 3.0j, 1.0 - 6.0j, 5.0 + 2.0j])
    c = np.array([0.4 - 0.3j, -0.7 + 0.2j, 0.5 + 0.1j, 0.2j])
    ctx.set_contour(z, c, 0.1)
    b = S.gaussian_spinor(dims, 3182, n=3)
    want, _ = sgn_gpu(ctx, b, nrhs=3, tol=TOL, mode="fp64_regen")
    got, st = sgn_gpu(ctx, b, nrhs=3, tol=TOL, mode="fp64_2pass")
    assert (st["iterations"] > 512) == (imag < 0.2) and st["iterations"] < 1024
    bound = 2 * np.sum(np.abs(c / z.imag)) * TOL
    for k in range(3):
        assert np.linalg.norm(got[k] - want[k]) <= bound * np.linalg.norm(b[k])


@pytest.mark.parametrize("dims,steps", [((4, 4, 4, 4), 4), ((3, 5, 4, 6), 7), ((8, 8, 8, 8), 40), ((12, 12, 12, 16), 24)])
def test_spectral_bounds(gpu_lib, dims, steps):
    """The Lanczos bounds from integer vectors (default) and, with the persistent loop enabled,
    from FP64 vectors.  Over so few steps no Ritz value has converged, so the tridiagonals
    differ by rounding alone, amplified by at most some thousands: 1e-11 ||H||."""
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 3191)
    got = ctx.place_contour(8, steps=steps)
    ctx.set_persistent(1)
    want = ctx.place_contour(8, steps=steps)
    assert got["steps"] == want["steps"] == steps
    for key in ("lambda_min", "lambda_max", "abs_max_bound"):
        assert abs(got[key] - want[key]) <= 1e-11 * 8
