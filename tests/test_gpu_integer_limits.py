"""Integer Lanczos vectors at the limits of what their dispatch admits (GPU).

An eigenvector of H_W, H b = lambda b, has the closed form S_N b = r_N(lambda) b with
r_N(lambda) = c0 + sum_j c_j / (z_j - lambda), exact up to the node residuals: at most
sum_j |c_j / Im z_j| tol ||b|| < 4 tol ||b|| for the nodes below.
"""
import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import sgn_gpu, to_dev

pytestmark = pytest.mark.gpu

Z = np.array([0.3 + 0.9j, 0.3 - 0.9j, -1.5 + 1.1j, -1.5 - 1.1j, 4.0 + 2.0j])
C = np.array([0.4 - 0.3j, 0.4 + 0.3j, -0.7 + 0.2j, -0.7 - 0.2j, 0.5 + 0.1j])
C0 = 0.2
TOL = 1e-12
MODES = ("fp64", "fp64_2pass", "f32x2", "fp64_regen")


def _r(lam):
    return C0 + np.sum(C / (Z - lam))


def _staggered(dims):
    lx, ly, lz, lt = dims
    t, z, y, x = np.meshgrid(np.arange(lt), np.arange(lz), np.arange(ly), np.arange(lx), indexing="ij")
    return (-1.0) ** (x + y + z + t)


def _ctx(lib, dims, U, m0):
    ctx = lib.Context(dims, bc_t=1, m0=m0)
    ctx.set_gauge(to_dev(U))
    ctx.set_contour(Z, C, C0)
    return ctx


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("spin", [0, 1, 2, 3])
@pytest.mark.parametrize("dims,m0", [((4, 4, 4, 4), 0.0), ((2, 4, 6, 4), 0.0), ((4, 4, 4, 4), 8.0), ((3, 5, 4, 6), 8.0)])
def test_eigenvalues_of_modulus_8(gpu_lib, dims, m0, spin, mode):
    """||H_W|| = |4 - m0| + 4 = 8 at both ends of the masses: free links, periodic time; a
    constant field has lambda = gamma5 (-m0), a staggered one gamma5 (8 - m0)."""
    field = np.ones(dims[::-1]) if m0 == 8.0 else _staggered(dims)
    lam = (-m0 if m0 == 8.0 else 8.0) * (1 if spin < 2 else -1)
    b = np.zeros(dims[::-1] + (4, 3), dtype=np.complex128)
    b[..., spin, :] = field[..., None] * np.array([0.7 - 0.2j, -1.1, 0.4j])
    ctx = _ctx(gpu_lib, dims, S.unit_links(dims), m0)
    got, st = sgn_gpu(ctx, b, tol=TOL, mode=mode)
    assert st["converged"] == 1
    assert np.linalg.norm(got - _r(lam) * b) <= 4 * TOL * np.linalg.norm(b)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("spin", [0, 2])
def test_links_of_unit_rows_and_larger_norm(gpu_lib, spin, mode):
    """All entries 1 / sqrt(3): rows and columns of norm 1, operator norm sqrt(3), and an
    eigenvalue of modulus 4 - m0 + 4 sqrt(3) = 9.33 on staggered colour singlets."""
    dims, m0 = (4, 4, 4, 4), 1.6
    lam = (4.0 - m0 + 4.0 * np.sqrt(3.0)) * (1 if spin < 2 else -1)
    b = np.zeros(dims[::-1] + (4, 3), dtype=np.complex128)
    b[..., spin, :] = _staggered(dims)[..., None]
    ctx = _ctx(gpu_lib, dims, np.full((4,) + dims[::-1] + (3, 3), 3.0**-0.5, dtype=np.complex128), m0)
    got, st = sgn_gpu(ctx, b, tol=TOL, mode=mode)
    assert st["converged"] == 1
    assert np.linalg.norm(got - _r(lam) * b) <= 4 * TOL * np.linalg.norm(b)


def _against_fp64_vectors(lib, dims, eps, b, modes):
    """Both forms run to node residuals far below rounding (tol 1e-16), so that rounding is all
    they differ by.  FP64 vectors commit about 2 units of 2^-53 per Lanczos step, independent
    of one another: 2 sqrt(500) 2^-53 < 5e-15 over the 500 steps of this contour, which the
    integer forms have to keep as well."""
    ctx = lib.Context(dims, bc_t=-1, m0=1.6)
    ctx.set_gauge(to_dev(S.su3_links(dims, eps, 6001)))
    ctx.set_contour_ellipse(64, 3.36, 3.36, 0.25)
    n = b.shape[0]
    want, _ = sgn_gpu(ctx, b, tol=1e-16, mode="fp64_regen")
    for mode in modes:
        got, st = sgn_gpu(ctx, b, tol=1e-16, mode=mode)
        assert st["converged"] == 1
        d, w = (got - want).reshape(n, -1), want.reshape(n, -1)
        assert np.all(np.linalg.norm(d, axis=1) <= 5e-15 * np.linalg.norm(w, axis=1)), mode


@pytest.mark.parametrize("dims,eps", [((8, 8, 8, 8), 0.5), ((16, 16, 16, 16), 0.5)])
def test_point_sources_round_as_fp64_vectors(gpu_lib, dims, eps):
    """A point source's largest component is its whole norm: noise in units of it on every
    other component of the lattice adds up to sqrt(24 V) units."""
    b = S.point_sources(dims, site=(1, 2, 3, 0))[[0, 7]]
    _against_fp64_vectors(gpu_lib, dims, eps, b, ("fp64",))


@pytest.mark.parametrize("kind", ["point", "gauss"])
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (16, 16, 16, 16)])
def test_sums_over_the_stored_basis_round_as_fp64_vectors(gpu_lib, dims, kind):
    """The coefficients of a point source's first vectors are orders of magnitude above those
    of the later ones, which reach the whole lattice."""
    b = S.point_sources(dims, site=(1, 2, 3, 0))[[0, 7]] if kind == "point" else S.gaussian_spinor(dims, 6003, n=2)
    _against_fp64_vectors(gpu_lib, dims, 0.5, b, ("fp64_2pass", "f32x2"))


@pytest.mark.parametrize("mode", ["fp64_2pass", "f32x2"])
def test_node_solutions_round_as_fp64_vectors(gpu_lib, mode):
    """The same for the per-node solutions behind the link force: products of two solutions,
    each within 5e-15 of the FP64 form (_against_fp64_vectors)."""
    import torch

    dims = (8, 8, 8, 8)
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=1.6)
    ctx.set_gauge(to_dev(S.su3_links(dims, 0.5, 6001)))
    ctx.set_contour_ellipse(64, 3.36, 3.36, 0.25)
    pt = S.point_sources(dims, site=(1, 2, 3, 0))
    out = {}
    for m in ("fp64_regen", mode):
        gb = torch.empty(dims[::-1] + (4, 3), dtype=torch.complex128, device="cuda")
        gl = torch.empty((4,) + dims[::-1] + (8,), dtype=torch.float64, device="cuda")
        st = ctx.sgn_vjp(to_dev(pt[7]), to_dev(pt[0]), gb, gl, ctx.opts(tol=1e-16, mode=m))
        torch.cuda.synchronize()
        assert st["converged"] == 1
        out[m] = gb.cpu().numpy(), gl.cpu().numpy()
    (b1, l1), (b0, l0) = out[mode], out["fp64_regen"]
    assert np.linalg.norm(b1 - b0) <= 5e-15 * np.linalg.norm(b0)
    assert np.linalg.norm(l1 - l0) <= 1e-14 * np.linalg.norm(l0)


def test_gradients_of_the_regeneration_form_keep_fp64_vectors(gpu_lib):
    """S_N is hermitian on nodes in conjugate pairs: the gradient of Re<eta, S_N b> in b is
    S_N eta, here from OV_MODE_FP64_REGEN on both sides."""
    import torch

    dims = (8, 8, 8, 8)
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=1.6)
    ctx.set_gauge(to_dev(S.su3_links(dims, 0.5, 6001)))
    ctx.set_contour_ellipse(64, 3.36, 3.36, 0.25)
    eta = S.point_sources(dims, site=(1, 2, 3, 0))[7]
    want, _ = sgn_gpu(ctx, eta, tol=1e-16, mode="fp64_regen")
    ed, grad_b = to_dev(eta), torch.empty(dims[::-1] + (4, 3), dtype=torch.complex128, device="cuda")
    st = ctx.sgn_vjp(ed, to_dev(S.gaussian_spinor(dims, 6002)), grad_b, None, ctx.opts(tol=1e-16, mode="fp64_regen"))
    torch.cuda.synchronize()
    assert st["converged"] == 1
    d = grad_b.cpu().numpy() - want
    assert np.linalg.norm(d) <= 5e-15 * np.linalg.norm(want)  # as in _against_fp64_vectors


@pytest.mark.parametrize("factor", [1e-6, 1e-2, 0.6, 1.0])
def test_short_links(gpu_lib, factor):
    """At m0 = 4 H_W is its hopping term alone, as small as the links: results are held to its
    size.  The stencil: 2^-43 of the largest component times the factor (the bound of the FP64
    kernels, whose partial sums all scale with it).  A solve with nodes that scale alike: as
    _against_fp64_vectors."""
    import torch

    dims, m0 = (4, 4, 4, 6), 4.0
    U = to_dev(factor * S.su3_links(dims, 0.5, 6011))
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=m0)
    ctx.set_gauge(U)
    ctx.set_contour(factor * Z, factor * C, C0)
    b = S.gaussian_spinor(dims, 6012, n=2)
    x = to_dev(b)
    got, want = torch.empty_like(x), torch.empty_like(x)
    ctx.apply_HW(x, got, 2, gpu_lib.OV_FP64)
    assert gpu_lib.apply_HW_noalloc(dims, -1, m0, U, x, want, 2) == gpu_lib.OV_OK
    torch.cuda.synchronize()
    assert (got - want).abs().max().item() <= 2.0**-43 * factor * np.abs(b).max()
    want, _ = sgn_gpu(ctx, b, tol=1e-16, mode="fp64_regen")
    for mode in ("fp64", "fp64_2pass"):
        got, _ = sgn_gpu(ctx, b, tol=1e-16, mode=mode)
        assert np.linalg.norm(got - want) <= 5e-15 * np.linalg.norm(want), mode


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 16, 16, 16), (16, 16, 16, 32)])
def test_norms_of_constant_vectors(gpu_lib, dims):
    """A constant field on free links stays constant: no component's low limb differs from
    site to site, and the sums of the norm add up without cancellation.  Upper spins have
    lambda = -m0, lower ones m0, so that the Krylov space ends after two vectors."""
    m0 = 1.6
    b = np.zeros(dims[::-1] + (4, 3), dtype=np.complex128)
    b[..., 0, 0], b[..., 1, 2], b[..., 2, 1] = 0.77123, 0.3j, 1.234567
    want = b.copy()
    want[..., :2, :] *= _r(-m0)
    want[..., 2:, :] *= _r(m0)
    ctx = _ctx(gpu_lib, dims, S.unit_links(dims), m0)
    got, st = sgn_gpu(ctx, b, tol=TOL, mode="fp64")
    assert st["converged"] == 1 and st["iterations"] == 2
    assert np.linalg.norm(got - want) <= 4 * TOL * np.linalg.norm(b)
