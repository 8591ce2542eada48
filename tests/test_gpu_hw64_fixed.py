"""ov_apply_HW in FP64 through integers against the FP64 kernel of ov_apply_HW_noalloc (GPU).

The integer stencil scales every site by its largest component.  With M the largest
component among a site and its eight neighbours, its error is a few units of 2^-58 M per hop
and the FP64 kernel's at most 2^-53 times the about 30 partial sums of at most 24 M per
component: both are within 2^-44 M of the exact value, their difference within 2^-43 M.
"""
import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import M0, to_dev, to_host

pytestmark = pytest.mark.gpu


def _both(lib, dims, U, psi, bc_t=-1, m0=M0):
    import torch

    ctx = lib.Context(dims, bc_t=bc_t, m0=m0)
    Ud, x = to_dev(U), to_dev(psi)
    ctx.set_gauge(Ud)
    got, want = torch.empty_like(x), torch.empty_like(x)
    ctx.apply_HW(x, got, psi.shape[0], lib.OV_FP64)
    assert lib.apply_HW_noalloc(dims, bc_t, m0, Ud, x, want, psi.shape[0]) == lib.OV_OK
    torch.cuda.synchronize()
    ctx.close()
    return to_host(got), to_host(want)


def _local_max(psi):
    m = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(axis=(-1, -2))
    out = m.copy()
    for ax in range(1, 5):
        for step in (1, -1):
            out = np.maximum(out, np.roll(m, step, ax))
    return out[..., None, None]


@pytest.mark.parametrize("bc_t", [-1, 1])
@pytest.mark.parametrize("dims,nrhs", [((4, 4, 4, 4), 1), ((3, 5, 4, 6), 7), ((1, 2, 3, 4), 2), ((2, 2, 2, 2), 13),
                                       ((33, 1, 2, 1), 3), ((8, 4, 6, 5), 12)])
def test_matches_fp64_kernel(gpu_lib, dims, nrhs, bc_t):
    U = S.su3_links(dims, 0.5, 5001)
    psi = S.gaussian_spinor(dims, 5002, n=nrhs)
    got, want = _both(gpu_lib, dims, U, psi, bc_t)
    assert np.all(np.abs(got - want) <= 2.0**-43 * _local_max(psi))


def test_magnitudes_that_vary_over_the_lattice(gpu_lib):
    """Sites from 1e-300 to 1e300 next to one another, zero sites and subnormal ones: each
    output as accurate as its own neighbourhood allows."""
    dims = (4, 6, 4, 5)
    U = S.su3_links(dims, 0.5, 5011)
    psi = S.gaussian_spinor(dims, 5012, n=4)
    rng = np.random.Generator(np.random.PCG64(5013))
    e = rng.uniform(-300, 300, psi.shape[:5])
    e[1] = rng.uniform(-12, 0, psi.shape[1:5])
    e[2] = -310
    psi = psi * 10.0 ** e[..., None, None]
    psi[3] = 0.0
    psi[3, 1, 2, 3, 0] = 1e-5
    psi[:, 2, 1] = 0.0
    got, want = _both(gpu_lib, dims, U, psi)
    # subnormal results are rounded to multiples of 5e-324
    assert np.all(np.abs(got - want) <= 2.0**-43 * _local_max(psi) + 64 * 5e-324)
    assert np.all(got[want == 0] == 0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_components_propagate_alike(gpu_lib, bad):
    dims = (4, 4, 6, 4)
    U = S.su3_links(dims, 0.5, 5021)
    psi = S.gaussian_spinor(dims, 5022, n=2)
    psi[1, 2, 3, 1, 2, 1, 0] = complex(bad, 1.0)
    got, want = _both(gpu_lib, dims, U, psi)
    for a, b in ((got.real, want.real), (got.imag, want.imag)):
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.array_equal(a[np.isinf(b)], b[np.isinf(b)]) and np.array_equal(np.isinf(a), np.isinf(b))
    ok = np.isfinite(want)
    assert np.all(np.abs(got - want)[ok] <= 2.0**-43 * np.abs(psi[0]).max() * 2)


@pytest.mark.parametrize("factor,m0", [(1.0, 0.0), (1.0, 8.0), (1.0, 8.5), (0.6, 1.6), (1.3, 1.6)])
def test_links_and_masses_on_both_sides_of_the_rule(gpu_lib, factor, m0):
    dims = (4, 4, 4, 6)
    U = factor * S.su3_links(dims, 0.5, 5031)
    psi = S.gaussian_spinor(dims, 5032, n=3)
    got, want = _both(gpu_lib, dims, U, psi, m0=m0)
    assert np.all(np.abs(got - want) <= 2.0**-42 * _local_max(psi))
