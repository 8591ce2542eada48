"""OV_MODE_FP64, its nodes spread over groups of blocks, against OV_MODE_FP64_REGEN (GPU).

m0 = 1.4 runs the Lanczos vectors in fixed point with batched node updates, m0 = -0.5
(|4 - m0| > 4) in FP64 with node updates in every iteration.  Both forms stop at a node residual of tol ||b||, so that each differs from the quadrature sum by
at most sum_j |c_j| tol / |Im z_j| ||b||.  The nodes below keep sum_j |c_j / Im z_j| < 4 for any
count, which bounds the difference of two results by 8 tol ||b|| in norm.
"""
import numpy as np
import pytest
import torch

import synthetic as S
from tests.gpu_common import make_ctx, sgn_gpu, to_dev, to_host

pytestmark = pytest.mark.gpu

Z = np.array([0.3 + 0.9j, 0.3 - 0.9j, -1.5 + 1.1j, -1.5 - 1.1j, 4.0 + 2.0j])
C = np.array([0.4 - 0.3j, 0.4 + 0.3j, -0.7 + 0.2j, -0.7 - 0.2j, 0.5 + 0.1j])
TOL = 1e-12


def _nodes(ns):
    k = np.arange(ns) // 5
    z = Z[np.arange(ns) % 5].real + 1j * Z[np.arange(ns) % 5].imag * (1.0 + 0.3 * k)
    return z, C[np.arange(ns) % 5] / (k[-1] + 1)


@pytest.mark.parametrize("m0", [1.4, -0.5])
@pytest.mark.parametrize("dims,nrhs,ns",
                         [((2, 2, 2, 3), 1, 1), ((2, 2, 2, 3), 1, 2), ((4, 4, 4, 4), 1, 37), ((3, 5, 4, 6), 5, 11),
                          ((4, 4, 4, 4), 30, 3), ((6, 6, 4, 5), 3, 700), ((8, 8, 8, 8), 2, 5)],
                         ids=["one-node", "two-nodes", "4^4-37", "ragged-5src-11", "many-sources", "more-nodes-than-blocks",
                              "8^4-one-group"])
def test_node_groups(gpu_lib, dims, nrhs, ns, m0):
    """One group per node, groups of unequal size, nodes that converge at different iterations
    (groups that run empty), and a single group."""
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 4101, m0=m0)
    ctx.set_contour(*_nodes(ns), 0.2)
    b = S.gaussian_spinor(dims, 4102, n=nrhs) if nrhs > 1 else S.gaussian_spinor(dims, 4102)
    want, _ = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64_regen")
    got, st = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64")
    again, _ = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64")
    assert st["converged"] == 1 and st["node_updates"] > 0
    assert np.array_equal(got, again)  # the groups' parts are added in a fixed order
    d = (got - want).reshape(nrhs, -1)
    assert np.all(np.linalg.norm(d, axis=1) <= 8 * TOL * np.linalg.norm(b.reshape(nrhs, -1), axis=1))


@pytest.mark.parametrize("m0", [1.4, -0.5])
@pytest.mark.parametrize("max_iter,nrhs", [(1, 1), (7, 2), (8, 1), (9, 3), (16, 1), (45, 2)])
def test_iteration_limit(gpu_lib, max_iter, nrhs, m0):
    """The best iterate at a limit inside, at and beyond a batch of iterations.  Both forms then
    hold the same Galerkin iterate of max_iter vectors; over so few iterations rounding differs
    by far less than 1e-12 ||b||, and converged nodes by at most the 8 tol ||b|| above."""
    dims = (4, 4, 4, 6)
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 4111, m0=m0)
    z, c = _nodes(12)
    ctx.set_contour(z.real + 0.05j * z.imag, c, 0.2)
    b = S.gaussian_spinor(dims, 4112, n=nrhs) if nrhs > 1 else S.gaussian_spinor(dims, 4112)

    def run(mode):
        bd = to_dev(b)
        out = torch.empty_like(bd)
        st = ctx.sgn(bd, out, nrhs, ctx.opts(tol=TOL, mode=mode, max_iter=max_iter), allow_not_converged=True)
        torch.cuda.synchronize()
        return to_host(out), st

    want, ws = run("fp64_regen")
    got, st = run("fp64")
    assert st["converged"] == ws["converged"] == 0
    assert st["iterations"] == max_iter and st["node_updates"] == 12 * nrhs * max_iter
    d = (got - want).reshape(nrhs, -1)
    assert np.all(np.linalg.norm(d, axis=1) <= 9 * TOL * np.linalg.norm(b.reshape(nrhs, -1), axis=1))


def test_zero_and_scaled_sources(gpu_lib):
    """A source that ends before its first iteration beside others of very different scale."""
    dims = (3, 4, 5, 4)
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 4121)
    ctx.set_contour(*_nodes(9), 0.2)
    b = S.gaussian_spinor(dims, 4122, n=4)
    b[1] = 0.0
    b[2] *= 1e-120
    b[3] *= 1e120
    want, _ = sgn_gpu(ctx, b, nrhs=4, tol=TOL, mode="fp64_regen")
    got, st = sgn_gpu(ctx, b, nrhs=4, tol=TOL, mode="fp64")
    assert st["converged"] == 1 and not np.any(got[1])
    for k in (0, 2, 3):
        assert np.linalg.norm((got[k] - want[k]) / np.abs(b[k]).max()) <= 8 * TOL * np.linalg.norm(b[k] / np.abs(b[k]).max())
