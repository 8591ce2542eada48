"""OV_MODE_FP64 with its nodes spread over groups of blocks, against OV_MODE_FP64_REGEN (GPU).

Both forms stop at a node residual of tol ||b||, so that each differs from the quadrature sum by
at most sum_j |c_j| tol / |Im z_j| ||b||.  The nodes below keep sum_j |c_j / Im z_j| < 4 for any
count, which bounds the difference of two results by 8 tol ||b|| in norm.
"""
import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import make_ctx, sgn_gpu

pytestmark = pytest.mark.gpu

Z = np.array([0.3 + 0.9j, 0.3 - 0.9j, -1.5 + 1.1j, -1.5 - 1.1j, 4.0 + 2.0j])
C = np.array([0.4 - 0.3j, 0.4 + 0.3j, -0.7 + 0.2j, -0.7 - 0.2j, 0.5 + 0.1j])
TOL = 1e-12


@pytest.mark.parametrize("dims,nrhs,ns",
                         [((2, 2, 2, 3), 1, 1), ((2, 2, 2, 3), 1, 2), ((4, 4, 4, 4), 1, 37), ((3, 5, 4, 6), 5, 11),
                          ((4, 4, 4, 4), 30, 3), ((6, 6, 4, 5), 3, 700), ((8, 8, 8, 8), 2, 5)],
                         ids=["one-node", "two-nodes", "4^4-37", "ragged-5src-11", "many-sources", "more-nodes-than-blocks",
                              "8^4-one-group"])
def test_node_groups(gpu_lib, dims, nrhs, ns):
    """One group per node, groups of unequal size, nodes that converge at different iterations
    (groups that run empty), and a single group."""
    ctx, _ = make_ctx(gpu_lib, dims, 0.5, 4101)
    k = np.arange(ns) // 5
    z = Z[np.arange(ns) % 5].real + 1j * Z[np.arange(ns) % 5].imag * (1.0 + 0.3 * k)
    c = C[np.arange(ns) % 5] / (k[-1] + 1)
    ctx.set_contour(z, c, 0.2)
    b = S.gaussian_spinor(dims, 4102, n=nrhs) if nrhs > 1 else S.gaussian_spinor(dims, 4102)
    want, _ = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64_regen")
    got, st = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64")
    again, _ = sgn_gpu(ctx, b, nrhs=nrhs, tol=TOL, mode="fp64")
    assert st["converged"] == 1 and st["node_updates"] > 0
    assert np.array_equal(got, again)  # the groups' parts are added in a fixed order
    d = (got - want).reshape(nrhs, -1)
    assert np.all(np.linalg.norm(d, axis=1) <= 8 * TOL * np.linalg.norm(b.reshape(nrhs, -1), axis=1))
