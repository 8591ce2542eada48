"""The first FP32 ov_apply_HW of a context and source count, which tries every variant (GPU)."""
import time

import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import make_ctx, to_dev

pytestmark = pytest.mark.gpu


def test_trials_cost_less_than_thirty_calls(gpu_lib):
    """Two runs of each of the six variants, the slowest of which takes twice the time of the
    fastest at this size: 19 calls of the chosen one, and allocations."""
    import torch

    dims, n = (16, 16, 16, 32), 12
    x = torch.randn((n,) + dims[::-1] + (4, 3), dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)

    def seconds(ctx, calls):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(calls):
            ctx.apply_HW(x, y, n, gpu_lib.OV_FP32)
        torch.cuda.synchronize()
        return (time.perf_counter() - t) / calls

    first, later = [], []
    for k in range(6):
        ctx, _ = make_ctx(gpu_lib, dims, 0.0, 0)
        first.append(seconds(ctx, 1))
        later.append(seconds(ctx, 20))
        ctx.close()
    assert np.median(first[1:]) <= 30 * np.median(later)  # the very first one loads the kernels


def test_trials_stay_out_of_the_kernel_times(gpu_lib):
    import torch

    dims, n = (8, 8, 8, 9), 8  # beyond the size up to which nothing is tried
    ctx, _ = make_ctx(gpu_lib, dims, 0.3, 8001)
    x = torch.randn((n,) + dims[::-1] + (4, 3), dtype=torch.complex64, device="cuda")
    ctx.set_kernel_timing(True)
    ctx.apply_HW(x, torch.empty_like(x), n, gpu_lib.OV_FP32)
    torch.cuda.synchronize()
    times = ctx.kernel_times()
    assert times["hw_kernel"][0] == 1 and times["layout_kernels"][0] in (1, 2)  # unpacking: some variants


@pytest.mark.parametrize("dims,n", [((4, 4, 4, 4), 1), ((8, 8, 8, 8), 2), ((16, 16, 16, 16), 12)])
def test_links_that_are_not_su3(gpu_lib, dims, n):
    """The forms that rebuild row 2 of a link from rows 0 and 1 are left out on links of another
    norm, and come back with SU(3) ones.  FP32 against FP64: 2e-6, the oracle tests' bound."""
    import torch

    U = to_dev(S.su3_links(dims, 0.5, 8011))
    ctx = gpu_lib.Context(dims, bc_t=-1, m0=1.6)
    x = torch.randn((n,) + dims[::-1] + (4, 3), dtype=torch.complex64, device="cuda")
    y, x64 = torch.empty_like(x), x.to(torch.complex128)
    want = torch.empty_like(x64)
    for factor in (1.0, 0.7, 1.2, 1.0):
        ctx.set_gauge(factor * U)
        ctx.apply_HW(x, y, n, gpu_lib.OV_FP32)
        ctx.apply_HW(x64, want, n, gpu_lib.OV_FP64)
        torch.cuda.synchronize()
        assert (y.to(torch.complex128) - want).abs().max().item() <= 2e-6 * want.abs().max().item(), factor


@pytest.mark.parametrize("dims,n", [((4, 4, 4, 4), 1), ((6, 10, 7, 9), 5), ((8, 8, 8, 8), 8), ((3, 5, 4, 6), 91)])
def test_small_calls_try_nothing(gpu_lib, dims, n):
    """Up to 32768 sites times sources one kernel is taken unseen: results do not depend on the
    context, and are within FP32 rounding (2e-6) of FP64."""
    import torch

    x = torch.randn((n,) + dims[::-1] + (4, 3), dtype=torch.complex64, device="cuda")
    out = []
    for _ in range(4):
        ctx, _ = make_ctx(gpu_lib, dims, 0.5, 8021)
        out.append(torch.empty_like(x))
        ctx.apply_HW(x, out[-1], n, gpu_lib.OV_FP32)
    x64 = x.to(torch.complex128)
    want = torch.empty_like(x64)
    ctx.apply_HW(x64, want, n, gpu_lib.OV_FP64)
    torch.cuda.synchronize()
    assert all(torch.equal(o, out[0]) for o in out)
    assert (out[0].to(torch.complex128) - want).abs().max().item() <= 2e-6 * want.abs().max().item()
