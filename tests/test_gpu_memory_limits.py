"""What calls do where device memory is short (GPU).  Memory is taken by a plain allocation."""
import numpy as np
import pytest

import synthetic as S
from tests.gpu_common import make_ctx, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture
def ballast():
    """ballast(n): allocate all but n bytes of the device, given back at the test's end."""
    import torch

    held = []

    def take(leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        held.append(torch.empty(torch.cuda.mem_get_info()[0] - int(leave), dtype=torch.uint8, device="cuda"))

    yield take
    held.clear()
    torch.cuda.empty_cache()


def test_vector_space_solves_without_room_for_the_integer_ring(gpu_lib, ballast):
    """With less than a tenth of the device free OV_MODE_FP64 declines its integer vectors before
    it allocates any: nothing is released, and a solve neither waits for other streams nor
    captures its graph again.  (A kernel on another stream outlives the solve.)"""
    import torch

    dims = (4, 4, 4, 4)
    ctx, _ = make_ctx(gpu_lib, dims, 0.3, 7001)
    ctx.set_contour_ellipse(16, 3.36, 3.36, 0.25)
    b = to_dev(S.gaussian_spinor(dims, 7002))
    out, other = torch.empty_like(b), torch.cuda.Stream()
    ballast(0.05 * torch.cuda.mem_get_info()[1])
    opts = ctx.opts(mode="fp64", tol=1e-12)
    for _ in range(2):
        st = ctx.sgn(b, out, 1, opts)
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(2_000_000_000)  # about a second
        end = torch.cuda.Event()
        end.record()
    again = ctx.sgn(b, out, 1, opts)
    running = not end.query()
    torch.cuda.synchronize()
    assert running
    assert again["iterations"] == st["iterations"] and again["converged"] == 1
