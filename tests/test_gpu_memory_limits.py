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

    take.release = held.clear
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


_LARGE = (32, 32, 32, 64)  # 402 MB per FP64 vector: what the allocator keeps for itself is small beside it
_VEC = 192 * 32**3 * 64


@pytest.mark.parametrize("vectors", [6, 8, 10, 12])
def test_spectral_bounds_without_room_for_integer_vectors(gpu_lib, ballast, vectors):
    """The FP64 forms of H^2 take a ring of three vectors, the start vector and two products; the
    integer ones more.  Over 8 steps no Ritz value has converged, and rounding differs by less
    than 1e-11 ||H|| (||H||^2 in the squared one, whose root the gap is)."""
    import torch

    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand((4,) + _LARGE[::-1] + (3, 3)).contiguous()
    ctx = gpu_lib.Context(_LARGE, bc_t=-1, m0=1.6)
    ctx.set_gauge(U)
    want = ctx.place_contour(8, steps=8)
    ctx.close()
    ctx = gpu_lib.Context(_LARGE, bc_t=-1, m0=1.6)
    ctx.set_gauge(U)
    ballast(vectors * _VEC + (300 << 20))
    got = ctx.place_contour(8, steps=8)
    assert got["steps"] == want["steps"] == 8
    for key in ("lambda_min", "lambda_max", "abs_max_bound"):
        assert abs(got[key] - want[key]) <= 1e-11 * 8
    assert abs(got["gap"] ** 2 - want["gap"] ** 2) <= 1e-11 * 64
    ctx.close()


@pytest.mark.parametrize("call,vectors", [("hw", 0), ("bounds", 3), ("sgn", 4)])
def test_integer_links_give_way(gpu_lib, ballast, call, vectors):
    """The integer copy of the links takes three vectors' memory.  A call that fits without it and
    not beside it runs in FP64: the stencil within 2^-43 of the largest component of the integer
    one, a solve within its tolerance (two solves: 8 tol ||b||, sum_j |c_j / Im z_j| < 4)."""
    import torch

    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand((4,) + _LARGE[::-1] + (3, 3)).contiguous()
    gen = torch.Generator(device="cuda").manual_seed(7011)
    b = torch.randn(_LARGE[::-1] + (4, 3), dtype=torch.complex128, device="cuda", generator=gen)
    z = np.array([0.3 + 0.9j, 0.3 - 0.9j, -1.5 + 1.1j, -1.5 - 1.1j])
    c = np.array([0.4 - 0.3j, 0.4 + 0.3j, -0.7 + 0.2j, -0.7 - 0.2j])
    out = []
    for limit in (False, True):
        ctx = gpu_lib.Context(_LARGE, bc_t=-1, m0=1.6)
        ctx.set_gauge(U)
        ctx.set_contour(z, c, 0.2)
        x = torch.empty_like(b)
        if limit:
            ballast(vectors * _VEC + (300 << 20))
        if call == "hw":
            ctx.apply_HW(b, x, 1, gpu_lib.OV_FP64)
        elif call == "sgn":
            ctx.sgn(b, x, 1, ctx.opts(mode="fp64_2pass", tol=1e-12))
        else:
            r = ctx.place_contour(8, steps=8)
            x = torch.tensor([r["lambda_min"], r["lambda_max"], r["gap"] ** 2])
        torch.cuda.synchronize()
        out.append(x)
        ctx.close()
    d = (out[1] - out[0]).abs()
    if call == "hw":
        assert d.max().item() <= 2.0**-43 * b.abs().max().item()
    elif call == "sgn":
        assert torch.linalg.norm(d).item() <= 8e-12 * torch.linalg.norm(b).item()
    else:
        assert d.max().item() <= 1e-11 * 64


def test_set_gauge_after_one_that_did_not_fit(gpu_lib, ballast):
    """The first of three link fields fits and the second does not: an error, and a later call
    with room for all of them starts anew."""
    import torch

    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand((4,) + _LARGE[::-1] + (3, 3)).contiguous()
    b = torch.ones(_LARGE[::-1] + (4, 3), dtype=torch.complex128, device="cuda")
    x = torch.empty_like(b)
    ctx = gpu_lib.Context(_LARGE, bc_t=1, m0=1.6)
    ballast(U.numel() * 16 + (300 << 20))
    with pytest.raises(gpu_lib.OvError) as e:
        ctx.set_gauge(U)
    assert e.value.code == gpu_lib.OV_ERR_OUT_OF_MEMORY
    ballast.release()
    torch.cuda.empty_cache()
    ctx.set_gauge(U)
    ctx.apply_HW(b, x, 1, gpu_lib.OV_FP64)
    torch.cuda.synchronize()
    ctx.close()
    want = b * torch.tensor([-1.6, -1.6, 1.6, 1.6], dtype=torch.float64, device="cuda")[:, None]  # gamma5 (-m0) on a constant field
    assert (x - want).abs().max().item() <= 2.0**-43
