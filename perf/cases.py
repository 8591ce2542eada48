"""Performance cases of the overlap library, through the calls a user's program makes.

A case names a lattice, a call and its options.  The lattices, node counts, source
counts and link roughnesses are those of the benchmark's workloads and of the tests
(4^4, 8^4, 16^4, 16^3 x 32, ragged lattices), the source kinds are the two a user has:
Gaussian noise vectors and spin-colour point sources.  Links and sources are drawn on
the GPU from the seed alone.

Kinds of call:
  hw       Context.apply_HW, FP64 or FP32, on canonical fields
  sgn      ops.sgn_apply: S_N b on a loaded gauge field and contour
  overlap  ops.overlap_apply: D_ov(m_q) b
  grad     ops.sgn and its backward: S_N b, its gradient in b and the link force
  solve    Context.overlap_solve: D_ov(m_q)^-1 b
  setup    what a new gauge configuration costs: Context.set_gauge, then the Lanczos
           bounds and the Zolotarev node set of Context.place_zolotarev
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2204_01583_gb300 import lib, ops

M0 = 1.6
# One ellipse for every sign workload: ||H_W|| <= 6.4 for SU(3) links at m0 = 1.6, so the
# ellipse from 0 to 6.72 encloses the positive spectrum of any configuration.
GAMMA, RHO, ALPHA = 3.36, 3.36, 0.25


def listed():
    return [
        # the smallest call: one stencil on the smallest lattice (latency of a call)
        dict(name="hw64-4^4-1rhs", kind="hw", lx=4, ly=4, lz=4, lt=4, eps=0.3, prec="fp64", nrhs=1),
        # multi-source stencil, the propagator's 12 spin-colour components, both precisions
        dict(name="hw64-16^3x32-12rhs", kind="hw", lx=16, ly=16, lz=16, lt=32, eps=0.6, prec="fp64", nrhs=12),
        dict(name="hw32-16^3x32-12rhs", kind="hw", lx=16, ly=16, lz=16, lt=32, eps=0.6, prec="fp32", nrhs=12),
        # ragged lattice, odd source count
        dict(name="hw32-6x10x7x9-5rhs", kind="hw", lx=6, ly=10, lz=7, lt=9, eps=0.5, prec="fp32", nrhs=5),
        # a single source on the smallest lattice with the default options (per-node vectors)
        dict(name="sgn-4^4-default-1src", kind="sgn", lx=4, ly=4, lz=4, lt=4, eps=0.3, mode="fp64", n_q=32,
             rule="ellipse", nsrc=1, src="gauss", tol=1e-12),
        # noise vectors on the paper's 8^4 lattice
        dict(name="overlap-8^4-2pass-4src", kind="overlap", lx=8, ly=8, lz=8, lt=8, eps=0.5, m_q=0.05,
             mode="fp64_2pass", n_q=64, rule="ellipse", nsrc=4, src="gauss", tol=1e-12),
        # ragged lattice, odd source count, optimal rational nodes, double-float mode
        dict(name="sgn-6x10x4x14-f32x2-3src", kind="sgn", lx=6, ly=10, lz=4, lt=14, eps=0.4, mode="f32x2", n_q=32,
             rule="zolotarev", nsrc=3, src="gauss", tol=1e-12),
        # point-source propagator columns, the batched double-float form
        dict(name="overlap-16^4-f32x2-12pt", kind="overlap", lx=16, ly=16, lz=16, lt=16, eps=0.5, m_q=0.05,
             mode="f32x2", n_q=64, rule="ellipse", nsrc=12, src="point", tol=1e-12),
        # the benchmark's own step: FP64, 12 point sources on the largest lattice
        dict(name="overlap-16^3x32-2pass-12pt", kind="overlap", lx=16, ly=16, lz=16, lt=32, eps=0.6, m_q=0.01,
             mode="fp64_2pass", n_q=64, rule="ellipse", nsrc=12, src="point", tol=1e-12),
        # forward and backward of the sign function (source gradient and link force)
        dict(name="grad-8^4-f32x2", kind="grad", lx=8, ly=8, lz=8, lt=8, eps=0.4, mode="f32x2", n_q=48,
             rule="ellipse", nsrc=1, src="gauss", tol=1e-12),
        # quark propagator: overlap inversions
        dict(name="solve-8^4-f32x2-4src", kind="solve", lx=8, ly=8, lz=8, lt=8, eps=0.5, m_q=0.05, mode="f32x2",
             n_q=64, rule="ellipse", nsrc=4, src="gauss", tol=1e-12, outer_tol=1e-10),
        # a new gauge configuration: load, spectral bounds, node set
        dict(name="setup-12^3x24", kind="setup", lx=12, ly=12, lz=12, lt=24, eps=0.5, n_poles=16, steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, vmax):
    """Extents of 4 to 16 (time to 32), odd ones among them, of at most vmax sites."""
    while True:
        d = [rng.randint(4, 16) for _ in range(3)] + [_log_int(rng, 4, 32)]
        v = d[0] * d[1] * d[2] * d[3]
        # spread over the logarithm of the volume, not crowded at its top
        if v <= vmax and v <= math.exp(rng.uniform(math.log(256), math.log(vmax))):
            return dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3])


def draw(rng):
    kind = rng.choice(["hw", "hw", "sgn", "overlap", "overlap", "grad", "solve", "setup"])
    c = dict(kind=kind)
    if kind == "hw":
        c.update(_dims(rng, 131072), eps=rng.choice([0.3, 0.5, 0.6]), prec=rng.choice(["fp64", "fp32"]),
                 nrhs=_log_int(rng, 1, 12))
        return c
    if kind == "setup":
        c.update(_dims(rng, 65536), eps=rng.choice([0.4, 0.5]), n_poles=rng.randint(8, 20), steps=rng.randint(60, 120))
        return c
    if kind == "grad":
        c.update(_dims(rng, 6144), eps=rng.choice([0.3, 0.4]), mode=rng.choice(["fp64_2pass", "f32x2"]),
                 n_q=2 * rng.randint(8, 24), rule="ellipse", nsrc=1, src="gauss", tol=1e-12)
        return c
    if kind == "solve":
        c.update(_dims(rng, 2048), eps=rng.choice([0.3, 0.5]), m_q=rng.choice([0.05, 0.1, 0.2]),
                 mode=rng.choice(["fp64_2pass", "f32x2"]), n_q=2 * rng.randint(12, 32), rule="ellipse",
                 nsrc=rng.randint(1, 3), src="gauss", tol=1e-12, outer_tol=rng.choice([1e-8, 1e-10]))
        return c
    mode = rng.choice(["fp64", "fp64_2pass", "fp64_2pass", "f32x2", "f32x2"])
    c.update(_dims(rng, 4096 if mode == "fp64" else 32768), eps=rng.choice([0.3, 0.4, 0.5]), mode=mode)
    if kind == "overlap":
        c.update(m_q=rng.choice([0.01, 0.05, 0.1]))
    if mode != "fp64" and rng.random() < 0.4:
        c.update(nsrc=12, src="point")
    else:
        c.update(nsrc=rng.randint(1, 6), src="gauss")
    rule = rng.choice(["ellipse", "ellipse", "zolotarev"])
    c.update(n_q=2 * rng.randint(8, 32), rule=rule, tol=rng.choice([1e-10, 1e-12]))
    return c


# ------------------------------------------------------------------ inputs

def _dims_of(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _volume(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"]


def _gell_mann(dev):
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    lam[0][0, 1] = lam[0][1, 0] = 1
    lam[1][0, 1], lam[1][1, 0] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[3][0, 2] = lam[3][2, 0] = 1
    lam[4][0, 2], lam[4][2, 0] = -1j, 1j
    lam[5][1, 2] = lam[5][2, 1] = 1
    lam[6][1, 2], lam[6][2, 1] = -1j, 1j
    lam[7][0, 0] = lam[7][1, 1] = 1 / math.sqrt(3)
    lam[7][2, 2] = -2 / math.sqrt(3)
    return torch.from_numpy(lam).to(dev)


def _links(case, gen):
    """SU(3) links exp(i eps sum_a theta_a lambda_a / 2), theta_a ~ N(0, 1)."""
    lx, ly, lz, lt = _dims_of(case)
    theta = torch.randn((4 * lt * lz * ly * lx, 8), generator=gen, device="cuda", dtype=torch.float64)
    x = (0.5j * case["eps"]) * (theta.to(torch.complex128) @ _gell_mann("cuda").reshape(8, 9)).reshape(-1, 3, 3)
    # exp by scaling and squaring of its Taylor series (||x|| is a few units at most)
    x = x / 64
    u = torch.eye(3, dtype=torch.complex128, device="cuda") + x / 14
    for k in range(13, 0, -1):
        u = torch.eye(3, dtype=torch.complex128, device="cuda") + (x @ u) / k
    for _ in range(6):
        u = u @ u
    return u.reshape(4, lt, lz, ly, lx, 3, 3).contiguous()


def _gauss(case, gen, n, dtype=torch.complex128):
    lx, ly, lz, lt = _dims_of(case)
    return torch.randn((n, lt, lz, ly, lx, 4, 3), generator=gen, device="cuda", dtype=dtype)


def _sources(case, gen):
    if case["src"] == "gauss":
        return _gauss(case, gen, case["nsrc"])
    # the 12 spin-colour point sources at one site of the lattice
    lx, ly, lz, lt = _dims_of(case)
    x, y, z, t = (int(torch.randint(0, m, (1,), generator=gen, device="cuda")) for m in (lx, ly, lz, lt))
    b = torch.zeros((12, lt, lz, ly, lx, 4, 3), device="cuda", dtype=torch.complex128)
    for k in range(12):
        b[k, t, z, y, x, k // 3, k % 3] = 1.0
    return b


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    U = _links(case, gen)
    ctx = lib.Context(_dims_of(case), bc_t=-1, m0=M0)
    s = dict(case=case, ctx=ctx)
    if case["kind"] == "setup":
        s["U"] = U
        return s
    ctx.set_gauge(U)
    if case["kind"] == "hw":
        fp32 = case["prec"] == "fp32"
        s["psi"] = _gauss(case, gen, case["nrhs"], torch.complex64 if fp32 else torch.complex128)
        s["out"] = torch.empty_like(s["psi"])
        s["prec"] = lib.OV_FP32 if fp32 else lib.OV_FP64
        return s
    if case["rule"] == "ellipse":
        ctx.set_contour_ellipse(case["n_q"], GAMMA, RHO, ALPHA)
    else:
        # the spectrum's usual bounds: gap about 0.2 to 0.3, ||H_W|| <= 6.4
        ctx.set_contour_zolotarev(case["n_q"] // 2, 0.2, 6.4)
    s["opts"] = ctx.opts(mode=case["mode"], tol=case["tol"])
    s["b"] = _sources(case, gen)
    if case["kind"] == "grad":
        s["b"] = s["b"][0].requires_grad_()
        s["eta"] = _gauss(case, gen, 1)[0]
        s["omega"] = torch.zeros(ops.force_shape(_dims_of(case)), dtype=torch.float64, device="cuda").requires_grad_()
    if case["kind"] == "solve":
        s["x"] = torch.empty_like(s["b"])
    return s


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "hw":
        ctx.apply_HW(state["psi"], state["out"], case["nrhs"], state["prec"])
        return state["out"]
    if kind == "sgn":
        return ops.sgn_apply(ctx, state["b"], state["opts"])
    if kind == "overlap":
        return ops.overlap_apply(ctx, case["m_q"], state["b"], state["opts"])
    if kind == "grad":
        s = ops.sgn(ctx, state["b"], state["omega"], state["opts"])
        gb, gw = torch.autograd.grad(s, (state["b"], state["omega"]), grad_outputs=state["eta"])
        return {"s": s.detach(), "grad_b": gb, "grad_links": gw}
    if kind == "solve":
        ctx.overlap_solve(case["m_q"], state["b"], state["x"], case["nsrc"], inner=state["opts"],
                          tol=case["outer_tol"])
        return state["x"]
    ctx.set_gauge(state["U"])
    ctx.place_zolotarev(case["n_poles"], case["steps"])
    z, c, _ = ctx.get_contour()
    return {"z": z, "c": c}


# -------------------------------------------------------------------- work

def work(case):
    """Bytes: links, inputs and outputs once.  Flops: 1368 per site for every application of
    H_W the path needs; a shifted solve to tol needs about (||H_W|| / gap) log(2 / tol)
    Krylov steps (6.4 / 0.36 for these links), an overlap inversion two of them in each of
    about 10 + 2 / m_q conjugate-gradient steps at a mean tolerance of 1e-8."""
    v, kind = _volume(case), case["kind"]
    per = 12 * v  # complex numbers of a spinor
    if kind == "hw":
        size = 8 if case["prec"] == "fp32" else 16
        return dict(bytes=36 * v * size + 2 * per * size * case["nrhs"], flops=1368.0 * v * case["nrhs"])
    if kind == "setup":
        return dict(bytes=36 * v * 16, flops=3 * 1368.0 * v * case["steps"])
    steps = 6.4 / 0.36 * math.log(2.0 / case["tol"])
    n = case["nsrc"]
    if kind == "grad":
        return dict(bytes=36 * v * 16 + 4 * per * 16 + 32 * v * 8, flops=3 * steps * 1368.0 * v)
    if kind == "solve":
        outer = 10 + 2 / case["m_q"]
        steps = 6.4 / 0.36 * math.log(2.0 / 1e-8) * 2 * outer
    return dict(bytes=36 * v * 16 + 2 * per * 16 * n, flops=steps * 1368.0 * v * n)


# ------------------------------------------------- the same numbers in 64 bits

def _gammas():
    s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
    z = np.zeros((2, 2))
    g = [np.block([[z, -1j * m], [1j * m, z]]) for m in s] + [np.block([[z, np.eye(2)], [np.eye(2), z]])]
    return [torch.from_numpy(np.asarray(m, dtype=np.complex128)).cuda() for m in g]


def _h_w(U, psi):
    """H_W psi for psi[n][t][z][y][x][4][3] in 64 bits, antiperiodic time."""
    g = _gammas()
    one = torch.eye(4, dtype=torch.complex128, device="cuda")
    out = (4.0 - M0) * psi
    for mu in range(4):
        ax = -3 - mu
        lt = psi.shape[1]
        fwd, bwd = torch.roll(psi, -1, ax), torch.roll(psi, 1, ax)
        if mu == 3:
            sign = torch.ones(lt, dtype=torch.float64, device="cuda")
            sign[lt - 1] = -1.0
            fwd = fwd * sign.reshape(1, lt, 1, 1, 1, 1, 1)
            bwd = bwd * torch.roll(sign, 1).reshape(1, lt, 1, 1, 1, 1, 1)
        u = U[mu].unsqueeze(0)
        ub = torch.roll(U[mu], 1, 3 - mu).unsqueeze(0)  # axes (t, z, y, x) of U[mu]
        # rows of psi are spins: (psi M^T) acts with M on colour
        out = out - 0.5 * ((one - g[mu]) @ (fwd @ u.transpose(-1, -2)) + (one + g[mu]) @ (bwd @ ub.conj()))
    out[..., 2:, :] *= -1
    return out


def _rule(case):
    n = case["n_q"]
    if case["rule"] == "ellipse":
        th = 2 * np.pi * (np.arange(1, n + 1) - 0.5) / n
        z = GAMMA + RHO * (np.cos(th) + 1j * ALPHA * np.sin(th))
        return z, 2 * RHO / n * (ALPHA * np.cos(th) + 1j * np.sin(th)), -1.0
    return None


def _lanczos(U, b, nodes, tol=1e-16, kmax=1200):
    """Orthonormal Krylov basis V (fully reorthogonalised), T, ||b||: H V = V T to within tol at
    every node."""
    shape, n = b.shape, b.numel()
    nrm = torch.linalg.vector_norm(b)
    V = torch.empty((kmax, n), dtype=torch.complex128, device="cuda")
    V[0] = b.reshape(-1) / nrm
    al, be = [], []
    for k in range(kmax - 1):
        w = _h_w(U, V[k].reshape((1,) + shape)).reshape(-1)
        al.append(float(torch.vdot(V[k], w).real))
        for _ in range(2):
            w = w - (V[: k + 1].conj() @ w) @ V[: k + 1]
        be.append(float(torch.linalg.vector_norm(w)))
        if be[-1] < 1e-13:
            break
        V[k + 1] = w / be[-1]
        if k % 25 == 24:
            th, Q = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
            last = np.abs((Q[-1] * Q[0]) @ (1.0 / (nodes[None, :] - th[:, None])))
            if be[-1] * last.max() < tol:
                break
    th, Q = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    return V[: len(al)], th, Q, float(nrm)


def _combine(V, y, shape):
    return (torch.from_numpy(np.ascontiguousarray(y, dtype=np.complex128)).cuda() @ V).reshape(shape)


def _sign(U, b, z, c, c0):
    V, th, Q, nrm = _lanczos(U, b, z)
    r = c0 + (c[None, :] / (z[None, :] - th[:, None])).sum(1)
    return _combine(V, nrm * (Q @ (r * Q[0])), b.shape)


def exact(case, seed):
    kind, v = case["kind"], _volume(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    U = _links(case, gen)
    if kind == "hw":
        single = case["prec"] == "fp32"
        psi = _gauss(case, gen, case["nrhs"], torch.complex64 if single else torch.complex128)
        return torch.cat([_h_w(U, p.to(torch.complex128)) for p in psi.split(1)])
    # an inversion, the Lanczos bounds (their start vector is the library's own) and the
    # solves that take too long have no such value
    if kind in ("solve", "setup") or case["rule"] != "ellipse" or v * case["nsrc"] > 40000:
        return None
    z, c, c0 = _rule(case)
    b = _sources(case, gen)
    if kind in ("sgn", "overlap"):
        s = torch.stack([_sign(U, x, z, c, c0) for x in b])
        if kind == "sgn":
            return s
        m = case["m_q"]
        s[..., 2:, :] *= -1
        return 0.5 * (1 + m) * b + 0.5 * (1 - m) * s
    # gradients of Re <eta, S_N b>: resolvent solutions from the Krylov bases of b and eta
    b, eta = b[0], _gauss(case, gen, 1)[0]
    sols = []
    for x, nodes in ((b, z), (eta, z.conj())):
        V, th, Q, nrm = _lanczos(U, x, nodes)
        y = nrm * ((Q[0] / (nodes[:, None] - th[None, :])) @ Q.T)
        sols.append((_combine(V, y, (len(z),) + tuple(x.shape)), V, th, Q, nrm))
    y, xi = sols[0][0], sols[1][0]

    def rational(entry, cc, shape):
        _, V, th, Q, nrm = entry
        nodes = z if cc is c else z.conj()
        r = np.conj(c0) + (cc[None, :] / (nodes[None, :] - th[:, None])).sum(1)
        return _combine(V, nrm * (Q @ (r * Q[0])), shape)

    s, gb = rational(sols[0], c, b.shape), rational(sols[1], c.conj(), b.shape)
    # dL = Re sum_j c_j <xi_j, dH y_j>, and H is linear in the links
    Ug = U.clone().requires_grad_()
    cj = torch.from_numpy(c).cuda()
    total = torch.zeros_like(U)
    for j in range(0, len(z), 8):
        hy = _h_w(Ug, y[j:j + 8])
        L = (cj[j:j + 8] * (xi[j:j + 8].conj() * hy).flatten(1).sum(1)).sum().real
        total += torch.autograd.grad(L, Ug)[0]
    # U -> exp(i omega_a lambda_a / 2) U
    f = [(total.conj() * (0.5j * (lam @ U))).sum((-1, -2)).real for lam in _gell_mann("cuda")]
    return {"s": s, "grad_b": gb, "grad_links": torch.stack(f, -1)}
