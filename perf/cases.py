"""The work that programs have this library do, as measurable cases.

Each case is one call (or one training step) through the package's public entry points:
``FmmPreconditioner.apply``, ``apply_bc``, ``solve``, ``FmmBatch.solve`` and the differentiable
``fmm_apply`` / ``fmm_solve``.  Sizes are the library's own: the 64, 1024, 2048 and 4096
grids, the 32 right-hand sides and the uneven batch of its benchmark, the Q1 and Dirichlet
problems of its tests.

Types follow the form.  The FP64 form and every solve (FP64 recurrences in every form) take
and return FP64 fields.  A bare apply in a single-precision form (FP32, mixed TF32 or BF16)
stands for the operator inside an FP32 program, a torch model with FP32 activations: its
fields are FP32, converted at the call, since the entry point takes FP64.

Solves run to a relative residual of 1e-10, the differentiable solve's default.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda"
EPS_CHUNK = 1 << 27  # values of one block of kernel entries in exact()


def listed():
    return [
        # smallest apply: a small grid inside a torch model or an outer loop; launches and
        # latency are all of it
        dict(name="apply_128_fp32", kind="apply", n=128, p=10, leaf=64, prec="fp32", nrhs=1),
        # the library's headline call: one preconditioner apply on the 1024 x 1024 grid
        dict(name="apply_1024_tf32", kind="apply", n=1024, p=10, leaf=64, prec="mixed_tf32", nrhs=1),
        # the same operator in the plain FP64 form, the accuracy reference of a user's study
        dict(name="apply_1024_fp64", kind="apply", n=1024, p=10, leaf=64, prec="fp64", nrhs=1),
        # the largest call: 32 right-hand sides on the 4096 x 4096 grid
        dict(name="apply_4096x32_tf32", kind="apply", n=4096, p=10, leaf=64, prec="mixed_tf32", nrhs=32),
        # a training step through the operator as a layer: forward and backward
        dict(name="layer_1024_tf32", kind="layer", n=1024, p=10, leaf=64, prec="mixed_tf32", nrhs=1),
        # the boundary-integral solution with Dirichlet data, plain FP32 form
        dict(name="dirichlet_1024_fp32", kind="bc", n=1024, p=10, leaf=64, prec="fp32", nrhs=1),
        # the smallest solve: 64 x 64, p = 8, FGMRES(30)
        dict(name="fgmres_64_fp32", kind="solve", n=64, p=8, leaf=64, prec="fp32", nrhs=1, method="fgmres", op="fd5"),
        # the headline solve: 1024 x 1024, FGMRES(30), mixed TF32
        dict(name="fgmres_1024_tf32", kind="solve", n=1024, p=10, leaf=64, prec="mixed_tf32", nrhs=1, method="fgmres",
             op="fd5"),
        # several right-hand sides at once by CG, mixed BF16
        dict(name="cg_1024x4_bf16", kind="solve", n=1024, p=10, leaf=64, prec="mixed_bf16", nrhs=4, method="cg",
             op="fd5"),
        # the Q1 finite-element discretisation by CG, plain FP32
        dict(name="q1_cg_512_fp32", kind="solve", n=512, p=10, leaf=64, prec="fp32", nrhs=1, method="cg", op="q1"),
        # one step of the source inversion: forward solve and adjoint solve on 2048 x 2048
        dict(name="inversion_2048_tf32", kind="inversion", n=2048, p=10, leaf=64, prec="mixed_tf32", nrhs=1),
        # independent problems of uneven size, solved side by side
        dict(name="batch_uneven_tf32", kind="batch", p=10, leaf=64, prec="mixed_tf32", count=12, sides_seed=0),
    ]


# ------------------------------------------------------------------ drawn cases
def _log_size(rng, lo, hi):
    """A power of two in [lo, hi], the sizes that a grid side can have, evenly over the logarithm."""
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "layer", "bc", "solve", "solve", "solve", "inversion", "batch"])
    single = ["fp32", "mixed_tf32", "mixed_tf32", "mixed_bf16"]
    p = rng.choice([6, 8, 10, 10, 12])
    if kind == "batch":
        return dict(kind=kind, p=p, leaf=64, prec=rng.choice(single), count=rng.randint(2, 15),
                    sides_seed=rng.randint(1, 1 << 20))
    prec = rng.choice(single + ["fp64"])
    leaf = rng.choice([16, 64, 64, 64] if prec == "fp64" else [16, 64, 64, 64, 256])
    # nodes over all right-hand sides that keep a drawn case below the largest listed one
    cap = {"apply": 1 << 24, "layer": 1 << 22, "bc": 1 << 21, "solve": 1 << 21, "inversion": 1 << 20}[kind]
    cap = min(cap, 1 << 20) if prec == "fp64" else cap
    cap = min(cap, 1 << 18) if prec == "fp64" and kind not in ("apply", "layer") else cap
    hi = 4096 if kind == "apply" and prec != "fp64" else 1024 if prec != "fp64" or kind == "apply" else 512
    n = _log_size(rng, 32, hi)
    if leaf == 256 and n < 64:
        leaf = 64
    nrhs = 1 if kind == "inversion" else _log_int(rng, 1, max(1, min(32, cap // (n * n))))
    c = dict(kind=kind, n=n, p=p, leaf=leaf, prec=prec, nrhs=nrhs)
    if kind == "solve":
        c["op"] = rng.choice(["fd5", "fd5", "fd5", "fd5_var", "q1"])
        c["method"] = rng.choice(["fgmres", "fgmres", "gmres", "cg"]) if c["op"] != "q1" else "cg"
    return c


# ------------------------------------------------------------------ inputs
def _mixture(n, rng):
    """Sum of 16 Gaussians on the unit square (centres U[0.1, 0.9], widths U[0.01, 0.05],
    amplitudes N(0, 1)) at the interior nodes: the library's synthetic source term."""
    c = rng.uniform(0.1, 0.9, size=(16, 2))
    s = rng.uniform(0.01, 0.05, size=16)
    a = rng.standard_normal(16)
    x = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) / (n + 1)
    cx, cy, sg, am = (torch.tensor(v, dtype=torch.float64, device=DEV) for v in (c[:, 0], c[:, 1], s, a))
    ex = torch.exp(-((x[None, :] - cx[:, None]) ** 2) / (2 * sg[:, None] ** 2))
    ey = torch.exp(-((x[None, :] - cy[:, None]) ** 2) / (2 * sg[:, None] ** 2)) * am[:, None]
    return ey.T @ ex


def _sources(case, seed):
    rng = np.random.default_rng(seed)
    n, k = case["n"], case["nrhs"]
    t = torch.float64 if case["prec"] == "fp64" or case["kind"] in ("solve", "inversion") else torch.float32
    f = torch.empty((k, n, n), dtype=t, device=DEV)
    for r in range(k):
        f[r] = _mixture(n, rng)
    return f


def _sides(case):
    return [int(s) for s in np.random.default_rng(case["sides_seed"]).choice([128, 256, 512, 1024, 2048], case["count"])]


def _coefficient(n):
    """a = 1 + 0.25 sin(3 pi x) sin(2 pi y) at the (n+2)^2 nodes of the full grid."""
    t = torch.arange(n + 2, dtype=torch.float64, device=DEV) / (n + 1)
    return (1 + 0.25 * torch.sin(2 * math.pi * t)[:, None] * torch.sin(3 * math.pi * t)[None, :]).contiguous()


def _dirichlet(case, seed):
    """Smooth boundary values at the 4n element midpoints, bottom, right, top, left in turn."""
    n, k = case["n"], case["nrhs"]
    rng = np.random.default_rng(seed + 7919)
    t = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    one, zero = torch.ones_like(t), torch.zeros_like(t)
    x = torch.cat([t, one, 1 - t, zero])
    y = torch.cat([zero, t, one, 1 - t])
    g = torch.empty((k, 4 * n), dtype=torch.float64, device=DEV)
    for r in range(k):
        a, b, c = rng.uniform(0.5, 3.0, size=3)
        g[r] = torch.cos(a * x) * torch.exp(b * y) + c * x * y
    return g if case["prec"] == "fp64" else g.float()


def prepare(case, seed):
    from paper_1308_3339_gb300 import FmmBatch, FmmPreconditioner
    kind = case["kind"]
    if kind == "batch":
        sides = _sides(case)
        rng = np.random.default_rng(seed)
        return dict(kind=kind, B=FmmBatch(sides, p=case["p"], leaf_max=case["leaf"], precision=case["prec"]),
                    fs=[_mixture(s, rng).contiguous() for s in sides])
    P = FmmPreconditioner(case["n"], p=case["p"], leaf_max=case["leaf"], precision=case["prec"], n_rhs=case["nrhs"])
    s = dict(kind=kind, P=P, f=_sources(case, seed), single=case["prec"] != "fp64")
    if kind == "layer":
        rng = np.random.default_rng(seed + 104729)
        s["zbar"] = torch.stack([_mixture(case["n"], rng) for _ in range(case["nrhs"])]).to(s["f"].dtype)
    elif kind == "bc":
        s["g"] = _dirichlet(case, seed)
    elif kind == "solve":
        s["method"] = case["method"]
        if case["op"] != "fd5":
            P.set_operator(case["op"], _coefficient(case["n"]) if case["op"] == "fd5_var" else None)
    elif kind == "inversion":
        # data of a known source, with noise a hundredth of its size; the step starts at half the source
        u = _dst_solve(s["f"], "fd5")
        g = torch.Generator(device=DEV).manual_seed(seed)
        s["u_obs"] = u + 0.01 * u.std() * torch.randn(u.shape, dtype=u.dtype, device=DEV, generator=g)
        s["f"] = 0.5 * s["f"]
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    from paper_1308_3339_gb300.autograd import fmm_apply, fmm_solve
    kind, f = state["kind"], state.get("f")
    if kind == "batch":
        return state["B"].solve(state["fs"], rtol=1e-10, use_graphs=2)[0]
    P = state["P"]
    if kind == "apply":
        return P.apply(f.double()).float() if state["single"] else P.apply(f)
    if kind == "bc":
        g = state["g"]
        return P.apply_bc(f.double(), g.double()).float() if state["single"] else P.apply_bc(f, g)
    if kind == "solve":
        return P.solve(f, method=state["method"], rtol=1e-10)[0]
    f = f.detach().requires_grad_(True)
    if kind == "layer":
        z = fmm_apply(f.double(), P).float() if state["single"] else fmm_apply(f, P)
        z.backward(state["zbar"])
        return z.detach(), f.grad
    u = fmm_solve(f, P, rtol=1e-10)
    ((u - state["u_obs"]) ** 2).sum().backward()
    return u.detach(), f.grad


# ------------------------------------------------------------------ work
def _apply_flops(n, p, leaf):
    """One apply's arithmetic: the near field (37 neighbouring leaves a leaf, a multiply and an
    add a pair), the translations (about 103 sources a cell, 8 p^2 operations each) and the
    expansions of the nodes."""
    side = {16: 4, 64: 8, 256: 16}[leaf]
    cells = (n / side) ** 2 * 4 / 3
    return 2.0 * 37 * side * side * n * n + 8.0 * p * p * 103 * cells + 16.0 * p * n * n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        s = _sides(case)
        return dict(bytes=16.0 * sum(v * v for v in s), flops=7 * sum(_apply_flops(v, case["p"], case["leaf"]) for v in s))
    n, k = case["n"], case["nrhs"]
    N, one = float(n) * n * k, _apply_flops(n, case["p"], case["leaf"]) * k
    w = 8 if case["prec"] == "fp64" or kind in ("solve", "inversion") else 4
    if kind == "apply":
        return dict(bytes=2 * w * N, flops=one)
    if kind == "bc":
        return dict(bytes=2 * w * N + w * 4.0 * n * k, flops=one)
    if kind == "layer":
        return dict(bytes=4 * w * N, flops=2 * one)
    if kind == "inversion":  # two solves: f, u_obs in, u and the gradient out; at least 7 applications each
        return dict(bytes=32.0 * N, flops=14 * one)
    return dict(bytes=16.0 * N, flops=7 * one)


# ------------------------------------------------------------------ exact values, 64 bits
# The operator that the FMM approximates, summed directly.  Node units: nodes at 1 .. n in
# both directions, the square's sides at 0 and n + 1, elements of length ell = (n + 1) / n.
# rot90(r, s) turns side s to the bottom: row d - 1 then holds the nodes at distance d.
def _volume(r):
    """V r at the nodes: the lattice convolution with G = -(1/2 pi) ln|d h|, its cell mean at 0."""
    k, n, _ = r.shape
    h = 1.0 / (n + 1)
    t = torch.arange(2 * n, dtype=torch.float64, device=DEV)
    t = torch.minimum(t, 2 * n - t)
    d2 = t[:, None] ** 2 + t[None, :] ** 2
    d2[0, 0] = 1.0
    G = 0.5 * torch.log(d2) + math.log(h)
    G[0, 0] = math.log(h) - 0.5 * math.log(2) - 1.5 + math.pi / 4
    Gf = torch.fft.rfft2(G)
    out = torch.empty_like(r)
    for i in range(k):
        out[i] = torch.fft.irfft2(torch.fft.rfft2(r[i], s=(2 * n, 2 * n)) * Gf, s=(2 * n, 2 * n))[:n, :n]
    return out * (-h * h / (2 * math.pi))


def _primitive(s, d):
    """Integral of ln sqrt(s^2 + d^2) ds."""
    q = s * s + d * d
    return 0.5 * s * torch.log(torch.where(q > 0, q, torch.ones_like(q))) - s + d * torch.atan2(s, d)


def _blocks(n):
    """(distances, collocation kernel C[d, e, u], element integrals D[d, u, e], angles A[d, u, e]) in blocks."""
    h, ell = 1.0 / (n + 1), (n + 1) / n
    u = torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
    te = torch.arange(n + 1, dtype=torch.float64, device=DEV) * ell
    step = max(1, EPS_CHUNK // ((n + 1) * n))
    for d0 in range(0, n, step):
        d = torch.arange(d0 + 1, min(n, d0 + step) + 1, dtype=torch.float64, device=DEV)[:, None, None]
        y = te[:-1] + ell / 2
        C = 0.5 * torch.log((y[None, :, None] - u[None, None, :]) ** 2 + d * d) + math.log(h)
        s = te[None, None, :] - u[None, :, None]
        D = torch.diff(_primitive(s, d), dim=2) + ell * math.log(h)
        yield slice(d0, min(n, d0 + step)), C, D, torch.diff(torch.atan2(s, d), dim=2)


def _sides_of(r):
    """[4, d, u, k] views of the fields r [k, n, n] from each side."""
    return torch.stack([torch.rot90(r, s, (1, 2)).permute(1, 2, 0) for s in range(4)])


def _nodes_of(v):
    """The fields [k, n, n] that _sides_of views, summed over the sides."""
    return sum(torch.rot90(v[s].permute(2, 0, 1), -s, (1, 2)) for s in range(4))


def _boundary_points(n):
    ell, e = (n + 1) / n, n + 1.0
    t = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * ell
    one, zero = torch.full_like(t, e), torch.zeros_like(t)
    return torch.cat([t, one, e - t, zero]), torch.cat([zero, t, one, e - t])


def _boundary_matrix(n, double):
    """The single layer S (or the angles of the double layer) between the 4n elements, [point, element]."""
    h, ell, e = 1.0 / (n + 1), (n + 1) / n, n + 1.0
    x, y = _boundary_points(n)
    te = torch.arange(n + 1, dtype=torch.float64, device=DEV) * ell
    cols = []
    for u, d in ((x, y), (y, e - x), (e - x, e - y), (e - y, x)):
        s, d = te[None, :] - u[:, None], d[:, None].expand(-1, n + 1)
        if double:
            a = torch.diff(torch.atan2(s, d), dim=1)
            cols.append(torch.where(d[:, :1] > 0, a, torch.zeros_like(a)))
        else:
            cols.append((torch.diff(_primitive(s, d), dim=1) + ell * math.log(h)) * (-h / (2 * math.pi)))
    return torch.cat(cols, dim=1)


def _collocation(r):
    """V r at the 4n element midpoints, [4n, k]."""
    k, n, _ = r.shape
    h = 1.0 / (n + 1)
    R = _sides_of(r)
    out = torch.zeros((4, n, k), dtype=torch.float64, device=DEV)
    for ds, C, _, _ in _blocks(n):
        out += torch.einsum("deu,sduk->sek", C, R[:, ds])
    return out.reshape(4 * n, k) * (-h * h / (2 * math.pi))


def _layer(q, n, g=None):
    """The single layer of q (minus the double layer of g) at the nodes, [k, n, n]."""
    h, k = 1.0 / (n + 1), q.shape[1]
    out = torch.zeros((4, n, n, k), dtype=torch.float64, device=DEV)
    qs = q.reshape(4, n, k)
    for ds, _, D, A in _blocks(n):
        out[:, ds] += torch.einsum("due,sek->sduk", D, qs) * (-h / (2 * math.pi))
        if g is not None:
            out[:, ds] += torch.einsum("due,sek->sduk", A, g.reshape(4, n, k)) / (2 * math.pi)
    return _nodes_of(out)


def _exact_apply(r, g=None):
    n = r.shape[-1]
    rhs = -_collocation(r)
    if g is not None:
        rhs = rhs + 0.5 * g - _boundary_matrix(n, True) @ g / (2 * math.pi)
    return _volume(r) + _layer(torch.linalg.solve(_boundary_matrix(n, False), rhs), n, g)


def _exact_transpose(zb):
    k, n, _ = zb.shape
    h = 1.0 / (n + 1)
    Z = _sides_of(zb)
    t = torch.zeros((4, n, k), dtype=torch.float64, device=DEV)
    for ds, _, D, _ in _blocks(n):
        t += torch.einsum("due,sduk->sek", D, Z[:, ds]) * (-h / (2 * math.pi))
    c = torch.linalg.solve(_boundary_matrix(n, False).T, -t.reshape(4 * n, k)).reshape(4, n, k)
    out = torch.zeros((4, n, n, k), dtype=torch.float64, device=DEV)
    for ds, C, _, _ in _blocks(n):
        out[:, ds] += torch.einsum("deu,sek->sduk", C, c) * (-h * h / (2 * math.pi))
    return _volume(zb) + _nodes_of(out)


def _dst_solve(f, op):
    """A^{-1} b of the five-point or the Q1 operator on the unit square, through its sine eigenvectors."""
    n = f.shape[-1]
    h = 1.0 / (n + 1)
    j = torch.arange(1, n + 1, device=DEV)
    Q = torch.sin(math.pi * ((j[:, None] * j[None, :]) % (2 * (n + 1))).double() / (n + 1)) * math.sqrt(2.0 / (n + 1))
    half = torch.sin(math.pi * j.double() / (2 * (n + 1))) ** 2
    if op == "q1":
        kap, mu = 4 * half, 1 - 4 * half / 6
        lam = (kap[:, None] * mu[None, :] + mu[:, None] * kap[None, :]) / (h * h)
    else:
        lam = (4 * half[:, None] + 4 * half[None, :]) / (h * h)
    return torch.stack([Q @ ((Q @ f[i] @ Q) / lam) @ Q for i in range(f.shape[0])])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng(seed)
        return [_dst_solve(_mixture(s, rng)[None], "fd5")[0] for s in _sides(case)]
    n = case["n"]
    if kind == "solve":
        # the variable-coefficient operator has no closed-form eigenvectors
        return None if case["op"] == "fd5_var" else _dst_solve(_sources(case, seed), case["op"])
    if kind == "inversion":
        f = _sources(case, seed)
        u_true = _dst_solve(f, "fd5")
        g = torch.Generator(device=DEV).manual_seed(seed)
        u_obs = u_true + 0.01 * u_true.std() * torch.randn(u_true.shape, dtype=u_true.dtype, device=DEV, generator=g)
        u = _dst_solve(0.5 * f, "fd5")
        return u, _dst_solve(2 * (u - u_obs), "fd5")
    if n > 2048 or n * n * case["nrhs"] > 1 << 23:
        return None  # the direct sums would take minutes
    r = _sources(case, seed).double()
    if kind == "layer":
        rng = np.random.default_rng(seed + 104729)
        zb = torch.stack([_mixture(n, rng) for _ in range(case["nrhs"])])
        zb = zb if case["prec"] == "fp64" else zb.float().double()
        return _exact_apply(r), _exact_transpose(zb)
    return _exact_apply(r, _dirichlet(case, seed).double().T if kind == "bc" else None)
