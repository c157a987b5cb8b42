"""What a program that uses the ghost-penalty library has it do, as cases that can be timed and compared.

A case is a mesh, a level set, a degree, a set of weights, an arithmetic and one public entry point:

  apply    y = G x on device vectors (gp_apply)
  add      y = f, then y += G x: the ghost penalty on top of another operator's result (gp_apply_add)
  host     y = G x on page-locked host vectors, transfers included (gp_apply_host)
  batched  many problems with several right-hand sides in one call (gp_apply_batched)
  system   y = (M + K + G) x, the model system of the solver study (gp_system_apply)
  solve    (M + K + G) u = b by defect correction or by FP64 CG (gp_system_solve)

The sizes are those of the repository's workloads (paper_2503_00246_gb300/workloads.py: the 32^2 disc at
k = 2, the 64^3 ball at k = 3, the 96^3 degree sweep, the 128^3 gyroid at k = 4, the batch of balls with
n in 16..96 and k in 2..6) and odd ones between them.

exact() restates the operator in plain torch on the full lattice in 64 bits: the 1D data in 50-digit
decimal arithmetic, one dense 1D matrix per direction and face, sums by index_add.
"""
from __future__ import annotations

import functools
import math
from decimal import Decimal, getcontext

import numpy as np
import torch

FP64, FP32, FF = 0, 1, 2          # gp.GP_FP64, gp.GP_FP32, gp.GP_FP64_FF
GAMMA = 0.5


def listed():
    return [
        # the smallest workload: one 2D vmult of a small mesh, where latency and launches count
        _case("disc2d_32_k2_fp64", "apply", 2, 32, 2, FP64),
        # a 2D mesh of everyday size with an odd number of cells: few ghost faces, many untouched DoFs;
        # macro-patch stabilisation
        _case("disc2d_1023_k4_macro_fp32", "apply", 2, 1023, 4, FP32, stab=1),
        # the middle-sized 3D workload in the default arithmetic
        _case("ball3d_64_k3_fp64", "apply", 3, 64, 3, FP64),
        # the high end of the degree range on an odd mesh, in single precision
        _case("ball3d_49_k8_fp32", "apply", 3, 49, 8, FP32),
        # one degree of the 96^3 sweep in the float-float arithmetic (FP64 data, FP32 pipes)
        _case("ball3d_96_k5_ff", "apply", 3, 96, 5, FF),
        # the headline workload, 59 million DoFs, in the default arithmetic and in single precision
        # (the operator of the inner iterations of a mixed-precision solver)
        _case("gyroid3d_128_k4_fp64", "apply", 3, 128, 4, FP64, shape="gyroid"),
        _case("gyroid3d_128_k4_fp32", "apply", 3, 128, 4, FP32, shape="gyroid"),
        # the ghost penalty added onto another operator's result, small odd mesh, the paper's weights
        _case("add_ball3d_41_k2_ff", "add", 3, 41, 2, FF, weights="paper"),
        # a program whose vectors live on the host (a coupled CPU code)
        _case("host_ball3d_96_k4_fp64", "host", 3, 96, 4, FP64),
        # parameter studies: independent problems of mixed sizes and degrees, four right-hand sides each
        _case("batched_12x4_fp32", "batched", 3, 96, 6, FP32, nprob=12, nrhs=4),
        # one application of the model system, the step of every outer iteration of the solver study
        _case("system_gyroid3d_64_k4_ff", "system", 3, 64, 4, FF, shape="gyroid", weights="paper"),
        # a whole solve by defect correction (FP64-accuracy residuals, FP32 inner CG)
        _case("solve_ball3d_24_k2_ff", "solve", 3, 24, 2, FF, weights="paper"),
    ]


def _case(name, kind, dim, n, k, prec, *, shape="ball", radius=0.7, weights="gamma", stab=0, nprob=1, nrhs=1, mode=0):
    c = {"kind": kind, "dim": dim, "n": n, "k": k, "prec": prec, "shape": shape, "radius": radius,
         "weights": weights, "stab": stab, "nprob": nprob, "nrhs": nrhs, "mode": mode, "cx": 0.031, "cy": -0.017, "cz": 0.042}
    if name:
        c["name"] = name
    return c


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["apply"] * 6 + ["add", "add", "host", "batched", "system", "solve"])
    dim = rng.choice([2, 3, 3, 3])
    prec = rng.choice([FP64, FP32, FF])
    if kind == "batched":
        c = _case("", kind, 3, log_int(24, 96), rng.randint(2, 6), prec, nprob=rng.randint(2, 12), nrhs=rng.randint(1, 4))
    elif kind == "solve":
        k = rng.randint(1, 3)
        n = log_int(16, 64) if dim == 2 else log_int(8, 24)
        c = _case("", kind, dim, n, k, rng.choice([FP64, FF]), weights="paper", mode=rng.choice([0, 0, 1]))
    else:
        k = rng.randint(1, 8)
        # lattice nodes per axis, so that no drawn mesh is larger than the 128^3 mesh at k = 4
        top = {"apply": 400, "add": 400, "host": 300, "system": 256}[kind]
        n = log_int(16, min(1024, 6000 // k)) if dim == 2 else log_int(8, min(128, top // k))
        if kind == "system":
            prec = rng.choice([FP64, FF, FP32])
        c = _case("", kind, dim, n, k, prec, weights=rng.choice(["gamma", "paper"]),
                  shape=rng.choice(["ball", "gyroid"]) if dim == 3 and n >= 12 else "ball",
                  stab=rng.choice([0, 0, 0, 1]) if kind in ("apply", "add") else 0)
        if c["stab"]:
            c["weights"] = "gamma"
    c["radius"] = round(rng.uniform(0.45, 0.8), 4)
    for a in ("cx", "cy", "cz"):
        c[a] = round(rng.uniform(-0.05, 0.05), 5)
    return c


# ------------------------------------------------------------------ the problems of a case --

def _problems(case):
    """One dict per problem: mesh, level set, degree (a batch has several, of mixed sizes and degrees)."""
    if case["kind"] != "batched":
        return [dict(dim=case["dim"], n=case["n"], k=case["k"], shape=case["shape"], radius=case["radius"],
                     off=[case["cx"], case["cy"], case["cz"]][:case["dim"]], weights=case["weights"], stab=case["stab"])]
    rng = np.random.Generator(np.random.PCG64([case["n"], case["k"], case["nprob"]]))
    out = []
    for _ in range(case["nprob"]):
        out.append(dict(dim=3, n=int(rng.integers(16, case["n"] + 1)), k=int(rng.integers(2, case["k"] + 1)), shape="ball",
                        radius=float(rng.uniform(0.4, 0.8)), off=[float(v) for v in rng.uniform(-0.05, 0.05, 3)],
                        weights=case["weights"], stab=case["stab"]))
    return out


def _weights(pr):
    k = pr["k"]
    if pr["weights"] == "paper":
        return [GAMMA / math.factorial(j) ** 2 for j in range(1, k + 1)]
    return [GAMMA] * k


def _box(pr):
    return (-math.pi, math.pi) if pr["shape"] == "gyroid" else (-1.0, 1.0)


def _context(gp, W, pr, prec):
    lo, hi = _box(pr)
    p = W.Problem(name="case", dim=pr["dim"], n=pr["n"], lo=lo, hi=hi, degree=pr["k"], gamma=GAMMA,
                  weights=None if pr["weights"] == "gamma" else _weights(pr), stabilization=pr["stab"])
    if pr["shape"] == "gyroid":
        p.ls_kind, p.iso = W.LS_GYROID, 0.3
    else:
        p.centers = np.zeros((1, 3))
        p.centers[0, :pr["dim"]] = pr["off"]
        p.radii = np.array([pr["radius"]])
    return gp.setup_problem(p, precision=prec)


def _dtype(prec):
    return torch.float32 if prec == FP32 else torch.float64


def _vectors(case, seed, sizes):
    """The random vectors of a case, ~ U[-1, 1], one tensor (times two for `add`) per size."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * seed + 17)
    dt = _dtype(case["prec"])
    per = 2 if case["kind"] == "add" else 1
    return [[torch.rand(case["nrhs"] * n, generator=g, device="cuda", dtype=dt).mul_(2).sub_(1) for _ in range(per)]
            for n in sizes]


def prepare(case, seed):
    from paper_2503_00246_gb300 import gp, workloads as W

    kind, prec = case["kind"], case["prec"]
    st = {"gp": gp, "kind": kind, "case": case}
    if kind in ("system", "solve"):
        pr = _problems(case)[0]
        hi = FF if prec == FP32 else prec
        st["ctx"] = [_context(gp, W, pr, hi), _context(gp, W, pr, FP32)]
        st["sys"] = gp.gp_system_create(*st["ctx"])
        st["which"] = 1 if prec == FP32 else 0
        sizes = [st["ctx"][0].n_active]
    else:
        st["ctx"] = [_context(gp, W, pr, prec) for pr in _problems(case)]
        sizes = [c.n_active for c in st["ctx"]]
    v = _vectors(case, seed, sizes)
    st["x"] = [t[0] for t in v]
    st["y"] = [torch.empty_like(t) for t in st["x"]]
    if kind == "add":
        st["f"] = v[0][1]
    if kind == "host":
        st["x"] = [t.cpu().pin_memory() for t in st["x"]]
        st["y"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True) for t in st["x"]]
    return st


def run(st):
    gp, kind, x, y = st["gp"], st["kind"], st["x"], st["y"]
    if kind == "apply":
        gp.gp_apply(st["ctx"][0], x[0], y[0])
    elif kind == "add":
        y[0].copy_(st["f"])
        gp.gp_apply_add(st["ctx"][0], x[0], y[0])
    elif kind == "host":
        gp.gp_apply_host(st["ctx"][0], x[0], y[0])
    elif kind == "batched":
        gp.gp_apply_batched(st["ctx"], st["case"]["nrhs"], x, y)
    elif kind == "system":
        gp.gp_system_apply(st["sys"], st["which"], x[0], y[0])
    else:
        gp.gp_system_solve(st["sys"], x[0], y[0], rtol=1e-10, inner_rtol=1e-4, mode=st["case"]["mode"])
    return y


def work(case):
    """Bytes: x on the DoFs that ghost faces touch (the others' values are not needed), y on every active
    DoF; the system reads every x, a solve reads b and writes u.  Flops: the factorised apply, k jump
    values per normal line and their expansion with the mirror symmetry of the patch halved, k tangential
    lines of k + 1 values per direction and face; a cell of the system applies 1D matrices in each direction."""
    w = 4 if case["prec"] == FP32 else 8
    nbytes = flops = 0
    for pr in _problems(case):
        m = _mesh(pr)
        d, k = pr["dim"], pr["k"]
        nf = sum(len(f) for f in m["faces"])
        lines = (k + 1) ** (d - 1)
        f = nf * lines * (2 * k * (2 * k + 1) + (d - 1) * k * (k + 1))
        if case["kind"] in ("system", "solve"):
            nbytes += w * 2 * m["n_active"]
            f += m["cells"].numel() * (2 * d + 1) * (k + 1) ** (d + 1)
        else:
            nbytes += case["nrhs"] * w * (m["n_touched"] + m["n_active"] * (2 if case["kind"] == "add" else 1))
        flops += case["nrhs"] * f
    return {"bytes": int(nbytes), "flops": int(flops)}


def tolerance(case):
    """About four times what the arithmetic shows against 64 bits over the ranges of draw().  Seen: single
    precision 1.6e-7 (2-norm) and 3.7e-6 (largest), float-float 7e-15 and 1.4e-13, FP64 2.7e-16 and 5e-15, where
    another order of the sums or of the 1D factors shows a few times that; a solve, which stops at a relative
    residual of 1e-10, 2e-11 and 6e-11."""
    if case["kind"] == "solve":
        return {"rel": 1e-9, "max": 1e-8}
    return {FP32: {"rel": 1e-6, "max": 2e-5}, FF: {"rel": 3e-14, "max": 1e-12}, FP64: {"rel": 2e-15, "max": 4e-14}}[case["prec"]]


# ------------------------------------------------------- the operator in plain torch, 64 bits --

def exact(case, seed):
    probs = _problems(case)
    meshes = [_mesh(pr) for pr in probs]
    x = _vectors(case, seed, [m["n_active"] for m in meshes])
    out = []
    for pr, m, v in zip(probs, meshes, x):
        xs = v[0].double().reshape(case["nrhs"], -1)
        if case["kind"] == "solve":
            y = _cg(lambda u: _apply(pr, m, u, True), xs[0])[None]
        else:
            y = torch.stack([_apply(pr, m, u, case["kind"] == "system") for u in xs])
            if case["kind"] == "add":
                y += v[1].double()
        out.append(y.reshape(-1))
    if case["kind"] == "host":
        out = [y.cpu() for y in out]
    return out


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _cell_classes(pr):
    """0 outside, 1 cut, 2 inside, shape (n,) * d with x the last axis."""
    d, n = pr["dim"], pr["n"]
    lo, hi = _box(pr)
    if pr["shape"] == "gyroid":
        m = 4
        hs = (hi - lo) / (n * m)
        t = torch.tensor(lo + np.arange(n * m + 1) * hs, dtype=torch.float64)
        s, c = torch.sin(t).to(_device()), torch.cos(t).to(_device())
        phi = (s[None, None, :] * c[None, :, None] + s[None, :, None] * c[:, None, None]
               + s[:, None, None] * c[None, None, :]) - 0.3
        big = -torch.nn.functional.max_pool3d(-phi[None], m + 1, stride=m)[0], torch.nn.functional.max_pool3d(phi[None], m + 1, stride=m)[0]
        margin = math.sqrt(6.0) * hs * math.sqrt(3.0) / 2
        cls = torch.ones((n,) * 3, dtype=torch.int8, device=_device())
        cls[big[1] < -margin] = 0
        cls[big[0] > margin] = 2
        return cls
    h = (hi - lo) / n
    i = np.arange(n, dtype=np.float64)
    a, b = lo + i * h, lo + (i + 1) * h
    near2, far2 = 0, 0
    for ax in range(d):
        c = pr["off"][ax]
        near = np.maximum(np.maximum(a - c, c - b), 0.0)
        far = np.maximum(np.abs(a - c), np.abs(b - c))
        shape = [1] * d
        shape[d - 1 - ax] = n
        near2 = near2 + (near * near).reshape(shape)
        far2 = far2 + (far * far).reshape(shape)
    r2 = pr["radius"] ** 2
    cls = np.ones((n,) * d, dtype=np.int8)
    cls[near2 >= r2] = 0
    cls[far2 < r2] = 2
    return torch.tensor(cls, device=_device())


def _mark(cells, k):
    """The lattice nodes of the marked cells (both with x the last axis)."""
    d, n = cells.dim(), cells.shape[0]
    out = torch.zeros((n * k + 1,) * d, dtype=torch.bool, device=cells.device)
    for p in np.ndindex(*(k + 1,) * d):
        out[tuple(slice(q, q + (n - 1) * k + 1, k) for q in p)] |= cells
    return out


def _mesh(pr):
    """Ghost faces (lower cells per axis), active cells, the lattice index of every active DoF."""
    return _mesh_of(tuple((k, tuple(v) if isinstance(v, list) else v) for k, v in sorted(pr.items()) if k not in ("weights", "stab")))


@functools.lru_cache(maxsize=2)
def _mesh_of(key):
    pr = dict(key)
    d, n, k = pr["dim"], pr["n"], pr["k"]
    cls = _cell_classes(pr)
    act, cut = cls != 0, cls == 1
    faces, inv = [], torch.zeros_like(act)
    for a in range(d):
        ax = d - 1 - a
        lo, hi = act.narrow(ax, 0, n - 1), act.narrow(ax, 1, n - 1)
        sel = lo & hi & (cut.narrow(ax, 0, n - 1) | cut.narrow(ax, 1, n - 1))
        faces.append(sel.nonzero())
        inv.narrow(ax, 0, n - 1).logical_or_(sel)
        inv.narrow(ax, 1, n - 1).logical_or_(sel)
    node = _mark(act, k).reshape(-1).nonzero()[:, 0]
    return {"faces": faces, "cells": act.nonzero(), "node": node, "n_active": node.numel(), "n_touched": int(_mark(inv, k).sum())}


@functools.lru_cache(maxsize=None)
def _one_d(k):
    """Mass and stiffness (k+1)^2 on the unit interval, the jumps of the derivatives 1..k of the 2k+1 patch
    functions at the face, and the macro-patch form, from Gauss-Lobatto nodes in 50-digit arithmetic."""
    getcontext().prec = 50
    D = Decimal

    def mul(a, b):
        out = [D(0)] * (len(a) + len(b) - 1)
        for i, u in enumerate(a):
            for j, v in enumerate(b):
                out[i + j] += u * v
        return out

    def der(a):
        return [D(i) * a[i] for i in range(1, len(a))] or [D(0)]

    def val(a, x):
        s = D(0)
        for c in reversed(a):
            s = s * x + c
        return s

    def integral(a, x0, x1):
        prim = [D(0)] + [c / D(i + 1) for i, c in enumerate(a)]
        return val(prim, D(x1)) - val(prim, D(x0))

    # interior nodes: roots of P_k' on [-1, 1]
    p0, p1 = [D(1)], [D(0), D(1)]
    for m in range(1, k):
        p2 = [D(2 * m + 1) / D(m + 1) * c for c in mul([D(0), D(1)], p1)]
        for i, c in enumerate(p0):
            p2[i] -= D(m) / D(m + 1) * c
        p0, p1 = p1, p2
    dp = der(p1)
    ddp = der(dp)
    nodes = [D(-1)]
    for i in range(1, k):
        x = D(repr(-math.cos(math.pi * i / k)))
        for _ in range(60):
            x -= val(dp, x) / val(ddp, x)
        nodes.append(x)
    nodes = sorted([(x + 1) / 2 for x in nodes + [D(1)]])
    basis = []
    for i in range(k + 1):
        a = [D(1)]
        for j in range(k + 1):
            if j != i:
                a = mul(a, [-nodes[j] / (nodes[i] - nodes[j]), D(1) / (nodes[i] - nodes[j])])
        basis.append(a)
    mass = [[integral(mul(a, b), 0, 1) for b in basis] for a in basis]
    stiff = [[integral(mul(der(a), der(b)), 0, 1) for b in basis] for a in basis]
    jumps, dl = [], basis
    for _ in range(k):
        dl = [der(a) for a in dl]
        left, right = [val(a, D(1)) for a in dl], [val(a, D(0)) for a in dl]
        jumps.append([left[b] - (right[0] if b == k else D(0)) if b <= k else -right[b - k] for b in range(2 * k + 1)])
    # macro patch: over [0, 1] the squared difference of the cell's polynomial and the extension of its
    # neighbour's (basis shifted by one), and the mirror image
    def shift(a, s):
        out = [D(0)]
        for c in reversed(a):
            out = mul(out, [D(s), D(1)])
            out[0] += c
        return out

    zero = [D(0)]
    macro = [[D(0)] * (2 * k + 1) for _ in range(2 * k + 1)]
    for side in (0, 1):
        diff = []
        for b in range(2 * k + 1):
            on_lo = basis[b] if b <= k else zero
            on_hi = basis[b - k] if b >= k else zero
            # the lower cell is [0, 1], the upper [1, 2]; both polynomials in the coordinate of cell `side`
            u, v = (on_lo, shift(on_hi, -1)) if side == 0 else (on_hi, shift(on_lo, 1))
            m = max(len(u), len(v))
            diff.append([(u[i] if i < len(u) else D(0)) - (v[i] if i < len(v) else D(0)) for i in range(m)])
        for b in range(2 * k + 1):
            for c in range(2 * k + 1):
                macro[b][c] += integral(mul(diff[b], diff[c]), 0, 1)
    return tuple(np.array([[float(v) for v in r] for r in t]) for t in (mass, stiff, jumps, macro))


def _add_blocks(x, y, cells, scale, mats, k, shape):
    """y += scale * (mats[0] x mats[1] x ...) x on the blocks of nodes that begin at k * cells (axes as x's, x last)."""
    d = len(mats)
    dev = x.device
    nl = shape[0]
    stride = [nl ** (d - 1 - i) for i in range(d)]
    off = torch.zeros(1, dtype=torch.int64, device=dev)
    for i, m in enumerate(mats):
        off = (off[:, None] + torch.arange(m.shape[0], device=dev)[None] * stride[i]).reshape(-1)
    step = max(1, (1 << 26) // off.numel())
    st = torch.tensor(stride, device=dev) * k
    for i0 in range(0, cells.shape[0], step):
        idx = (cells[i0:i0 + step] * st).sum(1)[:, None] + off
        v = x[idx].reshape([-1] + [m.shape[0] for m in mats])
        for i, m in enumerate(mats):
            v = torch.tensordot(v, m, dims=([i + 1], [1])).movedim(-1, i + 1)
        y.index_add_(0, idx.reshape(-1), v.reshape(-1), alpha=scale)


def _apply(pr, m, x, system):
    """G x, or (M + K + G) x, on the active DoFs."""
    d, n, k = pr["dim"], pr["n"], pr["k"]
    dev = m["node"].device
    lo, hi = _box(pr)
    h = (hi - lo) / n
    mass, stiff, jumps, macro = (torch.tensor(t, dtype=torch.float64, device=dev) for t in _one_d(k))
    if pr["stab"]:
        normal = GAMMA * h ** d * macro
    else:
        c = torch.tensor(_weights(pr), dtype=torch.float64, device=dev) * h ** (d - 2)
        normal = (jumps * c[:, None]).T @ jumps
    shape = (n * k + 1,) * d
    full = torch.zeros(math.prod(shape), dtype=torch.float64, device=dev)
    full[m["node"]] = x.to(dev)
    y = torch.zeros_like(full)
    for a in range(d):
        mats = [mass] * d
        mats[d - 1 - a] = normal
        _add_blocks(full, y, m["faces"][a], 1.0, mats, k, shape)
    if system:
        _add_blocks(full, y, m["cells"], h ** d, [mass] * d, k, shape)
        for a in range(d):
            mats = [mass] * d
            mats[a] = stiff
            _add_blocks(full, y, m["cells"], h ** (d - 2), mats, k, shape)
    return y[m["node"]]


def _cg(op, b):
    """Conjugate gradients to a relative residual of 1e-13, restarted twice on the true residual."""
    u = torch.zeros_like(b)
    for _ in range(3):
        r = b - op(u)
        p, rr = r.clone(), torch.dot(r, r)
        stop = 1e-26 * torch.dot(b, b)
        for it in range(20000):
            if it % 50 == 0 and rr <= stop:
                break
            q = op(p)
            a = rr / torch.dot(p, q)
            u = u + a * p
            r = r - a * q
            new = torch.dot(r, r)
            p = r + (new / rr) * p
            rr = new
    return u
