"""GPU: the error of y = G x against an extended-precision reference stays at the size of the rounding of each
arithmetic: products of constants are rounded once (line factors of the tangential masses) and the
expansions of compact face outputs are summed before they join a node's sum.  The reference takes the 1D data to
40 digits and applies it in long double (64 bits of mantissa or more).  Inputs are single-precision numbers,
so that every arithmetic sees the same x; the bounds are 2-norm errors in units of 2^-53, 2^-48 and 2^-24."""
import functools

import numpy as np
import pytest

from oracle.ghost_penalty import Oracle
from paper_2503_00246_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _ld(v):
    h = float(v)
    return LD(h) + LD(float(v - h))


@functools.lru_cache(maxsize=None)
def _one_d(k):
    """Mass and jumps of the derivatives 1..k of the Gauss-Lobatto basis in long double."""
    mp = pytest.importorskip("mpmath").mp
    mp.dps = 40
    f = mp.mpf
    val = lambda a, x: sum((v * x ** i for i, v in enumerate(a)), f(0))
    der = lambda a: [i * v for i, v in enumerate(a)][1:] or [f(0)]
    p0, p1 = [f(1)], [f(0), f(1)]
    for m in range(1, k):
        p2 = [f(0)] + [f(2 * m + 1) / (m + 1) * v for v in p1]
        for i, v in enumerate(p0):
            p2[i] -= f(m) / (m + 1) * v
        p0, p1 = p1, p2
    dp = der(p1)
    nodes = [f(-1), f(1)]
    for i in range(1, k):
        x = -mp.cos(mp.pi * i / k)
        for _ in range(40):
            x -= val(dp, x) / val(der(dp), x)
        nodes.append(x)
    nodes = sorted((x + 1) / 2 for x in nodes)
    basis = []
    for i in range(k + 1):
        a = [f(1)]
        for j in range(k + 1):
            if j != i:
                d, n = nodes[i] - nodes[j], [f(0)] * (len(a) + 1)
                for q, v in enumerate(a):
                    n[q] -= v * nodes[j] / d
                    n[q + 1] += v / d
                a = n
        basis.append(a)
    mass = [[sum(u * v / (i + j + 1) for i, u in enumerate(a) for j, v in enumerate(b)) for b in basis] for a in basis]
    jumps, dl = [], basis
    for _ in range(k):
        dl = [der(a) for a in dl]
        lo, hi = [val(a, f(1)) for a in dl], [val(a, f(0)) for a in dl]
        jumps.append([lo[b] - (hi[0] if b == k else 0) if b <= k else -hi[b - k] for b in range(2 * k + 1)])
    return tuple(np.array([[_ld(v) for v in row] for row in t]) for t in (mass, jumps))


@functools.lru_cache(maxsize=None)
def _reference(dim, n, k):
    pr = W.small_ball(dim, n, k, seed=3)
    o = Oracle(pr)
    mass, g = _one_d(k)
    h = LD(pr.h) if dim == 3 else LD(1)
    s = np.array([LD(c) * h for c in pr.cweights()])
    x = np.random.default_rng(5).uniform(-1, 1, o.n_active).astype(np.float32)
    y = np.zeros(o.n_active, LD)
    for a in range(dim):
        idx = o.patch_index(a)
        shape = [k + 1] * dim
        shape[dim - 1 - a] = 2 * k + 1                     # x is the last axis
        v = np.moveaxis(x.astype(LD)[idx].reshape([len(idx)] + shape), dim - a, 1)
        t = np.moveaxis(np.tensordot(g, v, axes=(1, 1)), 0, 1) * s.reshape([1, k] + [1] * (dim - 1))
        for q in range(dim - 1):
            t = np.moveaxis(np.tensordot(mass, t, axes=(1, 2 + q)), 0, 2 + q)
        w = np.moveaxis(np.tensordot(g.T, t, axes=(1, 1)), 0, 1)
        np.add.at(y, idx.ravel(), np.moveaxis(w, 1, dim - a).reshape(-1))
    return pr, x, y


# About a dozen independent roundings of up to half a unit each (the terms of the largest sums, the constants)
# come to 1 to 2 units in the 2-norm.  Measured: FP64 1.0 to 1.75, FP32 1.0 to 1.65, float-float 0.65 to 2.2 (k = 1 in
# 3D; 1.45 elsewhere).
BOUND = {0: 1.8 * 2.0 ** -53, 1: 1.7 * 2.0 ** -24, 2: 2.3 * 2.0 ** -48}


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("dim,n,k", [(3, 7, k) for k in (1, 2, 3, 4, 5)] + [(2, 20, k) for k in range(1, 9)]
                         + [(3, 5, 7), (3, 4, 8)])
def test_error_at_the_rounding_of_the_arithmetic(gplib, cuda, prec, dim, n, k):
    pr, x, ref = _reference(dim, n, k)
    ctx = gplib.setup_problem(pr, precision=prec, path=gplib.GP_PATH_FACE_LIFT)
    xd = cuda.tensor(x, dtype=cuda.float32 if prec == 1 else cuda.float64, device="cuda")
    yd = cuda.full_like(xd, float("nan"))
    gplib.gp_apply(ctx, xd, yd)
    cuda.cuda.synchronize()
    err = float(np.sqrt(((yd.cpu().numpy().astype(LD) - ref) ** 2).sum() / (ref ** 2).sum()))
    assert err <= BOUND[prec]
