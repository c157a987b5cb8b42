"""GPU: the triangular normal basis of native FP64 (every degree, the default and the factorial weights,
orders of weight 0) and the jump vectors that negative weights run, against the oracle at the
library's FP64 bound (1e-12), and energies x^T G x of rough and of smooth x; a batch that
mixes weights equals single applies bit for bit."""
import numpy as np
import pytest

from oracle.ghost_penalty import Oracle
from paper_2503_00246_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _weights(kind, k):
    if kind == "first":                # only the first order
        return [0.5] + [0.0] * (k - 1)
    if kind == "last":
        return [0.0] * (k - 1) + [0.5]
    if kind == "negative":
        return [0.5 - 0.7 * (j % 2) for j in range(k)]
    return W.paper_weights(0.5, k) if kind == "paper" else None


def _apply(gp, torch, ctx, x):
    xd = torch.tensor(x, device="cuda")
    yd = torch.full_like(xd, float("nan"))
    gp.gp_apply(ctx, xd, yd)
    torch.cuda.synchronize()
    return yd.cpu().numpy()


@pytest.mark.parametrize("kind", ["gamma", "paper", "first", "last", "negative"])
@pytest.mark.parametrize("dim,n,k", [(2, 12, k) for k in range(1, 9)] + [(3, 7, 2), (3, 6, 3), (3, 5, 5), (3, 4, 8)])
def test_fp64_weights(gplib, cuda, dim, n, k, kind):
    pr = W.small_ball(dim, n, k, seed=90 + k, weights=_weights(kind, k))
    o = Oracle(pr)
    x = W.x_vectors(pr, o.n_active)[0]
    ref = o.apply(x)
    ctx = gplib.setup_problem(pr, precision=0, path=gplib.GP_PATH_FACE_LIFT)
    y = _apply(gplib, cuda, ctx, x)
    assert np.abs(y - ref).max() <= 1e-12 * np.abs(ref).max()
    if kind != "negative":
        ex, co = W.poly_coeffs(pr)
        xs = W.poly_eval(ex, co, gplib.gp_active_dof_coords(ctx))
        for v in (x, xs):
            # a polynomial of degree k has no jumps: its energy is rounding of either sign
            assert v @ _apply(gplib, cuda, ctx, v) >= -1e-13 * np.abs(ref).max() * v.size * np.abs(v).max() ** 2


@pytest.mark.parametrize("k", [1, 3, 8])
def test_infinite_weight_is_not_dropped(gplib, cuda, k):
    pr = W.small_ball(2, 12, k, seed=90 + k, weights=[0.5] * (k - 1) + [float("inf")])
    ctx = gplib.setup_problem(pr, precision=0, path=gplib.GP_PATH_FACE_LIFT)
    assert not np.isfinite(_apply(gplib, cuda, ctx, W.x_vectors(pr, ctx.n_active)[0])).all()


@pytest.mark.parametrize("dim,n,k", [(3, 8, 3), (2, 12, 2), (3, 4, 8)])
def test_batch_of_mixed_weights(gplib, cuda, dim, n, k):
    probs = [W.small_ball(dim, n, k, seed=5, weights=_weights(kind, k)) for kind in ("gamma", "paper", "negative", "gamma")]
    ctxs = [gplib.setup_problem(pr, precision=0) for pr in probs]
    xs = [cuda.tensor(W.x_vectors(pr, c.n_active, 2).ravel(), device="cuda") for pr, c in zip(probs, ctxs)]
    ys = [cuda.full_like(x, float("nan")) for x in xs]
    b = gplib.gp_batch_create(ctxs, 2)
    assert gplib.gp_batch_info(b)[0] == 2    # the triangular bases of any weights, and the jump vectors of the negative ones
    gplib.gp_batch_apply(b, xs, ys)
    for c, x, y in zip(ctxs, xs, ys):
        for r in range(2):
            s = slice(r * c.n_active, (r + 1) * c.n_active)
            yr = cuda.empty(c.n_active, dtype=cuda.float64, device="cuda")
            gplib.gp_apply(c, x[s].contiguous(), yr)
            cuda.cuda.synchronize()
            assert cuda.equal(y[s], yr)
    gplib.gp_batch_destroy(b)
