"""GPU: the FP32 lift over compact face outputs at the sizes where it can go wrong: every degree that has them,
owner cells with every candidate face (a full box) and with few (a ball), lift tiles of one owner,
of more lines than threads, and larger than the shared memory (the kernel then takes fewer owners).
Against the oracle at the FP32 bound of the library (1e-5), and bitwise equal over the tiles."""
import numpy as np
import pytest

from oracle.ghost_penalty import Oracle
from paper_2503_00246_gb300 import workloads as W

pytestmark = pytest.mark.gpu


BALL = {3: 100, 4: 84, 5: 54, 6: 44, 7: 34, 8: 28}   # cells per direction of the 3D balls


# 3D meshes with more than 24 MB of W_F, above which FP32 stores compact outputs at every k >= 3, and
# small ones of the degrees that always do, as 2D does from k = 6 on (and W_F below)
@pytest.mark.parametrize("box", [False, True])
@pytest.mark.parametrize("dim,n,k", [(2, 9, k) for k in range(1, 9)] + [(3, 28, 3), (3, 22, 4), (3, 18, 5), (3, 16, 6),
                                                                       (3, 14, 7), (3, 13, 8), (3, 5, 5), (3, 3, 7),
                                                                       (3, 3, 8)])
def test_compact_lift(gplib, cuda, dim, n, k, box):
    pr = W.box_problem(dim, n, k, hi=1.0) if box else W.small_ball(dim, BALL.get(k, n) if dim == 3 and n > 5 else 2 * n, k, seed=70 + k)
    ctx = gplib.setup_problem(pr, precision=1)
    if dim == 3 and n > 5:
        assert ctx.n_faces * (2 * k + 1) * (k + 1) ** 2 * 4 > 24 << 20
    assert gplib.gp_kernel_form(ctx)["compact"] == (dim == 3 or k >= 6)
    x = W.x_vectors(pr, ctx.n_active)[0].astype(np.float32)
    o = Oracle(pr)
    rows = np.arange(ctx.n_active) if dim == 2 else np.unique(np.random.default_rng(k).integers(0, ctx.n_active, 1500))
    ref = o.apply_rows(x.astype(np.float64), rows)
    scale = np.abs(ref).max()
    xd = cuda.tensor(x, device="cuda")
    first = None
    for cells, threads in ((0, 0), (1, 32), (3, 64), (46 * 1024 // (4 * (37 if dim == 3 else 13)), 256)):
        gplib.gp_set_tiles(ctx, {"faces_per_cta": 0, "lift_cells_per_cta": cells, "lift_threads": threads})
        for add in (False, True):
            yd = cuda.ones_like(xd) if add else cuda.full_like(xd, float("nan"))
            (gplib.gp_apply_add if add else gplib.gp_apply)(ctx, xd, yd)
            cuda.cuda.synchronize()
            y = yd.double().cpu().numpy()[rows] - (1.0 if add else 0.0)
            assert np.abs(y - ref).max() <= 1e-5 * max(scale, 1.0 if add else 0.0)
            if not add:
                first = yd if first is None else first
                assert cuda.equal(yd, first), (cells, threads)


def test_batch_of_both_forms(gplib, cuda):
    """Large FP32 meshes store compact outputs and small ones W_F: a batch of both runs a pair of launches for
    each form, and every vector equals gp_apply's bit for bit."""
    probs = [W.small_ball(3, n, 4, seed=50 + n) for n in (8, 60, 10, 56)]
    ctxs = [gplib.setup_problem(pr, precision=1, path=gplib.GP_PATH_FACE_LIFT) for pr in probs]
    xs = [cuda.tensor(W.x_vectors(pr, c.n_active, 2).ravel(), dtype=cuda.float32, device="cuda") for pr, c in zip(probs, ctxs)]
    ys = [cuda.full_like(x, float("nan")) for x in xs]
    b = gplib.gp_batch_create(ctxs, 2)
    assert gplib.gp_batch_info(b)[0] == 2
    gplib.gp_batch_apply(b, xs, ys)
    for c, x, y in zip(ctxs, xs, ys):
        for r in range(2):
            s = slice(r * c.n_active, (r + 1) * c.n_active)
            yr = cuda.empty(c.n_active, dtype=cuda.float32, device="cuda")
            gplib.gp_apply(c, x[s].contiguous(), yr)
            cuda.cuda.synchronize()
            assert cuda.equal(y[s], yr)
    gplib.gp_batch_destroy(b)
