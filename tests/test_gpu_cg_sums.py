"""The solvers' products of long rows (13- and 27-point operators), untuned: a row's sum has the parts
that its lanes would make, whatever schedule the plain SpMM takes on such an operator (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu

N = 30  # 27000 rows: above the count from which one lane takes a row


def _operator(rb, points, k, dtype="f64"):
    rp, ci, va, nc = rb.stencil_assemble((N, N, N), [1.0 / N] * 3,
                                         rb.RB_STENCIL_27P if points == 27 else rb.RB_STENCIL_13P)
    return rb.Operator(rp, ci, -va, nc, dtype=dtype, k_max=k), rp.cpu().numpy(), ci.cpu().numpy(), -va.cpu().numpy()


PARTS = {(13, 1): (1, 4), (13, 3): (3, 4), (13, 8): (2, 2), (27, 1): (1, 8), (27, 2): (2, 8), (27, 3): (3, 8), (27, 8): (2, 2)}


@pytest.mark.parametrize("points,k", sorted(PARTS))
def test_residual_sums_in_parts(rb, points, k):
    """With b = A x rounded once, the reported residual of x is the rounding of the solver's own product:
    the same with the default as with the parts asked for (the two differ only in the sums of squares)."""
    A, rp, ci, va = _operator(rb, points, k)
    x = W.normal((N ** 3, k), 5)
    b = np.zeros((N ** 3, k), np.longdouble)
    for j in range(points):
        b += va[j::points, None].astype(np.longdouble) * x[ci[j::points]].astype(np.longdouble)
    b = b.astype(np.float64)
    prm = rb.cg_params(rtol=1e-30, max_iter=0)
    got = rb.cg_solve(A, to_dev(b), to_dev(x), params=prm).true_rel_res
    vec, parts = PARTS[points, k]
    A.set_schedule(k, vec, parts, 0, -1)
    want = rb.cg_solve(A, to_dev(b), to_dev(x), params=prm).true_rel_res
    assert all(0 < w < 3e-16 and abs(g - w) <= 1e-12 * w for g, w in zip(got, want)), (got, want)


@pytest.mark.parametrize("points,k", [(13, 1), (13, 3), (27, 1), (27, 3), (27, 8)])
@pytest.mark.parametrize("mixed", [0, 2])
def test_solves_take_the_same_parts(rb, points, k, mixed):
    A, *_ = _operator(rb, points, k)
    Ai = _operator(rb, points, k, "f32")[0] if mixed else None
    B = to_dev(W.zero_mean(W.normal((N ** 3, k), 6)))
    prm = rb.cg_params(rtol=1e-10, mixed=mixed, project_mean=True)
    X, Z = torch.zeros_like(B), torch.zeros_like(B)
    r = rb.cg_solve(A, B, X, A_inner=Ai, params=prm)
    vec, parts = PARTS[points, k]
    A.set_schedule(k, vec, parts, 0, -1)
    if mixed:
        Ai.set_schedule(k, *((4, 4) if k == 8 else (vec, parts)), 0, -1)
    s = rb.cg_solve(A, B, Z, A_inner=Ai, params=prm)
    assert r.status == s.status == rb.RB_OK and r.iters == s.iters
    assert torch.equal(X, Z)
