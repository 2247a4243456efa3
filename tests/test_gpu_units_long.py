"""The persistent refinement on units beyond the small grids: systems that finish many iterations before
the batch's last one (their blocks go on with bare barriers, whose verdict must not mix with the
loop's own flag), and systems whose r, q and d exceed the blocks' shared memory (GPU).

Bar: the true relative residual ||b - A x|| <= 1e-10 ||b|| recomputed on the CPU; solves of the same
batch are equal bit for bit (fixed orders throughout)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


def _system(rb, shape, wall, k, seed, smooth=False):
    axes = [W.tanh_axis(n, 1.3) if d == wall else W.uniform_axis(n, 1.0 + 0.3 * d) for d, n in enumerate(shape)]
    g = W.Grid(tuple(axes), "x".join(map(str, shape)))
    A = (-fvm.laplacian(g)).tocsr()
    if smooth:  # a Fourier mode of the periodic axes: a handful of iterations
        x = np.cos(2 * np.pi * np.arange(shape[0]) / shape[0])
        X = np.tile(x, shape[1] * shape[2])[:, None] * np.arange(1, k + 1)[None, :]
        B = A @ X
    else:
        B = W.normal((A.shape[0], k), seed)
    B = W.zero_mean(B)
    nodes, per = rb.grid_nodes(g)
    op = rb.Operator.from_scipy(A, k_max=k)
    return A, B, op, rb.Operator.stencil(nodes, per, scale=-1.0, dtype="f32", k_max=k)


def _check(A, B, X):
    R = B - A @ X
    R -= R.mean(axis=0, keepdims=True)
    assert np.all(np.linalg.norm(R, axis=0) <= 1e-10 * np.linalg.norm(B, axis=0))


def test_systems_that_finish_early(rb):
    sys_ = [_system(rb, (16, 12, 10), -1, 3, 1, smooth=True), _system(rb, (7, 5, 4), 1, 1, 2),
            _system(rb, (48, 40, 36), 1, 2, 3), _system(rb, (10, 8, 8), -1, 8, 4, smooth=True)]
    batch = rb.Batch([s[2] for s in sys_], [s[3] for s in sys_], [s[1].shape[1] for s in sys_],
                     rb.cg_params(rtol=1e-10, mixed=2, project_mean=True))
    Bd = [to_dev(s[1]) for s in sys_]
    first = None
    for _ in range(10):
        Xd = [torch.zeros_like(b) for b in Bd]
        res = batch.solve(Bd, Xd)
        assert all(r.status == rb.RB_OK for r in res), res
        X = [x.cpu().numpy() for x in Xd]
        first = first or X
        assert all(np.array_equal(x, f) for x, f in zip(X, first))
    assert 3 * max(res[0].iters[:3]) < res[2].iters[0], res  # the smooth systems are done long before
    for (A, B, *_), x in zip(sys_, X):
        _check(A, B, x)


# floats per block of 152: r alone in shared memory in part (8.0 M), r and some of q (6.3 M), all of r
# and q, part of d (3.1 M); one cell and several per unit
@pytest.mark.parametrize("shape,wall,k", [((126, 130, 122), 1, 4), ((129, 128, 127), 2, 3), ((128, 96, 85), 0, 3)])
def test_vectors_beyond_shared_memory(rb, shape, wall, k):
    A, B, op, inner = _system(rb, shape, wall, k, 50 + k)
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    res = rb.cg_solve(op, to_dev(B), X, A_inner=inner, params=rb.cg_params(rtol=1e-10, mixed=2, project_mean=True))
    assert res.status == rb.RB_OK, res
    _check(A, B, X.cpu().numpy())
