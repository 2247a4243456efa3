"""The persistent refinement on units of consecutive floats (matrix-free inner operators): every
unit width (4, 2 or 1 floats, by n_x k), units of one cell and of several, walls along each axis,
blocks without units, and column counts that take the general path instead (GPU).

Bar: the true relative residual ||b - A x|| <= 1e-10 ||b|| recomputed on the CPU, and so, with the
dense eigenvalues of A, ||x - x_ref|| <= 1e-10 ||b|| / lambda_min (x_ref the pseudo-inverse
solution; a hundredth more for its own rounding)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


def _grid(nx, ny, nz, wall):
    axes = [W.tanh_axis(n, 1.3) if d == wall else W.uniform_axis(n, 1.0 + 0.3 * d) for d, n in enumerate((nx, ny, nz))]
    return W.Grid(tuple(axes), f"{nx}x{ny}x{nz}-{wall}")


def _check(A, B, X):
    R = B - A @ X
    R -= R.mean(axis=0, keepdims=True)
    nb = np.linalg.norm(B, axis=0)
    assert np.all(np.linalg.norm(R, axis=0) <= 1e-10 * nb)
    lam, Q = np.linalg.eigh(A.toarray())
    Xr = Q[:, 1:] @ ((Q[:, 1:].T @ B) / lam[1:, None])
    assert np.all(np.linalg.norm(X - Xr, axis=0) <= 1.01e-10 * nb / lam[1])


# (n_x, n_y, n_z, wall axis or -1, k): widths 1, 2, 4 for k = 1, 3; 2, 4 for k = 2; one cell per unit
CASES = [(7, 5, 4, 1, 1), (6, 5, 4, 2, 1), (8, 5, 3, -1, 1), (5, 6, 7, 0, 2), (6, 3, 5, 1, 2), (8, 4, 3, 0, 2),
         (5, 4, 6, 2, 3), (7, 9, 5, 0, 3), (6, 7, 5, 1, 3), (8, 6, 5, 2, 3), (4, 3, 3, 0, 3), (12, 8, 7, -1, 3),
         (3, 4, 5, 1, 4), (9, 5, 6, 0, 4), (5, 4, 3, 2, 8), (6, 5, 4, -1, 16), (7, 4, 5, 1, 32), (2, 5, 4, 0, 3),
         (2, 4, 3, 0, 4), (6, 5, 4, 1, 5), (6, 5, 4, 2, 6), (4, 5, 3, 1, 12)]


@pytest.mark.parametrize("nx,ny,nz,wall,k", CASES)
@pytest.mark.parametrize("precond", [True, False])
def test_matrix_free_refinement(rb, nx, ny, nz, wall, k, precond):
    g = _grid(nx, ny, nz, wall)
    A = (-fvm.laplacian(g)).tocsr()
    B = W.zero_mean(W.normal((A.shape[0], k), 100 + nx + k))
    nodes, per = rb.grid_nodes(g)
    op = rb.Operator.from_scipy(A, k_max=k)
    inner = rb.Operator.stencil(nodes, per, scale=-1.0, dtype="f32", k_max=k)
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    prm = rb.cg_params(rtol=1e-10, mixed=2, project_mean=True, precond=precond)
    res = rb.cg_solve(op, to_dev(B), X, A_inner=inner, params=prm)
    assert res.status == rb.RB_OK, res
    _check(A, B, X.cpu().numpy())


def test_batch_of_unit_systems_and_its_timeout(rb):
    """Uneven systems of different unit kinds in one launch; a barrier that waits for one block more
    than the launch has gives up after 50 ms, and the next solve works."""
    systems = [(_grid(7, 5, 4, 1), 1), (_grid(8, 6, 5, 2), 3), (_grid(5, 6, 7, 0), 2), (_grid(5, 4, 3, -1), 8)]
    ops, inner, As, Bs = [], [], [], []
    for i, (g, k) in enumerate(systems):
        As.append((-fvm.laplacian(g)).tocsr())
        Bs.append(W.zero_mean(W.normal((As[-1].shape[0], k), 300 + i)))
        nodes, per = rb.grid_nodes(g)
        ops.append(rb.Operator.from_scipy(As[-1], k_max=k))
        inner.append(rb.Operator.stencil(nodes, per, scale=-1.0, dtype="f32", k_max=k))
    batch = rb.Batch(ops, inner, [k for _, k in systems], rb.cg_params(rtol=1e-10, mixed=2, project_mean=True))
    Bd = [to_dev(b) for b in Bs]
    Xd = [torch.zeros_like(b) for b in Bd]
    batch.set_barrier(timeout_ms=50.0, extra_arrivals=1)
    assert batch.solve(Bd, Xd)[0].status == rb.RB_ETIMEOUT
    batch.set_barrier(timeout_ms=2000.0, extra_arrivals=0)
    for x in Xd:
        x.zero_()
    res = batch.solve(Bd, Xd)
    assert all(r.status == rb.RB_OK for r in res), res
    for A, B, X in zip(As, Bs, Xd):
        _check(A, B, X.cpu().numpy())
