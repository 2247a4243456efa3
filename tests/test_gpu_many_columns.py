"""Solves of 51 to 63 columns: chunks of three columns, 17 to 21 of them, in blocks laid out for 32, where
the column sums' scratch holds 64 columns (GPU).  Bar: the true relative residual, recomputed on the CPU."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


def _system(k):
    g = W.channel_grid(12, 16, 8, gamma=1.5)
    A = (-fvm.laplacian(g)).tocsr()
    return g, A, W.zero_mean(W.normal((A.shape[0], k), 40 + k))


def _check(A, B, X, tol=1e-10):
    R = B - A @ X.cpu().numpy()
    R -= R.mean(axis=0, keepdims=True)
    assert np.all(np.linalg.norm(R, axis=0) <= tol * np.linalg.norm(B, axis=0))


@pytest.mark.parametrize("k", [48, 51, 54, 57, 60, 63])
@pytest.mark.parametrize("mixed", [False, True])
def test_multigrid(rb, k, mixed):
    g, A, B = _system(k)
    mg = rb.Multigrid(*rb.grid_nodes(g), k_max=k, smoother="jacobi")
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    for _ in range(2):
        X.zero_()
        res = mg.solve(to_dev(B), X, rb.mg_params(mixed=mixed))
        assert res.status == rb.RB_OK, res
        _check(A, B, X)


@pytest.mark.parametrize("k", [51, 54, 57, 63])
@pytest.mark.parametrize("mixed,persistent,free", [(0, False, False), (2, False, False), (2, True, False), (2, False, True)])
def test_cg(rb, k, mixed, persistent, free):
    g, A, B = _system(k)
    op = rb.Operator.from_scipy(A, k_max=k)
    inner = None
    if mixed:
        inner = (rb.Operator.stencil(*rb.grid_nodes(g), scale=-1.0, dtype="f32", k_max=k) if free
                 else rb.Operator.from_scipy(A, dtype="f32", k_max=k))
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    res = rb.cg_solve(op, to_dev(B), X, A_inner=inner,
                      params=rb.cg_params(mixed=mixed, persistent=persistent, project_mean=True))
    assert res.status == rb.RB_OK, res
    _check(A, B, X)


@pytest.mark.parametrize("ks", [(63,), (51, 3, 5)])
def test_batch(rb, ks):
    systems = [_system(k) for k in ks]
    ops = [rb.Operator.from_scipy(A, k_max=k) for (_, A, _), k in zip(systems, ks)]
    inner = [rb.Operator.from_scipy(A, dtype="f32", k_max=k) for (_, A, _), k in zip(systems, ks)]
    batch = rb.Batch(ops, inner, list(ks), rb.cg_params(mixed=2, project_mean=True))
    Bd = [to_dev(B) for _, _, B in systems]
    Xd = [torch.zeros_like(b) for b in Bd]
    assert all(r.status == rb.RB_OK for r in batch.solve(Bd, Xd))
    for (_, A, B), X in zip(systems, Xd):
        _check(A, B, X)
