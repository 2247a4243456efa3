"""Batches with matrix-free inner operators on both sides of the size from which the vectors stream (20 M
floats a vector in all), to the true relative residual 1e-10, recomputed on the CPU; equal bits from one
solve to the next (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("systems", [[((96, 96, 96), 12)] * 2, [((96, 96, 96), 8), ((40, 30, 20), 3)]])
def test_large_batches(rb, systems):
    ops, inner, As, Bs = [], [], [], []
    for i, (shape, k) in enumerate(systems):
        g = W.Grid(tuple(W.uniform_axis(n, 1.0 + 0.1 * d) for d, n in enumerate(shape)), "box")
        As.append((-fvm.laplacian(g)).tocsr())
        Bs.append(W.zero_mean(W.normal((As[-1].shape[0], k), 60 + i)))
        ops.append(rb.Operator.from_scipy(As[-1], k_max=k))
        inner.append(rb.Operator.stencil(*rb.grid_nodes(g), scale=-1.0, dtype="f32", k_max=k))
    batch = rb.Batch(ops, inner, [k for _, k in systems], rb.cg_params(rtol=1e-10, mixed=2, project_mean=True))
    Bd = [to_dev(b) for b in Bs]
    first = None
    for _ in range(2):
        Xd = [torch.zeros_like(b) for b in Bd]
        assert all(r.status == rb.RB_OK for r in batch.solve(Bd, Xd))
        first = first or Xd
        assert all(torch.equal(x, f) for x, f in zip(Xd, first))
    for A, B, X in zip(As, Bs, Xd):
        R = B - A @ X.cpu().numpy()
        assert np.all(np.linalg.norm(R - R.mean(axis=0), axis=0) <= 1e-10 * np.linalg.norm(B, axis=0))
