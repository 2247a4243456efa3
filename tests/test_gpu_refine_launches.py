"""Which launch a refinement sweep with the matrix-free inner operator takes by default: one for all its
iterations (a host read a sweep and residual), or two kernels an iteration with host checks on small long
grids at two and three columns; both reach the tolerance (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,k,one", [((128, 8, 8), 1, True), ((128, 8, 8), 2, False), ((8, 128, 8), 3, False),
                                         ((128, 8, 8), 4, True), ((64, 16, 16), 3, True), ((160, 16, 16), 3, True),
                                         ((128, 20, 15), 2, False)])
def test_default_launch(rb, shape, k, one):
    g = W.Grid(tuple(W.uniform_axis(n) for n in shape), "box")
    A = (-fvm.laplacian(g)).tocsr()
    B = W.zero_mean(W.normal((A.shape[0], k), 3))
    op = rb.Operator.from_scipy(A, k_max=k)
    inner = rb.Operator.stencil(*rb.grid_nodes(g), scale=-1.0, dtype="f32", k_max=k)
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    res = rb.cg_solve(op, to_dev(B), X, A_inner=inner, params=rb.cg_params(mixed=2, project_mean=True))
    assert res.status == rb.RB_OK, res
    assert (res.host_syncs <= 2 * res.sweeps + 2) == one, res
    R = B - A @ X.cpu().numpy()
    assert np.all(np.linalg.norm(R - R.mean(axis=0), axis=0) <= 1e-10 * np.linalg.norm(B, axis=0))
