"""The recorded refinement sweep of the multigrid solve: one graph serves every tolerance and iteration
limit of a k, several k alternate on one hierarchy, and more k than a hierarchy keeps graphs for come
and go (GPU).  Bar: the true relative residual, recomputed on the CPU."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import fvm
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def system(rb):
    g = W.channel_grid(16, 16, 16, gamma=1.5)
    return g, (-fvm.laplacian(g)).tocsr()


def _solve(rb, mg, A, k, seed, **kw):
    B = W.zero_mean(W.normal((A.shape[0], k), seed))
    X = torch.zeros((A.shape[0], k), dtype=torch.float64, device="cuda")
    res = mg.solve(to_dev(B), X, rb.mg_params(mixed=True, **kw))
    R = B - A @ X.cpu().numpy()
    R -= R.mean(axis=0, keepdims=True)
    return res, np.linalg.norm(R, axis=0) / np.linalg.norm(B, axis=0)


def test_one_recording_for_every_tolerance(rb, system):
    """After the first solve's recording no sweep is read but once, whatever the tolerances."""
    g, A = system
    nodes, per = rb.grid_nodes(g)
    mg = rb.Multigrid(nodes, per, k_max=3)
    _solve(rb, mg, A, 3, 1, rtol=1e-10, inner_rtol=1e-2)
    for i, (rtol, inner) in enumerate([(1e-10, 1e-2), (1e-10, 3e-3), (1e-8, 1e-1), (1e-11, 1e-4)]):
        res, rel = _solve(rb, mg, A, 3, 2 + i, rtol=rtol, inner_rtol=inner)
        assert res.status == rb.RB_OK and np.all(rel <= rtol), (res, rel)
        fresh, _ = _solve(rb, rb.Multigrid(nodes, per, k_max=3), A, 3, 2 + i, rtol=rtol, inner_rtol=inner)
        assert (res.sweeps, res.iters) == (fresh.sweeps, fresh.iters)  # each tolerance acts
        assert res.host_syncs == res.sweeps + 2, res  # the residuals' reads and the report's


@pytest.mark.parametrize("limit", [0, 1, 3, 7])
def test_iteration_limit(rb, system, limit):
    g, A = system
    mg = rb.Multigrid(*rb.grid_nodes(g), k_max=2)
    for _ in range(2):  # recorded during the first solve
        assert _solve(rb, mg, A, 2, 9, rtol=1e-10, inner_rtol=1e-2)[0].status == rb.RB_OK
    res, rel = _solve(rb, mg, A, 2, 9, rtol=1e-10, inner_rtol=1e-2, max_iter=limit)
    assert res.status == rb.RB_ENOCONV and max(res.iters) == limit, res
    assert np.all(rel <= 1.0 + 1e-12) and (limit == 0 or np.all(rel < 0.9))


def test_more_shapes_than_graphs(rb, system):
    g, A = system
    mg = rb.Multigrid(*rb.grid_nodes(g), k_max=64)
    ks = [k for k in range(1, 65) if k <= 8 or k % 2 == 0]
    for k in ks + ks[:6] + [1, 3, 1, 3]:
        res, rel = _solve(rb, mg, A, k, 20 + k, rtol=1e-9)
        assert res.status == rb.RB_OK and np.all(rel <= 1e-9), (k, res)
