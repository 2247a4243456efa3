"""Rounding of the SpMM's long rows: a row that one lane walks in the ring sums in as many parts as the
lanes that would split it, so its result equals theirs bit for bit (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import spmm
from tests.conftest import to_dev
from tests.test_gpu_spmm_long_rows import _matrix

pytestmark = pytest.mark.gpu


def _run(op, X, c=None):
    Y = torch.full((op.n_rows, X.shape[1]), float("nan"), dtype=X.dtype, device="cuda")
    op.spmm(X, Y, c=c)
    op.check()
    return Y.cpu().numpy()


def _x(n, k, dtype, seed):
    return to_dev(W.normal((n, k), seed).astype(np.float64 if dtype == "f64" else np.float32))


def _lanes(k, vec):
    kp = 1
    while kp < k // vec:
        kp *= 2
    return max(1, min(8, 32 // kp // 4))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("lens", [(16,), (27,), (39,), (20, 24), (25, 26, 27), (8, 31)])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 8])
def test_ring_sums_as_lanes_do(rb, dtype, lens, k):
    """Every width of the ring's long-row form against a split over eight or four lanes."""
    A = _matrix(1291, lens, 3 + k)
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    X = _x(A.shape[1], k, dtype, 70 + k)
    c = to_dev(W.normal(k, 12))
    for vec in (1, 2, 3, 4):
        if k % vec:
            continue
        op.set_schedule(k, vec, 1, 2, 0)
        ring = _run(op, X, c)
        op.set_schedule(k, vec, 4 if k > 4 or vec == 4 else 8, 0, -1)
        assert np.array_equal(ring, _run(op, X, c)), vec


@pytest.mark.parametrize("k", [1, 2, 3, 4, 8])
def test_rows_of_13_lose_nothing(rb, k):
    """FP32 rows of 13: the error against 64 bits is no larger than with the row split over lanes."""
    A = _matrix(5000, (13,), 5)
    op = rb.Operator.from_scipy(A, dtype="f32", k_max=k)
    X = _x(A.shape[1], k, "f32", 80 + k)
    ref = spmm.spmm(spmm.round_f32(A), X.cpu().numpy().astype(np.float64))
    for vec in (1, 2, 3, 4):
        if k % vec or _lanes(k, vec) < 4:
            continue
        op.set_schedule(k, vec, 1, 2, 0)
        ring = np.linalg.norm(_run(op, X) - ref)
        op.set_schedule(k, vec, _lanes(k, vec), 0, -1)
        assert ring <= np.linalg.norm(_run(op, X) - ref), vec
