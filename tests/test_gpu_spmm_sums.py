"""Rounding of the SpMM's long rows: a row that one lane walks, in the ring or direct, sums in as many
parts as the lanes that would split it, so its result equals theirs bit for bit; rows of uneven length
and hinted row blocks are split over lanes (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import spmm
from tests.conftest import to_dev
from tests.test_gpu_spmm_long_rows import _matrix

pytestmark = pytest.mark.gpu

N = 24500  # above the row count from which one lane takes a row
FEW = 3000


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
        op.set_schedule(k, vec, 4 if k > 4 or (vec == 4 and dtype == "f64") else 8, 0, -1)
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


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("lens", [(12,), (13,), (15, 16), (27,), (36, 39)])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 8, 9, 12, 16])
def test_default_schedule_sums_as_lanes_do(rb, dtype, lens, k):
    A = _matrix(N, lens, 21)
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    X = _x(N, k, dtype, 90 + k)
    s = op.schedule(X, torch.empty_like(X))
    few = rb.Operator.from_scipy(A[:FEW], dtype=dtype, k_max=k)
    wide = few.schedule(X, torch.empty((FEW, k), dtype=X.dtype, device="cuda"))
    long = np.mean(lens) >= 16
    parts = s["lpr"] if s["stage"] == 0 else (8 if long and k <= 4 else 4)
    assert parts >= (wide["lpr"] if long else min(4, wide["lpr"])), (s, wide)
    if s["stage"] == 2 and dtype == "f32" and s["vec"] <= 2 and 13 <= np.mean(lens) < 16:
        return  # the batch of 13: test_rows_of_13_lose_nothing
    got = _run(op, X)[:FEW]
    while parts * (s_kp := 8 // _lanes(k, s["vec"])) > 32:
        parts //= 2
    few.set_schedule(k, s["vec"], parts, 0, -1)
    assert np.array_equal(got, _run(few, X)), (s, parts)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8, 9, 16])
def test_uneven_rows_and_row_blocks_keep_the_lanes(rb, dtype, k):
    A = _matrix(N, (12, 12, 12, 60), 31)  # average 24, maximum 60
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    few = rb.Operator.from_scipy(A[:FEW], dtype=dtype, k_max=k)
    X = _x(N, k, dtype, 95 + k)
    s = op.schedule(X, torch.empty_like(X))
    assert s == few.schedule(X, torch.empty((FEW, k), dtype=X.dtype, device="cuda"))
    assert (s["lpr"], s["stage"], s["grid_cap"]) == (_lanes(k, s["vec"]), 0, 0 if s["lpr"] == 1 and dtype == "f64" else -1)
    assert np.array_equal(_run(op, X)[:FEW], _run(few, X))
    even = rb.Operator.from_scipy(_matrix(N, (27,), 32), dtype=dtype, k_max=k)
    even.set_row_blocks([0, 8000, 16000])
    h = even.schedule(X, torch.empty_like(X))
    assert (h["lpr"], h["stage"]) == (_lanes(k, h["vec"]), 0)
