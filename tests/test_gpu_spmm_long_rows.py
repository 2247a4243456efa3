"""Rows of 12 to 40 entries, the 13- and 27-point operators' kind, in the pipelined kernel's long-row
form and under the default schedule: row lengths around the gather batches (8 and 13), a ragged last
tile, rows that do not fit a stage (read in place), every vector width, strided blocks, a column scale;
few rows (the general kernel) (GPU).  Bar as for every SpMM: componentwise 1e-12 (FP64) and 1e-5
(FP32) of |A| |X| |c|."""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

import workloads as W
from oracle import spmm
from tests.conftest import componentwise_ok, to_dev

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5}


def _matrix(n, lens, seed):
    """n x n, row i with lens[i % len(lens)] entries in consecutive columns from a seeded start."""
    g = np.random.default_rng(seed)
    ln = np.array([lens[i % len(lens)] for i in range(n)])
    rp = np.concatenate([[0], np.cumsum(ln)])
    start = g.integers(0, n - max(lens), n)
    ci = np.concatenate([np.arange(s, s + l) for s, l in zip(start, ln)])
    return sp.csr_matrix((g.standard_normal(rp[-1]), ci, rp), shape=(n, n))


def _check(op, A, X, dtype, ld_pad=0, c=None):
    n, k = X.shape
    npdt, tdt = (np.float64, torch.float64) if dtype == "f64" else (np.float32, torch.float32)
    Xb = torch.zeros((n, k + ld_pad), dtype=tdt, device="cuda")
    Xb[:, :k] = to_dev(X.astype(npdt))
    Y = torch.full((n, k + ld_pad), float("nan"), dtype=tdt, device="cuda")
    op.spmm(Xb[:, :k], Y[:, :k], c=None if c is None else to_dev(c))
    op.check()
    Aref = A if dtype == "f64" else spmm.round_f32(A)
    cref = c if c is None or dtype == "f64" else c.astype(np.float32).astype(np.float64)
    Xref = X.astype(npdt).astype(np.float64)
    ok, worst = componentwise_ok(Y[:, :k].cpu().numpy(), spmm.spmm(Aref, Xref, cref), spmm.abs_bound(Aref, Xref, cref),
                                 TOL[dtype])
    assert ok, worst
    assert ld_pad == 0 or bool(torch.isnan(Y[:, k:]).all())


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("lens", [(12,), (13,), (15, 16, 17), (25, 26, 27), (8, 40), (39,), (1, 24, 70)])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8])
def test_long_rows_pipelined(rb, dtype, lens, k):
    n = 1291  # not a multiple of any tile
    A = _matrix(n, lens, 5 + k)
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    for vec in (1, 2, 3, 4):
        if k % vec:
            continue
        op.set_schedule(k, vec, 1, 2, 0)
        _check(op, A, W.normal((n, k), 11), dtype, c=W.normal(k, 12) if vec == 1 else None)
        _check(op, A, W.normal((n, k), 13), dtype, ld_pad=4)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [500, 24500])
@pytest.mark.parametrize("length", [13, 27])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 8, 16, 40])
def test_long_rows_default_schedule(rb, dtype, n, length, k):
    A = _matrix(n, (length,), 21)
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    _check(op, A, W.normal((n, k), 31 + k), dtype)
    if k < 32:  # odd row starts: scalar widths
        _check(op, A, W.normal((n, k), 41 + k), dtype, ld_pad=1)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k", [4, 8, 12, 16, 32])
def test_short_rows_default_schedule(rb, dtype, k):
    A = _matrix(3001, (7, 6), 51)
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    _check(op, A, W.normal((3001, k), 61), dtype)
    _check(op, A, W.normal((3001, k), 62), dtype, ld_pad=1)
