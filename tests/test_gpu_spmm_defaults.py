"""The untuned schedule where a wider or pipelined choice does not pay: FP32 rows of seven at 20 and
above 32 columns stay direct, FP64 rows of two at 32 columns keep two doubles a thread, FP64 rows of 27 in
few rows are split over lanes or take the ring (GPU; results have their own tests)."""
import pytest
import torch

import paper_2508_06710_gb300 as pkg
import workloads as W

pytestmark = pytest.mark.gpu


def _schedule(rb, csr, dtype, k):
    op = rb.Operator(*csr, dtype=dtype, k_max=k)
    td = torch.float64 if dtype == "f64" else torch.float32
    X, Y = (torch.empty((n, k), dtype=td, device="cuda") for n in (op.n_cols, op.n_rows))
    return op.schedule(X, Y)


@pytest.fixture(scope="module")
def channel(rb):
    g = W.channel_grid(192, 128, 96, gamma=1.5)
    return {kind: rb.fvm_assemble(*rb.grid_nodes(g), kind) for kind in (pkg.RB_FVM_LAPLACIAN, pkg.RB_FVM_GRADIENT)}


@pytest.mark.parametrize("k,stage", [(8, 0), (12, 2), (16, 2), (20, 0), (24, 2), (32, 2), (36, 0), (48, 0), (64, 0)])
def test_short_rows_of_many_columns(rb, channel, k, stage):
    s = _schedule(rb, channel[pkg.RB_FVM_LAPLACIAN], "f32", k)
    assert (s["vec"], s["stage"]) == (4, stage)


@pytest.mark.parametrize("k,vec", [(8, 4), (16, 4), (32, 2)])
def test_rows_of_two_in_doubles(rb, channel, k, vec):
    assert _schedule(rb, channel[pkg.RB_FVM_GRADIENT], "f64", k)["vec"] == vec


@pytest.mark.parametrize("n,k,want", [(30, 3, (3, 1, 2, 0)), (30, 4, (2, 4, 0, -1)), (34, 6, (3, 4, 0, -1)),
                                      (48, 3, (3, 8, 0, -1)), (40, 4, (2, 4, 0, 0)), (30, 8, (2, 2, 0, 0))])
def test_few_rows_of_27(rb, n, k, want):
    s = _schedule(rb, rb.stencil_assemble((n, n, n), [1.0 / n] * 3, rb.RB_STENCIL_27P), "f64", k)
    assert (s["vec"], s["lpr"], s["stage"], s["grid_cap"]) == want
