"""Short FP32 rows of a matrix beyond L2 in the ring by default: the channel's gradient (rows of two) and
Laplacian (many columns), equal bit for bit to the direct kernel's one sum per row (GPU)."""
import pytest
import torch

import paper_2508_06710_gb300 as pkg
import workloads as W
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,k", [(pkg.RB_FVM_GRADIENT, 3), (pkg.RB_FVM_GRADIENT, 1), (pkg.RB_FVM_LAPLACIAN, 16),
                                    (pkg.RB_FVM_LAPLACIAN, 12)])
def test_default_is_the_ring_and_sums_as_direct(rb, kind, k):
    g = W.channel_grid(192, 128, 96, gamma=1.5)
    op = rb.Operator(*rb.fvm_assemble(*rb.grid_nodes(g), kind), dtype="f32", k_max=k)
    X = to_dev(W.normal((op.n_cols, k), 3).astype("float32"))
    Y, Z = (torch.full((op.n_rows, k), float("nan"), device="cuda") for _ in range(2))
    s = op.schedule(X, Y)
    assert s["stage"] == 2
    op.spmm(X, Y)
    op.check()
    op.set_schedule(k, s["vec"], 1, 0, -1)
    op.spmm(X, Z)
    assert torch.equal(Y, Z)
