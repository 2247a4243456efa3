"""The FP32 cycle's restriction by rows: line lengths of 4- and 2-float units, one and several rows
per block, walls along each axis (longer 1-D maps next to them), rows that do not fit the kernel's
shared memory (the general kernel), against the oracle's cycle (GPU).  Bar as for every FP32 cycle:
1e-4 relative, means removed."""
import numpy as np
import pytest

import workloads as W
from oracle import mg
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,wall,k", [((8, 8, 8), -1, 1), ((10, 8, 12), 0, 1), ((10, 12, 8), 1, 3), ((18, 8, 10), 2, 2),
                                          ((12, 10, 8), 0, 5), ((8, 16, 10), 1, 8), ((40, 8, 8), -1, 4),
                                          ((208, 8, 8), 1, 64)])
def test_vcycle_row_restriction(rb, shape, wall, k):
    axes = [W.tanh_axis(n, 1.3) if d == wall else W.uniform_axis(n, 1.0 + 0.2 * d) for d, n in enumerate(shape)]
    g = W.Grid(tuple(axes), "rows")
    nodes, per = rb.grid_nodes(g)
    m = rb.Multigrid(nodes, per, k_max=k, smoother="jacobi")
    lv = mg.hierarchy(g, smoother="jacobi")
    R = W.zero_mean(W.normal((lv[0].A.shape[0], k), 900 + k))
    Z = m.vcycle(to_dev(R), dtype="f32").cpu().numpy()
    for j in sorted({0, k // 2, k - 1}):
        zr = mg.vcycle(lv, R[:, j], level=0)
        zr -= zr.mean()
        z = Z[:, j] - Z[:, j].mean()
        assert np.linalg.norm(z - zr) <= 1e-4 * np.linalg.norm(zr), (j, np.linalg.norm(z - zr) / np.linalg.norm(zr))
