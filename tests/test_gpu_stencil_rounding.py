"""Rounding of the FP64 matrix-free Laplacian against extended precision, on nodes whose widths and
distances are exact, for every vector width (GPU).

Bar: 1.28e-16 of the product's 2-norm on random values (the kernel's operations emulated on the CPU: at
most 1.24e-16 on these grids; rows of seven entries with the diagonal first at least 1.29e-16) and
0.98e-16 of |A| |x| on smooth ones (at most 0.69e-16; 0.84 to 0.99e-16)."""
import numpy as np
import pytest
import torch

import workloads as W
from tests.conftest import to_dev

pytestmark = pytest.mark.gpu


def _grid(shape, wall):
    axes = []
    for d, n in enumerate(shape):
        x = np.tanh(1.5 * (2.0 * np.arange(n + 1) / n - 1)) / np.tanh(1.5) if d == wall else (1.0 + 0.3 * d) * np.arange(n + 1) / n
        axes.append(W.Axis(np.round(x * 2.0 ** 24) / 2.0 ** 24, d != wall))
    return W.Grid(tuple(axes), "exact widths")


def _terms(g, x):
    """The product and sum |c_f| (|x_f| + |x_0|) in extended precision; x [z, y, x, k]."""
    L = np.longdouble
    w = [np.diff(a.nodes).astype(L) for a in g.axes]
    y = np.zeros(x.shape, L)
    bound = np.zeros(x.shape, L)
    for d in range(3):
        ax = 2 - d
        dist = 0.5 * (w[d] + np.roll(w[d], 1))  # below cell i
        area = L(1)
        for e in range(3):
            if e != d:
                area = area * w[e].reshape([-1 if 2 - e == q else 1 for q in range(4)])
        line = dist.reshape([-1 if ax == q else 1 for q in range(4)])
        c = np.broadcast_to(area / line, x.shape[:3] + (1,)).copy()  # coefficient of the face below each cell
        if not g.axes[d].periodic:
            c[tuple(0 if ax == q else slice(None) for q in range(4))] = 0
        lo, up = np.roll(x, 1, ax), np.roll(x, -1, ax)
        cu = np.roll(c, -1, ax)
        y += c * (lo - x) + cu * (up - x)
        bound += c * (abs(lo) + abs(x)) + cu * (abs(up) + abs(x))
    return y, bound


@pytest.mark.parametrize("shape,wall", [((95, 33, 47), 1), ((96, 64, 24), 1), ((48, 48, 32), -1), ((60, 52, 32), 2)])
@pytest.mark.parametrize("k", [1, 2, 3, 4])
@pytest.mark.parametrize("scale", [1.0, -0.7])
def test_rounding(rb, shape, wall, k, scale):
    g = _grid(shape, wall)
    nodes, per = rb.grid_nodes(g)
    op = rb.Operator.stencil(nodes, per, scale=scale, k_max=k)
    nx, ny, nz = shape
    i, j, m = np.arange(nx) + 0.5, np.arange(ny) + 0.5, np.arange(nz) + 0.5
    smooth = (1.0 + 0.5 * np.sin(2 * np.pi * i / nx)[None, None, :] * np.cos(2 * np.pi * j / ny)[None, :, None]
              + 0.1 * np.cos(2 * np.pi * m / nz)[:, None, None])[..., None] * np.arange(1, k + 1)
    rand = W.normal((nz, ny, nx, k), 7 + k)
    for x, bar in ((rand, 1.28e-16), (smooth, 0.98e-16)):
        y = op.spmm(to_dev(x.reshape(-1, k))).cpu().numpy().reshape(x.shape)
        ref, bound = _terms(g, x.astype(np.longdouble))
        ref, bound = np.longdouble(scale) * ref, abs(np.longdouble(scale)) * bound / 2
        den = ref if bar > 1e-16 else bound
        err = float(np.sqrt(((y - ref) ** 2).sum() / (den ** 2).sum()))
        assert err <= bar, (err, bar)
