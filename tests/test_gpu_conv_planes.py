"""Level-0 convolutions on 128-cell rows that march z planes: rows per CTA that do not divide ny, runs
of several planes that do not divide nz, walls and wrapped planes in z, one or two input groups and
8 or 16 output columns per plane, against the FP64 oracle with BF16 rounding at the same points.

Bounds: those of the other convolution kernels (a BF16 rounding flip, 2^-8 of a value, on a few of
the activations of a layer): 2e-2 on the output's and 5e-2 on the gradients' 2-norms."""
import numpy as np
import pytest
import torch

from oracle import unet as U
from tests.conftest import to_dev
from tests.test_gpu_guess import _rel, _setup

pytestmark = pytest.mark.gpu

CASES = [((128, 2, 2), (8, 16), (1, 1, 1)), ((128, 6, 4), (8, 16), (0, 0, 0)), ((128, 10, 6), (16, 24), (1, 0, 1)),
         ((128, 6, 2), (16, 8), (0, 1, 0)),
         ((128, 66, 42), (8, 8), (1, 1, 0))]


@pytest.mark.parametrize("shape,channels,periodic", CASES)
def test_planes_against_oracle(rb, shape, channels, periodic):
    g, spec, pref, _, (b, p1, p2, t), zyx = _setup(rb, shape, channels, 2100, periodic)
    out = g.predict(to_dev(b), to_dev(p1), to_dev(p2)).cpu().numpy()
    ref = U.predict(spec, pref, b, p1, p2, zyx, bf=True)
    assert np.linalg.norm(out - ref) < 2e-2 * np.linalg.norm(ref - (p1 - p1.mean()))
    if np.prod(shape) > 100000:  # runs of several planes: the oracle's forward pass alone takes its time
        return
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    g.loss_grad(to_dev(b), to_dev(p1), to_dev(p2), to_dev(t), accumulate=False, loss=loss)
    _, gref = U.loss_and_grad(spec, pref, b, p1, p2, t, zyx, bf=True)
    gg = U.from_flat(spec, g.grad().cpu().numpy().astype(np.float64))
    for name, *_ in U.layers(spec):
        for part in ("W", "b"):
            key = f"{name}.{part}"
            if key != "head.b":  # sum of a zero-mean output gradient: zero up to rounding
                assert _rel(gg[key], gref[key]) < 5e-2, key
