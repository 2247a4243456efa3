"""Tiles of the pipelined SpMM kernel's long-row form.  A tile's row pointers are one bulk copy, whose
source must be 16-byte aligned, so every tile has a multiple of four rows: the rule on the CPU, for
every element size and chunk count, and the kernel at the widest chunk count (32), where rows of
several hundred entries leave the fewest rows a tile (GPU).

Bar: (len + 2) unit roundoffs of |A| |X| componentwise, the worst case of a sum in any order."""
import os
import subprocess

import numpy as np
import pytest
import torch

import workloads as W
from oracle import spmm
from tests.conftest import ROOT, componentwise_ok, to_dev
from tests.test_gpu_spmm_long_rows import _matrix

PROGRAM = """
#include <cstdio>
#include "spmm_tma.cuh"
int main() {
  for (int eb : {4, 8})
    for (int kp = 1; kp <= 32; kp *= 2)
      for (double len = 12; len < 20000; len *= 1.05) {
        const int c = rb::tma_long_threads(len, eb, kp);
        std::printf("%d %d %.0f %d\\n", eb, kp, len, c);
      }
}
"""


def test_tiles_hold_a_multiple_of_four_rows(tmp_path):
    from paper_2508_06710_gb300 import build

    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I" + build.CSRC, "-I" + os.path.join(ROOT, "include"), "-o", str(exe),
                    str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    plans = [tuple(int(v) for v in line.split()) for line in out if line]
    assert len(plans) > 1000
    bad = [p for p in plans if p[3] % 32 or p[3] % p[1] or p[3] // p[1] % 4]
    assert not bad, bad[:5]
    assert min(p[3] for p in plans) == 64  # long rows still take fewer threads


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,length", [("f64", 700), ("f64", 740), ("f64", 3000), ("f32", 1100), ("f32", 5000)])
@pytest.mark.parametrize("k,vec", [(32, 1), (64, 2), (16, 1)])
def test_longest_rows_at_many_chunks(rb, dtype, length, k, vec):
    n = max(203, length + 3)
    A = _matrix(n, (length,), 7)[:203]
    A.sort_indices()
    op = rb.Operator.from_scipy(A, dtype=dtype, k_max=k)
    op.set_schedule(k, vec, 1, 2, 0)
    npdt = np.float64 if dtype == "f64" else np.float32
    X = W.normal((n, k), 9).astype(npdt)
    Y = torch.full((203, k), float("nan"), dtype=torch.float64 if dtype == "f64" else torch.float32, device="cuda")
    op.spmm(to_dev(X), Y)
    op.check()
    Aref = A if dtype == "f64" else spmm.round_f32(A)
    X = X.astype(np.float64)
    ok, worst = componentwise_ok(Y.cpu().numpy(), spmm.spmm(Aref, X), spmm.abs_bound(Aref, X),
                                 (length + 2) * (2.0 ** -53 if dtype == "f64" else 2.0 ** -24))
    assert ok, worst
