"""A single system's persistent launch whose grid barrier gives up: with the library's own choice of the
launch the sweep is dropped and the solve goes on launch by launch, without spending one of the caller's
sweeps; asked for (persistent = 1), RB_ETIMEOUT.  The barrier waits for one block more than the launch has,
50 ms, in a library built for this test from the same sources; it runs in a process of its own (GPU)."""
import os
import subprocess
import sys

import pytest

from tests.conftest import ROOT

pytestmark = pytest.mark.gpu

PROGRAM = """
import sys
import numpy as np, torch
import paper_2508_06710_gb300 as rb
import workloads as W
from oracle import fvm
g = W.channel_grid(24, 16, 12, gamma=1.5)
A = (-fvm.laplacian(g)).tocsr()
B = W.zero_mean(W.normal((A.shape[0], 3), 7))
op = rb.Operator.from_scipy(A, k_max=3)
inner = rb.Operator.stencil(*rb.grid_nodes(g), scale=-1.0, dtype="f32", k_max=3)
def solve(sweeps, persistent=False):
    X = torch.zeros((A.shape[0], 3), dtype=torch.float64, device="cuda")
    prm = rb.cg_params(mixed=1, inner_rtol=1e-3, project_mean=True, max_sweeps=sweeps, persistent=persistent)
    res = rb.cg_solve(op, torch.as_tensor(B, device="cuda"), X, A_inner=inner, params=prm)
    R = B - A @ X.cpu().numpy()
    R -= R.mean(axis=0)
    return res, (np.linalg.norm(R, axis=0) / np.linalg.norm(B, axis=0)).max()
res, rel = solve(60)
assert res.status == rb.RB_OK and rel <= 1e-10, (res, rel)
sweeps = int(sys.argv[2]) if len(sys.argv) > 2 else res.sweeps
again, rel = solve(sweeps)  # no more sweeps than the solve takes
assert again.status == rb.RB_OK and rel <= 1e-10 and again.sweeps <= sweeps, (again, rel)
if sys.argv[1] == "expires":
    try:
        solve(60, persistent=True)
        raise SystemExit("no timeout")
    except rb.RbError as e:
        assert e.status == rb.RB_ETIMEOUT, e
    res, rel = solve(60)  # and the context is as good as before
    assert res.status == rb.RB_OK and rel <= 1e-10
print(sweeps)
"""


def _run(*args, lib=None):
    code = PROGRAM if lib is None else f"import paper_2508_06710_gb300 as rb\nrb.LIB_PATH = {lib!r}\n" + PROGRAM
    r = subprocess.run([sys.executable, "-c", code, *args], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.split()[-1]


def test_expired_barrier_falls_back(rb, tmp_path):
    from paper_2508_06710_gb300 import build

    objs = {s: os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()}
    if not all(os.path.exists(o) for o in objs.values()):
        build.build(force=True)
    src = os.path.join(build.CSRC, "cg.cu")
    objs[src] = str(tmp_path / "cg.o")
    subprocess.run([build.nvcc(), *build.flags(), "-DRB_SOLO_EXTRA_ARRIVALS=1", "-DRB_SOLO_TIMEOUT_NS=50000000ull", "-c",
                    src, "-o", objs[src]], check=True)
    lib = str(tmp_path / "librbspmm.so")
    subprocess.run([build.nvcc(), build.ARCH, "-shared", "-o", lib, *objs.values()], check=True)
    sweeps = _run("meets")
    _run("expires", sweeps, lib=lib)
