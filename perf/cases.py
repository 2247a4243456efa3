"""Timed cases of the library's main path: the discrete operators applied to k columns (SpMM),
the Poisson solves built on them, the projection step and the learned initial guess, each
through the public Python entry points as a user's program calls them.

A case is a dict of plain values; `prepare` makes the inputs (on the GPU, from the seed alone)
and the handles a program keeps, `run` is one pass, `exact` the same outputs in 64 bits from
plain torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2508_06710_gb300 as rb
from paper_2508_06710_gb300.flow_step import ProjectionStep

DEV = "cuda"
F64 = torch.float64


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # the 32^3 correctness grid with one column: a call whose launch counts most
        dict(name="spmm-f64-small", kind="spmm", op="laplacian", fmt="csr", grid="box", nx=32, ny=32, nz=32,
             dtype="f64", k=1),
        # the channel's Laplacian on the three velocity components (diffusion; the outer residual)
        dict(name="spmm-f64-laplacian", kind="spmm", op="laplacian", fmt="csr", grid="channel", nx=192, ny=128, nz=96,
             dtype="f64", k=3),
        # the channel's gradient in FP32: two entries per row, rows of three blocks of faces
        dict(name="spmm-f32-gradient", kind="spmm", op="gradient", fmt="csr", grid="channel", nx=192, ny=128, nz=96,
             dtype="f32", k=3),
        # the densest pattern (27 entries per row) on eight states, FP32
        dict(name="spmm-f32-27p", kind="spmm", op="27p", fmt="csr", grid="box", nx=160, ny=160, nz=160, dtype="f32",
             k=8),
        # an extruded unstructured mesh: 149k vertices, 64 periodic planes as the columns
        dict(name="spmm-f64-extruded", kind="extruded", side=386, dtype="f64", k=64),
        # the matrix-free Laplacian in FP64 on a channel of ragged sizes
        dict(name="free-f64-laplacian", kind="spmm", op="laplacian", fmt="free", grid="channel", nx=190, ny=127, nz=95,
             dtype="f64", k=3),
        # the pressure solve of the channel by multigrid CG (FP32 cycle inside FP64 refinement)
        dict(name="mg-channel", kind="mg", grid="channel", nx=192, ny=128, nz=96, k=3, mixed=True),
        # the same solve by Jacobi CG: FP32 inner iterations on the matrix-free Laplacian
        dict(name="cg-channel", kind="cg", grid="channel", nx=192, ny=128, nz=96, k=3),
        # uneven systems in one persistent launch: a coarse and a fine box, three channels
        dict(name="batch-uneven", kind="batch", coarse=64, fine=128, nx=96, ny=64, nz=48, channels=3),
        # one Heun RK3 projection step of two stacked flow states, multigrid pressure solves
        dict(name="projection-step", kind="projection", nx=128, ny=128, nz=128, m=2),
        # the learned guess on the Rayleigh-Benard box: one forward pass
        dict(name="guess-predict", kind="predict", nx=128, ny=128, nz=128),
        # and one sample of its training: loss and every parameter's gradient
        dict(name="guess-train", kind="train", nx=128, ny=128, nz=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "spmm", "free", "extruded", "mg", "mg", "cg", "projection", "predict", "train"])
    if kind in ("spmm", "free"):
        op = rng.choice(["laplacian", "laplacian", "gradient", "divergence", "13p", "27p"]) if kind == "spmm" else "laplacian"
        dense = op in ("13p", "27p")
        nx, ny, nz = (_log_int(rng, 24, 150 if dense else 190) for _ in range(3))
        dtype = rng.choice(["f64", "f64", "f32", "f32", "df64"]) if not dense else rng.choice(["f64", "f32"])
        k = rng.choice([1, 2, 3, 4, 5, 6, 8, 12, 16]) if not dense else rng.choice([1, 2, 3, 4, 8])
        while nx * ny * nz * k > 3e7:
            k = (k + 1) // 2
        return dict(kind="spmm", op=op, fmt="csr" if kind == "spmm" else "free",
                    grid="box" if dense else rng.choice(["box", "channel", "channel", "rbc"]), nx=nx, ny=ny, nz=nz,
                    dtype=dtype, k=k)
    if kind == "extruded":
        return dict(kind="extruded", side=_log_int(rng, 90, 386), dtype=rng.choice(["f64", "f32"]),
                    k=rng.choice([16, 24, 32, 48, 64]))
    if kind in ("mg", "cg"):
        # multiples of 16 where the hierarchy halves the counts; the sizes differ by axis
        nx, ny, nz = (16 * _log_int(rng, 2, 12) if kind == "mg" else _log_int(rng, 30, 130) for _ in range(3))
        c = dict(kind=kind, grid=rng.choice(["box", "channel", "rbc"]), nx=nx, ny=ny, nz=nz, k=rng.choice([1, 2, 3, 4, 8]))
        while nx * ny * nz * c["k"] > 7e6:
            c["k"] = (c["k"] + 1) // 2
            if c["k"] == 1:
                break
        if kind == "mg":
            c["mixed"] = rng.random() < 0.7
        return c
    if kind == "projection":
        nx, ny, nz = (16 * _log_int(rng, 2, 8) for _ in range(3))
        return dict(kind="projection", nx=nx, ny=ny, nz=nz, m=rng.choice([1, 2, 3]))
    nx, ny, nz = (16 * rng.randint(2, 8) for _ in range(3))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz)


# ----------------------------------------------------------------------------- grids
def _tanh(n, gamma, lo, hi):
    s = np.tanh(gamma * (2.0 * np.arange(n + 1) / n - 1.0)) / np.tanh(gamma)
    s[0], s[-1] = -1.0, 1.0
    return lo + (hi - lo) * 0.5 * (s + 1.0)


def _axes(grid, nx, ny, nz):
    """Node coordinates (x, y, z) and periodic flags: the unit periodic box, the channel (walls
    in y), the Rayleigh-Benard box (walls in z)."""
    if grid == "channel":
        return [np.linspace(0, 2 * math.pi, nx + 1), _tanh(ny, 1.5, -1.0, 1.0), np.linspace(0, math.pi, nz + 1)], (True, False, True)
    if grid == "rbc":
        return [np.linspace(0, 1, nx + 1), np.linspace(0, 1, ny + 1), _tanh(nz, 1.4, 0.0, 1.0)], (True, True, False)
    if grid == "tau":
        return [np.linspace(0, 2 * math.pi, n + 1) for n in (nx, ny, nz)], (True, True, True)
    return [np.linspace(0, 1, n + 1) for n in (nx, ny, nz)], (True, True, True)


def _nodes(grid, nx, ny, nz):
    axes, per = _axes(grid, nx, ny, nz)
    return [torch.as_tensor(a, dtype=F64, device=DEV) for a in axes], per


def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * salt + int(seed))


def _normal(shape, seed, salt=0, dtype=F64):
    return torch.randn(shape, generator=_gen(seed, salt), dtype=dtype, device=DEV)


def _smooth(k, nx, ny, nz, seed, salt=0):
    """k smooth random fields [k, nz, ny, nx] of zero mean and unit rms (a spectrum that falls
    off over a few grid-spanning modes, as a flow's pressure and divergence do)."""
    f = torch.fft.rfftn(_normal((k, nz, ny, nx), seed, salt), dim=(1, 2, 3))
    kz = torch.fft.fftfreq(nz, 1.0 / nz, dtype=F64, device=DEV)[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, dtype=F64, device=DEV)[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, dtype=F64, device=DEV)[None, None, :]
    f *= (1.0 + (kx * kx + ky * ky + kz * kz) / 9.0) ** -1.5
    f[:, 0, 0, 0] = 0
    v = torch.fft.irfftn(f, s=(nz, ny, nx), dim=(1, 2, 3))
    return v / v.square().mean(dim=(1, 2, 3), keepdim=True).sqrt()


def _volume(grid, nx, ny, nz):
    axes, _ = _axes(grid, nx, ny, nz)
    w = [torch.as_tensor(np.diff(a), dtype=F64, device=DEV) for a in axes]
    return w[2][:, None, None] * w[1][None, :, None] * w[0][None, None, :]


def _columns(f):
    """[k, nz, ny, nx] -> the library's interleaved (n, k) block."""
    x = f.reshape(f.shape[0], -1)
    return torch.empty((x.shape[1], x.shape[0]), dtype=x.dtype, device=x.device).copy_(x.t())


def _rhs(grid, nx, ny, nz, k, seed, salt=0):
    """Right-hand sides of the pressure equation: volume-integrated smooth sources, zero sum."""
    b = _columns(_smooth(k, nx, ny, nz, seed, salt) * _volume(grid, nx, ny, nz))
    return b - b.mean(dim=0, keepdim=True)


# ----------------------------------------------------------------------------- SpMM
def _n_faces(grid, nx, ny, nz):
    n = (nx, ny, nz)
    per = _axes(grid, 2, 2, 2)[1]
    return sum(nx * ny * nz if per[d] else nx * ny * nz // n[d] * (n[d] - 1) for d in range(3))


def _spmm_sizes(c):
    """rows, columns, stored entries of the case's operator."""
    n = c["nx"] * c["ny"] * c["nz"]
    nf = _n_faces(c["grid"], c["nx"], c["ny"], c["nz"])
    return {"laplacian": (n, n, n + 2 * nf), "gradient": (nf, n, 2 * nf), "divergence": (n, nf, 2 * nf),
            "13p": (n, n, 13 * n), "27p": (n, n, 27 * n)}[c["op"]]


def _spmm_x(c, seed):
    x = _normal((_spmm_sizes(c)[1], c["k"]), seed)
    return x.float() if c["dtype"] == "f32" else x


def _prepare_spmm(c, seed):
    nodes, per = _nodes(c["grid"], c["nx"], c["ny"], c["nz"])
    k, dt = c["k"], c["dtype"]
    if c["fmt"] == "free":
        A = rb.Operator.stencil(nodes, per, dtype=dt, k_max=k)
    else:
        if c["op"] in ("13p", "27p"):
            h = [1.0 / c["nx"]] * 3 if c["op"] == "27p" else [1.0 / c["nx"], 1.0 / c["ny"], 1.0 / c["nz"]]
            csr = rb.stencil_assemble((c["nx"], c["ny"], c["nz"]), h,
                                      rb.RB_STENCIL_27P if c["op"] == "27p" else rb.RB_STENCIL_13P)
        else:
            csr = rb.fvm_assemble(nodes, per, {"laplacian": rb.RB_FVM_LAPLACIAN, "gradient": rb.RB_FVM_GRADIENT,
                                               "divergence": rb.RB_FVM_DIVERGENCE}[c["op"]])
        A = rb.Operator(*csr, dtype=dt, k_max=k)
    x = _spmm_x(c, seed)
    if dt == "df64":
        x = rb.df_split(x)
    return {"A": A, "X": x, "Y": torch.empty((A.n_rows,) + tuple(x.shape[1:]), dtype=x.dtype, device=DEV)}


def _pairs(v):
    hi = v.float()
    return torch.stack([hi, (v - hi.double()).float()], dim=-1)


def _faces(c, d, axes, per):
    """Inverse centre distances of direction d's faces, as a line, and the two transverse widths."""
    w = np.diff(axes[d])
    dist = 0.5 * (np.roll(w, 1) + w) if per[d] else 0.5 * (w[:-1] + w[1:])
    return torch.as_tensor(dist, dtype=F64, device=DEV)


def _diff(x, d, periodic):
    """x[cell of the face] - x[cell below it] over direction d's faces; x is [nz, ny, nx, k]."""
    dim = 2 - d
    if periodic:
        return x - x.roll(1, dim)
    return x.diff(dim=dim)


def _undiff(f, d, periodic):
    """Face values to cells: f[face above the cell] - f[face below] (0 on the walls)."""
    dim = 2 - d
    if periodic:
        return f.roll(-1, dim) - f
    shape = list(f.shape)
    shape[dim] = 1
    z = torch.zeros(shape, dtype=f.dtype, device=f.device)
    return torch.cat([f, z], dim) - torch.cat([z, f], dim)


def _line(v, d):
    s = [1, 1, 1, 1]
    s[2 - d] = -1
    return v.reshape(s)


def _exact_spmm(c, seed):
    axes, per = _axes(c["grid"], c["nx"], c["ny"], c["nz"])
    shape = (c["nz"], c["ny"], c["nx"])
    k = c["k"]
    x = _spmm_x(c, seed).double()
    w = [torch.as_tensor(np.diff(a), dtype=F64, device=DEV) for a in axes]
    area = [_line(w[(d + 1) % 3], (d + 1) % 3) * _line(w[(d + 2) % 3], (d + 2) % 3) for d in range(3)]
    if c["op"] == "divergence":
        y, at = 0, 0
        for d in range(3):
            fs = list(shape)
            fs[2 - d] -= 0 if per[d] else 1
            nf = fs[0] * fs[1] * fs[2]
            y = y + area[d] * _undiff(x[at:at + nf].reshape(*fs, k), d, per[d])
            at += nf
        y = y.reshape(-1, k)
    elif c["op"] == "27p":
        x = x.reshape(*shape, k)
        h = 1.0 / c["nx"]
        one = [x.roll(-1, d) + x.roll(1, d) for d in range(3)]  # faces
        two = [one[a].roll(-1, b) + one[a].roll(1, b) for a, b in ((0, 1), (0, 2), (1, 2))]  # edges
        three = two[0].roll(-1, 2) + two[0].roll(1, 2)  # corners
        y = (h / 30.0) * (-128.0 * x + 14.0 * (one[0] + one[1] + one[2]) + 3.0 * (two[0] + two[1] + two[2]) + three)
        y = y.reshape(-1, k)
    elif c["op"] == "13p":
        x = x.reshape(*shape, k)
        h = [1.0 / c["nx"], 1.0 / c["ny"], 1.0 / c["nz"]]
        y = 0
        for d in range(3):
            m = 2 - d
            y = y + (-x.roll(2, m) + 16 * x.roll(1, m) - 30 * x + 16 * x.roll(-1, m) - x.roll(-2, m)) / (12 * h[d] ** 2)
        y = (h[0] * h[1] * h[2] * y).reshape(-1, k)
    else:
        x = x.reshape(*shape, k)
        g = [_diff(x, d, per[d]) / _line(_faces(c, d, axes, per), d) for d in range(3)]
        if c["op"] == "gradient":
            y = torch.cat([v.reshape(-1, k) for v in g])
        else:
            y = sum(area[d] * _undiff(g[d], d, per[d]) for d in range(3)).reshape(-1, k)
    return _pairs(y) if c["dtype"] == "df64" else y


# ----------------------------------------------------------------------------- extruded mesh
def _mesh(c, seed):
    """CSR of a vertex-centred Laplacian on a triangulated square (six neighbours, a few edges
    missing, vertices numbered along the rows with a local shuffle) and its spanwise weights."""
    s = c["side"]
    n = s * s
    g = _gen(seed, 7)
    rank = torch.argsort(torch.arange(n, device=DEV, dtype=F64) + 48.0 * torch.rand(n, generator=g, device=DEV, dtype=F64))
    new = torch.empty_like(rank)
    new[rank] = torch.arange(n, device=DEV)
    v = torch.arange(n, device=DEV).reshape(s, s)
    a = torch.cat([v[:, :-1].reshape(-1), v[:-1].reshape(-1), v[:-1, :-1].reshape(-1)])
    b = torch.cat([v[:, 1:].reshape(-1), v[1:].reshape(-1), v[1:, 1:].reshape(-1)])
    keep = torch.rand(a.numel(), generator=g, device=DEV) > 0.01
    a, b = new[a[keep]], new[b[keep]]
    wt = torch.exp(0.4 * torch.randn(a.numel(), generator=g, device=DEV, dtype=F64))
    diag = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, a, wt).index_add_(0, b, wt)
    i = torch.arange(n, device=DEV)
    rows, cols, vals = torch.cat([a, b, i]), torch.cat([b, a, i]), torch.cat([wt, wt, -diag])
    order = torch.argsort(rows * n + cols)
    rp = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    dz = 2.0 / c["k"]
    area = (0.5 + torch.rand(n, generator=g, device=DEV, dtype=F64)) / n
    return rp, cols[order].int(), vals[order], area / dz, dz


def _prepare_extruded(c, seed):
    rp, ci, va, zw, dz = _mesh(c, seed)
    n = rp.numel() - 1
    A = rb.Operator(rp, ci, va, n, dtype=c["dtype"], k_max=c["k"], extruded_nz=c["k"], z_weight=zw, dz=dz)
    x = _normal((n, c["k"]), seed)
    x = x.float() if c["dtype"] == "f32" else x
    return {"A": A, "X": x, "Y": torch.empty_like(x)}


def _exact_extruded(c, seed):
    rp, ci, va, zw, dz = _mesh(c, seed)
    n = rp.numel() - 1
    x = _normal((n, c["k"]), seed)
    x = x.float().double() if c["dtype"] == "f32" else x
    y = torch.empty_like(x)
    for j in range(0, c["k"], 8):  # eight columns of gathered rows at a time
        g = x[ci.long(), j:j + 8] * va[:, None]
        rows = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).long())
        y[:, j:j + 8] = torch.zeros((n, g.shape[1]), dtype=F64, device=DEV).index_add_(0, rows, g)
    return dz * y + zw[:, None] * (x.roll(1, 1) - 2 * x + x.roll(-1, 1))


# ----------------------------------------------------------------------------- Poisson solves
def _solve_exact(grid, nx, ny, nz, b):
    """Zero-mean solution of -L x = b: Fourier along the two uniform periodic axes, the
    eigenvectors of the third axis' generalised problem along that one."""
    axes, per = _axes(grid, nx, ny, nz)
    g = 2 if grid == "rbc" else 1  # the general axis
    h = [float(a[1] - a[0]) for a in axes]
    w = np.diff(axes[g])
    n = w.size
    T = np.zeros((n, n))
    for f in range(n if per[g] else n - 1):
        lo, up = (f, (f + 1) % n)
        t = 1.0 / (0.5 * (w[lo] + w[up]))
        T[lo, lo] += t
        T[up, up] += t
        T[lo, up] -= t
        T[up, lo] -= t
    s = 1.0 / np.sqrt(w)
    lam, Q = np.linalg.eigh(s[:, None] * T * s[None, :])
    lam[0] = 0.0
    Q = torch.as_tensor(s[:, None] * Q, dtype=F64, device=DEV)  # Q^T diag(w) Q = 1
    lam = torch.as_tensor(lam, dtype=F64, device=DEV)
    k = b.shape[1]
    v = b.t().reshape(k, nz, ny, nx)
    others = [d for d in range(3) if d != g]
    if g == 1:
        v = v.permute(0, 2, 1, 3)  # [k, general, other, x]
    fh = torch.fft.rfft2(v, dim=(2, 3))
    m0, m1 = others  # m0 = x (last), m1 = the other one
    n0, n1 = (nx, ny, nz)[m0], (nx, ny, nz)[m1]
    k0 = torch.arange(n0 // 2 + 1, dtype=F64, device=DEV)
    k1 = torch.arange(n1, dtype=F64, device=DEV)
    e0 = 4 * torch.sin(math.pi * k0 / n0) ** 2 * (h[m1] / h[m0])
    e1 = 4 * torch.sin(math.pi * k1 / n1) ** 2 * (h[m0] / h[m1])
    den = lam[:, None, None] * (h[m0] * h[m1]) + e1[None, :, None] + e0[None, None, :]
    den[0, 0, 0] = 1.0
    r = torch.einsum("gi,kgab->kiab", Q.to(fh.dtype), fh) / den
    r[:, 0, 0, 0] = 0
    x = torch.fft.irfft2(torch.einsum("gi,kiab->kgab", Q.to(fh.dtype), r), s=(n1, n0), dim=(2, 3))
    if g == 1:
        x = x.permute(0, 2, 1, 3)
    x = x.reshape(k, -1)
    return (x - x.mean(dim=1, keepdim=True)).t()


def _prepare_mg(c, seed):
    nodes, per = _nodes(c["grid"], c["nx"], c["ny"], c["nz"])
    B = _rhs(c["grid"], c["nx"], c["ny"], c["nz"], c["k"], seed)
    return {"mg": rb.Multigrid(nodes, per, k_max=c["k"]), "B": B, "X": torch.zeros_like(B),
            "prm": rb.mg_params(rtol=1e-10, mixed=c["mixed"])}


def _poisson(nodes, per, k):
    """The FP64 CSR operator A = -L and the matrix-free FP32 one of the inner iterations."""
    A = rb.Operator(*rb.fvm_assemble(nodes, per, rb.RB_FVM_LAPLACIAN, scale=-1.0), dtype="f64", k_max=k)
    return A, rb.Operator.stencil(nodes, per, scale=-1.0, dtype="f32", k_max=k)


def _prepare_cg(c, seed):
    nodes, per = _nodes(c["grid"], c["nx"], c["ny"], c["nz"])
    A, Ai = _poisson(nodes, per, c["k"])
    B = _rhs(c["grid"], c["nx"], c["ny"], c["nz"], c["k"], seed)
    prm = rb.cg_params(rtol=1e-10, mixed=2, project_mean=True)
    return {"A": A, "Ai": Ai, "B": B, "X": torch.zeros_like(B), "prm": prm,
            "work": torch.empty(rb.cg_workspace_bytes(A, c["k"], prm), dtype=torch.uint8, device=DEV)}


def _systems(c):
    return ([("box", c["coarse"], c["coarse"], c["coarse"], 8), ("box", c["fine"], c["fine"], c["fine"], 1)]
            + [("channel", c["nx"], c["ny"], c["nz"], 3)] * c["channels"])


def _prepare_batch(c, seed):
    sys_ = _systems(c)
    ops = [_poisson(*_nodes(*s[:4]), s[4]) for s in sys_]
    Bs = [_rhs(*s, seed, salt=i + 1) for i, s in enumerate(sys_)]
    batch = rb.Batch([o[0] for o in ops], [o[1] for o in ops], [s[4] for s in sys_],
                     rb.cg_params(rtol=1e-10, mixed=2, project_mean=True))
    return {"batch": batch, "Bs": Bs, "Xs": [torch.zeros_like(b) for b in Bs]}


# ----------------------------------------------------------------------------- projection step
NU, DT = 0.01, 0.01


def _flow(c, seed):
    """Stacked Taylor-Green vortices of growing amplitude with noise, and their face velocities."""
    nx, ny, nz, m = c["nx"], c["ny"], c["nz"], c["m"]
    axes, _ = _axes("tau", nx, ny, nz)
    x, y = (torch.as_tensor(0.5 * (a[1:] + a[:-1]), dtype=F64, device=DEV) for a in axes[:2])
    u = 0.01 * _normal((nz, ny, nx, 3, m), seed)
    for s in range(m):
        u[..., 0, s] += (1 + 0.1 * s) * torch.cos(y)[:, None] * torch.sin(x)[None, :]
        u[..., 1, s] -= (1 + 0.1 * s) * torch.sin(y)[:, None] * torch.cos(x)[None, :]
    return u, [0.5 * (u[..., d, :] + u[..., d, :].roll(1, 2 - d)) for d in range(3)]


def _prepare_projection(c, seed):
    nodes, _ = _nodes("tau", c["nx"], c["ny"], c["nz"])
    u, us = _flow(c, seed)
    return {"step": ProjectionStep(torch, nodes, c["m"], NU, DT, mixed=2, solver="mg"),
            "u_c": u.reshape(-1, 3 * c["m"]).contiguous(), "u_s": torch.cat([f.reshape(-1, c["m"]) for f in us])}


def _exact_projection(c, seed):
    nx, ny, nz, m = c["nx"], c["ny"], c["nz"], c["m"]
    h = [2 * math.pi / n for n in (nx, ny, nz)]
    vol = h[0] * h[1] * h[2]
    u0, us = _flow(c, seed)

    def force(u, us):
        out = torch.zeros_like(u)
        for d in range(3):
            dim = 2 - d
            a = vol / h[d]
            out += NU * (a / h[d]) * (u.roll(-1, dim) - 2 * u + u.roll(1, dim))
            flux = 0.5 * (u + u.roll(1, dim)) * us[d][..., None, :]
            out -= a * (flux.roll(-1, dim) - flux)
        return out / vol

    def project(u, cdt):
        ut = [0.5 * (u[..., d, :] + u[..., d, :].roll(1, 2 - d)) for d in range(3)]
        div = sum((vol / h[d]) * (ut[d].roll(-1, 2 - d) - ut[d]) for d in range(3))
        p = _solve_exact("tau", nx, ny, nz, -div.reshape(-1, m) / cdt).reshape(nz, ny, nx, m)
        g = [(p - p.roll(1, 2 - d)) / h[d] for d in range(3)]
        uc = torch.stack([u[..., d, :] - cdt * 0.5 * (g[d] + g[d].roll(-1, 2 - d)) for d in range(3)], dim=3)
        return uc, [ut[d] - cdt * g[d] for d in range(3)]

    f0 = force(u0, us)
    f1 = force(*project(u0 + DT / 3 * f0, DT / 3))
    f2 = force(*project(u0 + 2 * DT / 3 * f1, 2 * DT / 3))
    u, us = project(u0 + DT * (0.25 * f0 + 0.75 * f2), DT)
    return {"u_c": u.reshape(-1, 3 * m), "u_s": torch.cat([f.reshape(-1, m) for f in us])}


# ----------------------------------------------------------------------------- learned guess
CHANNELS = (8, 16, 32, 48)


def _layers():
    """(kind, c_in, c_out) in the order of the flat parameter vector."""
    out, cin = [], 3
    for ch in CHANNELS:
        out += [("conv", cin, ch), ("conv", ch, ch)]
        cin = ch
    for l in range(len(CHANNELS) - 2, -1, -1):
        ch = CHANNELS[l]
        out += [("up", CHANNELS[l + 1], ch), ("conv", 2 * ch, ch), ("conv", ch, ch)]
    return out + [("head", CHANNELS[0], 1)]


def _theta(seed):
    """He-scaled weights, small biases, the head's weights a tenth (as training starts)."""
    g = _gen(seed, 11)
    parts = []
    for kind, ci, co in _layers():
        n, fan = {"conv": (27 * ci * co, 27 * ci), "up": (8 * ci * co, ci), "head": (ci, ci)}[kind]
        wt = torch.randn(n, generator=g, device=DEV) * math.sqrt(2.0 / fan) * (0.1 if kind == "head" else 1.0)
        parts += [wt, 0.01 * torch.randn(co, generator=g, device=DEV)]
    return torch.cat(parts)


def _pressures(c, seed):
    """b and the pressures of three consecutive steps on the Rayleigh-Benard box (walls in z)."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    f = _smooth(3, nx, ny, nz, seed)
    p2 = f[0]
    p1 = 0.95 * p2 + math.sqrt(1 - 0.95 ** 2) * f[1]
    p = 0.95 * p1 + math.sqrt(1 - 0.95 ** 2) * f[2]
    b = -_exact_laplacian(p, nx, ny, nz)
    return [v.reshape(-1).contiguous() for v in (b, p1, p2, p)]


def _exact_laplacian(p, nx, ny, nz):
    axes, per = _axes("rbc", nx, ny, nz)
    w = [torch.as_tensor(np.diff(a), dtype=F64, device=DEV) for a in axes]
    x = p[..., None]
    y = 0
    for d in range(3):
        g = _diff(x, d, per[d]) / _line(_faces(None, d, axes, per), d)
        y = y + _line(w[(d + 1) % 3], (d + 1) % 3) * _line(w[(d + 2) % 3], (d + 2) % 3) * _undiff(g, d, per[d])
    return y[..., 0]


def _prepare_guess(c, seed):
    net = rb.Guess(rb.guess_cfg(c["nx"], c["ny"], c["nz"], CHANNELS, (1, 1, 0)))
    net.set_params(_theta(seed))
    b, p1, p2, p = _pressures(c, seed)
    return {"net": net, "b": b, "p1": p1, "p2": p2, "p": p, "out": torch.empty_like(b),
            "loss": torch.zeros(1, dtype=F64, device=DEV)}


def _network(theta, x):
    """The U-Net in 64 bits on x [1, 3, nz, ny, nx]: circular along x and y, zero-padded in z."""
    at = 0
    it = iter(_layers())

    def take(n):
        nonlocal at
        at += n
        return theta[at - n:at]

    def conv(v):
        _, ci, co = next(it)
        wt = take(27 * ci * co).reshape(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        bias = take(co)
        v = F.pad(F.pad(v, (1, 1, 1, 1, 0, 0), mode="circular"), (0, 0, 0, 0, 1, 1))
        return torch.relu(F.conv3d(v, wt.contiguous(), bias))

    skips = []
    L = len(CHANNELS)
    for l in range(L):
        x = conv(conv(x))
        if l < L - 1:
            skips.append(x)
            x = F.avg_pool3d(x, 2)
    for l in range(L - 2, -1, -1):
        _, ci, co = next(it)
        wt = take(8 * ci * co).reshape(co, 2, 2, 2, ci).permute(4, 0, 1, 2, 3)
        bias = take(co)
        x = torch.cat([F.conv_transpose3d(x, wt.contiguous(), bias, stride=2), skips[l]], dim=1)
        x = conv(conv(x))
    _, ci, co = next(it)
    wt, bias = take(ci), take(1)
    return torch.einsum("c,bczyx->zyx", wt, x) + bias


def _exact_guess(c, seed):
    b, p1, p2, p = _pressures(c, seed)
    shape = (1, 1, c["nz"], c["ny"], c["nx"])
    sb, sp = b.square().mean().sqrt(), p1.square().mean().sqrt()
    x = torch.cat([(b / sb).reshape(shape), (p1 / sp).reshape(shape), (p2 / sp).reshape(shape)], dim=1)
    theta = _theta(seed).double()
    if c["kind"] == "predict":
        with torch.no_grad():
            y = _network(theta, x).reshape(-1)
        return p1 - p1.mean() + sp * (y - y.mean())
    theta.requires_grad_(True)
    y = _network(theta, x).reshape(-1)
    t = (p - p1) / sp
    loss = ((y - y.mean()) - (t - t.mean())).square().mean()
    loss.backward()
    return {"loss": loss.detach().reshape(1), "grad": theta.grad}


# ----------------------------------------------------------------------------- interface
def prepare(case, seed):
    return dict({"spmm": _prepare_spmm, "extruded": _prepare_extruded, "mg": _prepare_mg, "cg": _prepare_cg,
                 "batch": _prepare_batch, "projection": _prepare_projection, "predict": _prepare_guess,
                 "train": _prepare_guess}[case["kind"]](case, seed), kind=case["kind"])


def run(s):
    kind = s["kind"]
    if kind in ("spmm", "extruded"):
        return s["A"].spmm(s["X"], s["Y"])
    if kind == "mg":  # every solve from a zero guess
        s["X"].zero_()
        s["mg"].solve(s["B"], s["X"], s["prm"])
        return s["X"]
    if kind == "cg":
        s["X"].zero_()
        rb.cg_solve(s["A"], s["B"], s["X"], A_inner=s["Ai"], params=s["prm"], work=s["work"])
        return s["X"]
    if kind == "batch":
        for x in s["Xs"]:
            x.zero_()
        s["batch"].solve(s["Bs"], s["Xs"])
        return s["Xs"]
    if kind == "projection":  # the flow advances in place, as in a time loop
        s["step"].step(s["u_c"], s["u_s"])
        return {"u_c": s["u_c"], "u_s": s["u_s"]}
    if kind == "predict":
        return s["net"].predict(s["b"], s["p1"], s["p2"], out=s["out"])
    s["loss"].zero_()
    s["net"].loss_grad(s["b"], s["p1"], s["p2"], s["p"], loss=s["loss"])
    return {"loss": s["loss"], "grad": s["net"].grad()}


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "spmm":
        return _exact_spmm(c, seed)
    if kind == "extruded":
        return _exact_extruded(c, seed)
    if kind in ("mg", "cg"):
        g = (c["grid"], c["nx"], c["ny"], c["nz"])
        return _solve_exact(*g, _rhs(*g, c["k"], seed))
    if kind == "batch":
        return [_solve_exact(*s[:4], _rhs(*s, seed, salt=i + 1)) for i, s in enumerate(_systems(c))]
    if kind == "projection":
        return _exact_projection(c, seed)
    return _exact_guess(c, seed)


def work(case):
    c = case
    kind = c["kind"]
    if kind == "spmm":
        nr, nc, nnz = _spmm_sizes(c)
        s = 4 if c["dtype"] == "f32" else 8
        matrix = 0 if c["fmt"] == "free" else nnz * (4 + s) + 4 * (nr + 1)
        return {"bytes": matrix + s * c["k"] * (nr + nc), "flops": 2 * nnz * c["k"]}
    if kind == "extruded":
        n = c["side"] ** 2
        s = 4 if c["dtype"] == "f32" else 8
        return {"bytes": 7 * n * (4 + s) + (4 + s) * n + 2 * s * c["k"] * n, "flops": (14 + 4) * n * c["k"]}
    if kind == "batch":
        nk = [s[1] * s[2] * s[3] * s[4] for s in _systems(c)]
        return {"bytes": 24 * sum(nk), "flops": 25 * 300 * sum(nk)}
    n = c["nx"] * c["ny"] * c["nz"]
    if kind == "mg":  # b and the guess read, x written; about ten cycles of ~100 flops per unknown
        return {"bytes": 24 * n * c["k"], "flops": 1000 * n * c["k"]}
    if kind == "cg":  # the matrix too; about 25 flops per unknown, six iterations per cell of the longest axis
        return {"bytes": 24 * n * c["k"] + 88 * n, "flops": 25 * 6 * max(c["nx"], c["ny"], c["nz"]) * n * c["k"]}
    if kind == "projection":  # (u_c, u_s) read and written; three solves and about 500 flops per cell and state
        return {"bytes": 96 * n * c["m"], "flops": 3500 * n * c["m"]}
    f = 2 * 27 * sum(ci * co * n / 8 ** l for l, ci, co in _conv_levels())
    return {"bytes": 32 * n, "flops": f if kind == "predict" else 3 * f}


def _conv_levels():
    L = len(CHANNELS)
    cin = 3
    for l, ch in enumerate(CHANNELS):
        yield l, cin, ch
        yield l, ch, ch
        cin = ch
        if l < L - 1:
            yield l, 2 * ch, ch
            yield l, ch, ch
