"""What the library is used for, as cases that can be timed and compared.

A case is one call, or one short sequence of calls, that a program makes
through the package's public entry points (`device.Preconditioner`, `amdd.*`,
`learned.ProposalModel`):

  spmv    y = A x
  apply   z = M^-1 r with a handle that is already set up
  pcg     preconditioned conjugate gradients with such a handle, one or
          several right-hand sides
  gmres   GMRES(30) with the deflated two-level form
  setup   the whole way from a matrix and a partition to a solution: setup,
          solve, in FP64 also the singular values of the local block rows,
          release
  train   one optimiser step of the proposal network

The mixed form (`precision` 1) is measured where it is used: inside a solve,
whose result carries the accuracy of the FP64 outer iteration.
"""
import math

import numpy as np
import torch

from paper_2109_05908_gb300 import amdd
from paper_2109_05908_gb300 import learned
from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner, stream_ptr


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # one product of a small system inside somebody's own iteration: launch latency
        {"name": "spmv_7pt_16", "kind": "spmv", "pattern": "grid", "nx": 16, "ny": 16, "nz": 16},
        # the operator of a large 2D problem, odd sides, about 2.1M unknowns
        {"name": "spmv_5pt_2m", "kind": "spmv", "pattern": "grid", "nx": 1501, "ny": 1399, "nz": 1},
        # a vector problem: three unknowns a node, 27-point neighbourhood, up to 81 entries a row
        {"name": "spmv_27pt_3dof", "kind": "spmv", "pattern": "nodes", "nx": 31, "ny": 32, "nz": 33},
        # the two-level operator of a small 2D Laplacian in a user's own Krylov method
        {"name": "apply_lap64_fp64", "kind": "apply", "nx": 64, "ny": 64, "nz": 1, "px": 4, "py": 4, "pz": 1,
         "jitter": 0.0, "contrast": 0.0, "channels": 0, "overlap": 1, "tau": 50.0, "precision": 0, "nrhs": 1},
        # the one-level operator of many small subdomains (a tau that selects nothing): bandwidth of the local solves
        {"name": "apply_lap512_onelevel", "kind": "apply", "nx": 512, "ny": 512, "nz": 1, "px": 32, "py": 32, "pz": 1,
         "jitter": 0.0, "contrast": 0.0, "channels": 0, "overlap": 1, "tau": 1e-17, "precision": 0, "nrhs": 1},
        # repeated solves with one setup: uneven 3D subdomains, channelled diffusion, mixed form
        {"name": "pcg_diff24_mixed", "kind": "pcg", "nx": 24, "ny": 24, "nz": 24, "px": 4, "py": 2, "pz": 2,
         "jitter": 0.3, "contrast": 2.0, "channels": 16, "overlap": 2, "tau": 100.0, "precision": 1, "nrhs": 1},
        # eight right-hand sides solved together
        {"name": "pcg_diff20_8rhs", "kind": "pcg", "nx": 20, "ny": 20, "nz": 20, "px": 3, "py": 2, "pz": 2,
         "jitter": 0.3, "contrast": 2.0, "channels": 8, "overlap": 2, "tau": 100.0, "precision": 1, "nrhs": 8},
        # deflated GMRES(30) with a partial coarse space, plain FP64
        {"name": "gmres_lap96_fp64", "kind": "gmres", "nx": 96, "ny": 96, "nz": 1, "px": 6, "py": 6, "pz": 1,
         "jitter": 0.0, "contrast": 0.0, "channels": 0, "overlap": 1, "tau": 0.5, "precision": 0, "nrhs": 1},
        # a small problem from matrix to solution, mixed form
        {"name": "setup_lap64_mixed", "kind": "setup", "nx": 64, "ny": 64, "nz": 1, "px": 4, "py": 4, "pz": 1,
         "jitter": 0.0, "contrast": 0.0, "channels": 0, "overlap": 1, "tau": 50.0, "precision": 1, "nrhs": 1},
        # the benchmark's shape: 24^3 channelled diffusion, 16 uneven subdomains, mixed form
        {"name": "setup_diff24_mixed", "kind": "setup", "nx": 24, "ny": 24, "nz": 24, "px": 4, "py": 2, "pz": 2,
         "jitter": 0.3, "contrast": 2.0, "channels": 16, "overlap": 2, "tau": 100.0, "precision": 1, "nrhs": 1},
        # plain FP64 with a partial selection: eigenvectors and a small coarse space
        {"name": "setup_diff13_fp64", "kind": "setup", "nx": 13, "ny": 12, "nz": 12, "px": 2, "py": 2, "pz": 2,
         "jitter": 0.3, "contrast": 1.0, "channels": 0, "overlap": 1, "tau": 0.5, "precision": 0, "nrhs": 1},
        # training of the proposal network on 2000 subdomains
        {"name": "train_2000", "kind": "train", "samples": 2000},
    ]


def _log(rng, lo, hi):
    return lo * math.exp(rng.random() * math.log(hi / lo))


def draw(rng):
    kind = rng.choice(["spmv", "spmv", "apply", "apply", "pcg", "gmres", "setup", "setup", "train"])
    if kind == "train":
        return {"kind": "train", "samples": int(_log(rng, 60, 2000))}
    if kind == "spmv":
        what = rng.choice(["2d", "3d", "nodes"])
        if what == "2d":
            n = _log(rng, 900, 2.0e6)
            nx = max(8, int(math.sqrt(n) * rng.uniform(0.7, 1.3)))
            return {"kind": "spmv", "pattern": "grid", "nx": nx, "ny": max(8, int(n / nx)), "nz": 1}
        if what == "3d":
            s = _log(rng, 1000, 1.4e6) ** (1 / 3)
            a, b = s * rng.uniform(0.85, 1.15), s * rng.uniform(0.85, 1.15)
            return {"kind": "spmv", "pattern": "grid", "nx": int(a), "ny": int(b), "nz": int(s ** 3 / (a * b))}
        s = _log(rng, 200, 3.0e4) ** (1 / 3)
        return {"kind": "spmv", "pattern": "nodes", "nx": int(s), "ny": int(s) + 1, "nz": int(s) + rng.randint(0, 2)}
    flat = rng.random() < 0.5
    mixed = kind in ("pcg", "setup") and rng.random() < 0.7
    c = {"kind": kind, "nz": 1, "pz": 1, "jitter": 0.0, "contrast": 0.0, "channels": 0, "overlap": 1,
         "precision": 1 if mixed else 0, "nrhs": 1}
    if kind == "apply" and rng.random() < 0.5:  # one-level, many boxes
        c["px"], c["py"] = rng.randint(6, 30), rng.randint(6, 30)
        side = rng.randint(9, 16)
        c["nx"], c["ny"] = c["px"] * side + rng.randint(0, 5), c["py"] * side
        c["tau"], c["nrhs"] = 1e-17, rng.choice([1, 1, 3, 8])
        return c
    if flat or kind == "gmres":
        c["px"], c["py"] = rng.randint(2, 5), rng.randint(2, 5)
        side = rng.randint(10, 17)
        c["nx"], c["ny"] = c["px"] * side + rng.randint(0, 3), c["py"] * side + rng.randint(0, 3)
    else:
        c["px"], c["py"], c["pz"] = rng.randint(2, 3), 2, 2
        side = rng.randint(6, 9 if mixed else 6)
        c["nx"], c["ny"], c["nz"] = c["px"] * side + rng.randint(0, 2), c["py"] * side + 1, c["pz"] * side
        c["jitter"] = 0.3
        if mixed:
            c["contrast"], c["channels"], c["overlap"] = 2.0, rng.randint(2, 8), rng.randint(1, 2)
        else:
            c["contrast"] = 1.0
    c["tau"] = 0.5 if kind == "gmres" else rng.choice([50.0, 100.0])
    if kind in ("apply", "pcg"):
        c["nrhs"] = rng.choice([1, 1, 3, 8])
    return c


# ---------------------------------------------------------------- inputs
class _Csr:
    def __init__(self, n, rowptr, colind, val):
        self.n, self.rowptr, self.colind, self.val = n, rowptr, colind, val


def _csr(n, rows, cols, vals):
    order = torch.from_numpy(rows * np.int64(n) + cols).cuda().argsort().cpu().numpy()
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=ptr[1:])
    return _Csr(n, ptr, cols[order].astype(np.int32), vals[order])


def _smooth_field(shape, corr, rng):
    """Unit-variance Gaussian field of correlation length `corr` (periodic)."""
    g = rng.standard_normal(shape)
    half = int(math.ceil(3 * corr))
    t = np.arange(-half, half + 1)
    k = np.exp(-0.5 * (t / corr) ** 2)
    for ax in range(len(shape)):
        if shape[ax] > 1:
            g = sum(w * np.roll(g, int(o), axis=ax) for o, w in zip(t, k / k.sum()))
    return (g - g.mean()) / g.std()


def _diffusion(c, rng):
    """Cell-centred finite volumes on an nz x ny x nx grid, Dirichlet boundary:
    harmonic face means of exp(contrast * field) with one-cell channels of 1e6
    along x.  contrast 0: the 5- or 7-point Laplacian."""
    shape = (c["nz"], c["ny"], c["nx"])
    kappa = np.ones(shape)
    if c["contrast"]:
        kappa = np.exp(c["contrast"] * _smooth_field(shape, min(8.0, c["nx"] / 3), rng))
        for _ in range(c["channels"]):
            kappa[rng.integers(shape[0]), rng.integers(shape[1]), :] = 1e6
    n = kappa.size
    idx = np.arange(n).reshape(shape)
    diag = np.zeros(shape)
    rows, cols, vals = [], [], []
    for ax in range(3):
        if shape[ax] == 1:
            continue
        lo, hi = [slice(None)] * 3, [slice(None)] * 3
        lo[ax], hi[ax] = slice(0, -1), slice(1, None)
        lo, hi = tuple(lo), tuple(hi)
        t = 2.0 * kappa[lo] * kappa[hi] / (kappa[lo] + kappa[hi])
        diag[lo] += t
        diag[hi] += t
        i, j, v = idx[lo].ravel(), idx[hi].ravel(), -t.ravel()
        rows += [i, j]
        cols += [j, i]
        vals += [v, v]
        for face in (0, -1):
            at = [slice(None)] * 3
            at[ax] = face
            diag[tuple(at)] += (2.0 if c["contrast"] else 1.0) * kappa[tuple(at)]
    rows.append(idx.ravel())
    cols.append(idx.ravel())
    vals.append(diag.ravel())
    return _csr(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))


def _nodes(c, rng):
    """Symmetric matrix of three unknowns a node on the 27-point neighbourhood."""
    shape = (c["nz"], c["ny"], c["nx"])
    nodes = shape[0] * shape[1] * shape[2]
    idx = np.arange(nodes).reshape(shape)
    rows, cols = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                a = [slice(max(0, -d), s - max(0, d)) for d, s in zip((dz, dy, dx), shape)]
                b = [slice(max(0, d), s - max(0, -d)) for d, s in zip((dz, dy, dx), shape)]
                rows.append(idx[tuple(a)].ravel())
                cols.append(idx[tuple(b)].ravel())
    r, q = np.concatenate(rows), np.concatenate(cols)
    r = (3 * r[:, None, None] + np.arange(3)[None, :, None]).repeat(3, axis=2).ravel()
    q = (3 * q[:, None, None] + np.arange(3)[None, None, :]).repeat(3, axis=1).ravel()
    return _csr(3 * nodes, r, q, np.where(r == q, 30.0, -0.3))


def _partition(c):
    """Boxes px x py x pz (jitter 0), else the cells nearest in the 1-norm to
    points moved off the box centres: uneven connected regions, the same for
    every matrix on a grid."""
    rng = np.random.default_rng([c["nx"], c["ny"], c["nz"]])
    size, parts = (c["nz"], c["ny"], c["nx"]), (c["pz"], c["py"], c["px"])
    z, y, x = np.meshgrid(*[np.arange(s) for s in size], indexing="ij")
    if not c["jitter"]:
        b = [np.minimum(v * p // s, p - 1) for v, s, p in zip((z, y, x), size, parts)]
        return ((b[0] * parts[1] + b[1]) * parts[2] + b[2]).ravel().astype(np.int32)
    best = np.full(size, np.inf)
    part = np.zeros(size, np.int32)
    k = 0
    for i in range(parts[0]):
        for j in range(parts[1]):
            for q in range(parts[2]):
                at = [(v + 0.5 + (rng.uniform(-1, 1) * c["jitter"] if p > 1 else 0.0)) * s / p
                      for v, s, p in zip((i, j, q), size, parts)]
                d = abs(z + 0.5 - at[0]) + abs(y + 0.5 - at[1]) + abs(x + 0.5 - at[2]) + 1e-9 * k
                part[d < best] = k
                best = np.minimum(best, d)
                k += 1
    return np.unique(part.ravel(), return_inverse=True)[1].reshape(-1).astype(np.int32)


def _problem(case, seed):
    rng = np.random.default_rng([seed, 77])
    A = _diffusion(case, rng)
    part = _partition(case)
    b = rng.uniform(-1.0, 1.0, (case["nrhs"], A.n))
    return A, part, b


def _opts(case):
    o = amdd.opts_default()
    o.precision = case["precision"]
    return o


def _train_inputs(case, seed):
    rng = np.random.default_rng([seed, 78])
    n = case["samples"]
    feat = rng.standard_normal((n, learned.NF)).astype(np.float32)
    basis = np.linalg.qr(rng.standard_normal((n, learned.NB, 6)))[0]
    target = (basis @ basis.transpose(0, 2, 1)).reshape(n, -1).astype(np.float32)
    return feat, target, learned.init_weights(seed)


def _bf16(w):
    return w.to(torch.bfloat16).to(torch.float32)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "spmv":
        rng = np.random.default_rng([seed, 79])
        A = _nodes(case, rng) if case["pattern"] == "nodes" else _diffusion(dict(case, contrast=0.0), rng)
        d = rng.uniform(0.5, 1.5, A.n)  # symmetric scaling: other values with another seed
        A.val = A.val * np.repeat(d, np.diff(A.rowptr)) * d[A.colind]
        s["A"] = DeviceMatrix(A)
        s["x"] = torch.from_numpy(rng.standard_normal(A.n)).cuda()
        return s
    if case["kind"] == "train":
        feat, target, w = _train_inputs(case, seed)
        n = case["samples"]
        s["x"], s["q"] = torch.from_numpy(feat).cuda(), torch.from_numpy(target).cuda()
        s["w0"] = torch.from_numpy(w).cuda()
        s["wb0"] = _bf16(s["w0"])
        for k in ("w", "wb", "m", "v", "grad"):
            s[k] = torch.empty_like(s["w0"])
        s["work"] = torch.empty(amdd.mlp_sizes(n)[1], dtype=torch.float32, device="cuda")
        s["loss"] = torch.empty(1, dtype=torch.float32, device="cuda")
        return s
    A, part, b = _problem(case, seed)
    s["A"], s["part"], s["N"] = DeviceMatrix(A), torch.from_numpy(part).cuda(), int(part.max()) + 1
    s["b"] = torch.from_numpy(b).cuda()
    if case["kind"] != "setup":
        s["P"] = Preconditioner(s["A"], s["part"], s["N"], case["overlap"], case["tau"], _opts(case))
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c = s["case"]
    if c["kind"] == "spmv":
        y = torch.empty_like(s["x"])
        amdd.spmv(s["A"].csr, s["x"].data_ptr(), y.data_ptr(), stream_ptr())
        return y
    if c["kind"] == "train":  # a step from the same weights and moments each time
        s["w"].copy_(s["w0"])
        s["wb"].copy_(s["wb0"])
        s["m"].zero_()
        s["v"].zero_()
        amdd.mlp_train_step(*(s[k].data_ptr() for k in ("w", "wb", "m", "v")), 1, 1e-3, s["x"].data_ptr(),
                            s["q"].data_ptr(), c["samples"], s["grad"].data_ptr(), s["work"].data_ptr(),
                            s["loss"].data_ptr(), stream_ptr())
        return {k: s[k] for k in ("grad", "m", "v", "w", "loss")}
    b = s["b"]
    if c["kind"] == "apply":
        z = torch.empty_like(b)
        s["P"].apply(b, z, c["nrhs"])
        return z
    x = torch.zeros_like(b)
    if c["kind"] == "pcg":
        s["P"].solve(b, x, c["nrhs"])
        return x
    if c["kind"] == "gmres":
        s["P"].gmres(b, x, amdd.FORM_DEFLATED, c["nrhs"])
        return x
    P = Preconditioner(s["A"], s["part"], s["N"], c["overlap"], c["tau"], _opts(c))
    P.solve(b, x, c["nrhs"])
    if c["precision"]:  # a result in FP64 accuracy: the solution (the local spectra are FP32 ones)
        P.close()
        return {"x": x}
    sigma = np.concatenate([amdd.get_singular_values(P.h, i) for i in range(s["N"])])
    P.close()
    return {"x": x, "sigma": sigma}


# ---------------------------------------------------------------- what a pass cannot do without
def _grid_nnz(c):
    s = (c["nx"], c["ny"], c["nz"])
    if c.get("pattern") == "nodes":
        nnz = 9
        for d in s:
            nnz *= 3 * d - 2
        return 3 * s[0] * s[1] * s[2], nnz
    n = s[0] * s[1] * s[2]
    return n, n + sum(2 * n // d * (d - 1) for d in s)


def work(case):
    if case["kind"] == "train":
        n, p = case["samples"], learned.NP
        return {"bytes": 4.0 * (n * (learned.NF + 256) + 9 * p), "flops": 6.0 * n * p}
    n, nnz = _grid_nnz(case)
    matrix = 12.0 * nnz + 8.0 * n
    if case["kind"] == "spmv":
        return {"bytes": matrix + 16.0 * n, "flops": 2.0 * nnz}
    own = np.bincount(_partition(case)).astype(np.float64)
    dims = 3 if case["nz"] > 1 else 2
    ov = case["overlap"]
    ni = np.minimum((own ** (1 / dims) + 2 * ov) ** dims, n)       # with the overlap
    nt = np.minimum((own ** (1 / dims) + 2 * ov + 2) ** dims, n)   # and one layer more
    word = 4.0 if case["precision"] else 8.0
    factor = word * float(np.sum(ni * (ni + 1) / 2))               # each local factor once
    vec = 16.0 * n * case["nrhs"]
    one = {"bytes": factor + vec, "flops": case["nrhs"] * 4.0 * float(np.sum(ni * ni / 2))}
    if case["kind"] == "apply":
        return one
    its = 20.0
    solve = {"bytes": its * (one["bytes"] + matrix + 3 * vec), "flops": its * (one["flops"] + 2.0 * nnz * case["nrhs"])}
    if case["kind"] != "setup":
        return solve
    svd = float(np.sum(4 * ni * ni * nt + 8 * ni ** 3))
    dense = float(np.sum(ni * ni * nt + nt ** 3 / 3 + ni ** 3 / 3 + 16 / 3 * own ** 3))
    return {"bytes": solve["bytes"] + word * float(np.sum(ni * nt + nt * nt)), "flops": solve["flops"] + svd + dense}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _dense(A):
    D = torch.zeros((A.n, A.n), dtype=torch.float64, device="cuda")
    rows = torch.from_numpy(np.repeat(np.arange(A.n), np.diff(A.rowptr))).cuda()
    D[rows, torch.from_numpy(A.colind.astype(np.int64)).cuda()] = torch.from_numpy(A.val).cuda()
    return D


def _overlapping(A, part, overlap):
    """The unknowns of each subdomain with its overlap."""
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    out = []
    for i in range(int(part.max()) + 1):
        inside = part == i
        for _ in range(overlap):
            grown = inside.copy()
            grown[A.colind[inside[rows]]] = True
            inside = grown
        out.append(np.flatnonzero(inside))
    return out


def _submatrix(A, at):
    pos = np.full(A.n, -1)
    pos[at] = np.arange(len(at))
    start, count = A.rowptr[at], A.rowptr[at + 1] - A.rowptr[at]
    k = np.repeat(start - np.concatenate([[0], np.cumsum(count)[:-1]]), count) + np.arange(count.sum())
    r, q = np.repeat(np.arange(len(at)), count), pos[A.colind[k]]
    S = np.zeros((len(at), len(at)))
    S[r[q >= 0], q[q >= 0]] = A.val[k][q >= 0]
    return torch.from_numpy(S).cuda()


def _exact_train(case, seed):
    feat, target, w = _train_inputs(case, seed)
    w = torch.from_numpy(w).cuda()
    x, qt = (torch.from_numpy(v).cuda().double() for v in (feat, target))
    wb = _bf16(w).double().requires_grad_(True)
    nf, h = learned.NF, 256
    at, lay = 0, []
    for shape in ((nf, h), (h,), (h, h), (h,), (h, h), (h,)):
        k = math.prod(shape)
        lay.append(wb[at:at + k].view(shape))
        at += k
    y = torch.relu(x @ lay[0] + lay[1])
    y = torch.relu(y @ lay[2] + lay[3]) @ lay[4] + lay[5]
    y = y.view(-1, learned.NB, learned.NB)
    q = 0.5 * (y + y.transpose(1, 2))
    loss = (q.reshape(len(x), -1) - qt).square().sum(1).mean()
    loss.backward()
    g = wb.grad
    m, v = 0.1 * g, 0.001 * g * g
    step = (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"grad": g, "m": m, "v": v, "w": w.double() - 1e-3 * step, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "spmv":
        s = prepare(case, seed)
        rows = torch.repeat_interleave(torch.arange(s["A"].n, device="cuda"), s["A"].rowptr.diff())
        return torch.zeros_like(s["x"]).index_add_(0, rows, s["A"].val * s["x"][s["A"].colind.long()])
    A, part, b = _problem(case, seed)
    bt = torch.from_numpy(b).cuda().T
    sets = _overlapping(A, part, case["overlap"])
    if case["kind"] == "apply":
        z = torch.zeros_like(bt)
        for at in sets:
            t = torch.from_numpy(at).cuda()
            z[t] += torch.linalg.solve(_submatrix(A, at), bt[t])
        if case["tau"] > 1.0:  # every eigenvector is selected: the coarse space is everything
            z += torch.linalg.solve(_dense(A), bt)
        return z.T.contiguous()
    D = _dense(A)
    x = torch.cholesky_solve(bt, torch.linalg.cholesky(D)).T.contiguous()
    if case["kind"] != "setup":
        return x
    if case["precision"]:
        return {"x": x}
    # the rows of the subdomain, whole: X_i up to columns of zeros
    return {"x": x, "sigma": torch.cat([torch.linalg.svdvals(D[torch.from_numpy(at).cuda()]) for at in sets])}
