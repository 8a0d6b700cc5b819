"""The measured workloads: what a program that uses this library has it do.

Products y = alpha*A*x + beta*y through a tuned plan (from a 4096-row grid
operator to a 116 M entry graph, in the three storage types), raw CSR arrays
through the allocation-free call, several independent products side by side,
a multigrid hierarchy as one batch, a mixed-precision CG solve, the way from
a CSR matrix to its first product, and a training step of the selector.

Matrices are the structures the library is configured and tested on (grid
stencils, box stencils of coarse multigrid levels, random graphs with Poisson
or Zipf row lengths, dense diagonal blocks), generated on the GPU from a seed.
"""
import math

import numpy as np
import torch

import paper_1210_2536_gb300 as smat

DEV = "cuda:0"
ALPHA, CAP = 1.8, 10000          # Zipf exponent and longest row of the power-law graphs
VT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
XT = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}
ESZ = {"f64": 8, "f32": 4, "bf16": 2}


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a 64 x 64 grid operator: the smallest product, bound by launch latency
        {"name": "spmv_grid2d_64_f64", "op": "spmv", "kind": "grid2d", "size": 64, "dtype": "f64", "residual": False},
        # the 7-point operator of a 128^3 PDE grid in single precision
        {"name": "spmv_grid3d_128_f32", "op": "spmv", "kind": "grid3d", "size": 128, "dtype": "f32", "residual": False},
        # a residual r = b - A x on a random graph, as an iterative solver forms it
        {"name": "residual_uniform_1000000_f64", "op": "spmv", "kind": "uniform", "size": 1000000, "dtype": "f64",
         "residual": True},
        # a graph product (ranking, eigenvectors) with power-law rows
        {"name": "spmv_powerlaw_2000000_f64", "op": "spmv", "kind": "powerlaw", "size": 2000000, "dtype": "f64",
         "residual": False},
        # the largest graph, values stored in bfloat16 to halve its bytes
        {"name": "spmv_powerlaw_8000000_bf16", "op": "spmv", "kind": "powerlaw", "size": 8000000, "dtype": "bf16",
         "residual": False},
        # CSR arrays that the caller owns, through the call that allocates nothing
        {"name": "noalloc_powerlaw_1500007_f32", "op": "noalloc", "kind": "powerlaw", "size": 1500007, "dtype": "f32",
         "residual": False},
        # four structures in two precisions, eight independent products side by side
        {"name": "many_structures_f64_f32", "op": "many", "grid": 128, "uniform": 1000000, "powerlaw": 2000000,
         "blocks": 1000000},
        # the levels of a multigrid hierarchy with unrelated matrices of other sizes, one batch
        {"name": "batch_hierarchy_128_f64", "op": "batch", "top": 128, "levels": 5, "mixed": 24, "dtype": "f64"},
        # an implicit time step on a 256^3 grid: mixed-precision CG with a fixed number of steps
        {"name": "cg_grid3d_256", "op": "cg", "size": 256, "shift": 1.0, "inner": 40, "outer": 4, "inner_dtype": "f32"},
        # from CSR to the first product: intake, features, the selector's own pick, conversion
        {"name": "setup_powerlaw_2000000_f64", "op": "setup", "kind": "powerlaw", "size": 2000000, "dtype": "f64",
         "variant": "learned"},
        # the same for a caller that knows its format
        {"name": "setup_uniform_1000000_f32_sell", "op": "setup", "kind": "uniform", "size": 1000000, "dtype": "f32",
         "variant": "sell"},
        # one optimiser step of the selector at the training driver's batch size
        {"name": "train_128", "op": "train", "batch": 128},
    ]


def draw(rng):
    op = rng.choice(["spmv"] * 8 + ["noalloc"] * 3 + ["many", "batch"] + ["cg"] * 3 + ["setup"] * 4 + ["train"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if op in ("spmv", "noalloc", "setup"):
        kind = rng.choice(["grid2d", "grid3d", "box", "uniform", "uniform", "powerlaw", "powerlaw", "blocks"])
        size = {"grid2d": lambda: log_int(32, 2000), "grid3d": lambda: log_int(10, 160), "box": lambda: log_int(8, 64),
                "uniform": lambda: log_int(1000, 3000000), "powerlaw": lambda: log_int(1000, 4000000),
                "blocks": lambda: log_int(1000, 4000000)}[kind]()
        c = {"op": op, "kind": kind, "size": size, "dtype": rng.choice(["f64", "f64", "f32", "f32", "bf16"])}
        if op == "setup":
            fits = {"grid2d": ["dia", "ell", "csr_vec4"], "grid3d": ["dia", "ell", "hyb"], "box": ["csr_vec32", "sell"],
                    "uniform": ["sell", "hyb", "coo"], "powerlaw": ["coo", "csr_merge", "hyb"],
                    "blocks": ["bcsr", "ell", "dia"]}
            c["variant"] = rng.choice(["learned", "learned"] + fits[kind])
        else:
            c["residual"] = rng.random() < 0.4
        return c
    if op == "many":
        return {"op": op, "grid": log_int(16, 128), "uniform": log_int(1000, 1000000),
                "powerlaw": log_int(1000, 2000000), "blocks": log_int(1000, 1000000)}
    if op == "batch":
        return {"op": op, "top": log_int(24, 128), "levels": rng.randint(2, 5), "mixed": rng.randint(0, 24),
                "dtype": rng.choice(["f64", "f32"])}
    if op == "cg":
        return {"op": op, "size": log_int(16, 200), "shift": round(rng.uniform(0.8, 3.0), 3),
                "inner": rng.randint(38, 48), "outer": 4, "inner_dtype": rng.choice(["f32", "f32", "bf16"])}
    return {"op": op, "batch": log_int(32, 4096)}


# ---------------------------------------------------------------------------
# Matrices: (m, n, rowptr int32, colidx int32, values float64), on the GPU
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _offsets(kind, r):
    """Neighbours (z, y, x) in the order of their columns."""
    k = range(-r, r + 1)
    box = [(z, y, x) for z in k for y in k for x in k]
    if kind in ("grid2d", "grid3d"):
        box = [d for d in box if sum(map(abs, d)) <= 1]
    return [d for d in box if d[0] == 0] if kind == "grid2d" else box


def _stencil(kind, size, r=1):
    """Rows, in-range columns and the diagonal of a grid stencil, in CSR order."""
    nz = 1 if kind == "grid2d" else size
    n = nz * size * size
    i = torch.arange(n, device=DEV)
    z, y, x = i // (size * size), (i // size) % size, i % size
    ok, cols = [], []
    for dz, dy, dx in _offsets(kind, r):
        ok.append((z + dz >= 0) & (z + dz < nz) & (y + dy >= 0) & (y + dy < size) & (x + dx >= 0) & (x + dx < size))
        cols.append((i + (dz * size + dy) * size + dx).to(torch.int32))
    ok, cols = torch.stack(ok, 1), torch.stack(cols, 1)
    length = ok.sum(1)
    return n, length, cols[ok]


def _zipf_cdf(cap):
    k = np.arange(1, cap + 1, dtype=np.float64)
    w = k ** -ALPHA
    return np.cumsum(w) / w.sum()


def _random_columns(length, n, g):
    """Sorted columns, uniform over [0, n), a row's repeated draws dropped."""
    m = length.numel()
    row = torch.repeat_interleave(torch.arange(m, device=DEV), length)
    key = row * n + torch.randint(0, n, (row.numel(),), device=DEV, generator=g)
    del row
    key = torch.unique_consecutive(torch.sort(key).values)
    row = key // n
    return torch.bincount(row, minlength=m), (key - row * n).to(torch.int32)


def matrix(kind, size, seed):
    g = _gen(seed)
    if kind in ("grid2d", "grid3d", "box", "grid27"):
        n, length, col = _stencil(kind, size, 2 if kind == "box" else 1)
        m = n
    elif kind == "blocks":
        m = n = size
        b = torch.arange(m, device=DEV) // 8 * 8
        c = b[:, None] + torch.arange(8, device=DEV)[None, :]
        ok = c < n
        length, col = ok.sum(1), c[ok].to(torch.int32)
    else:
        m = n = size
        if kind == "uniform":
            length = torch.poisson(torch.full((m,), 16.0, device=DEV), generator=g).long()
        else:
            cdf = torch.from_numpy(_zipf_cdf(min(CAP, n))).to(DEV)
            u = torch.rand(m, dtype=torch.float64, device=DEV, generator=g)
            length = torch.searchsorted(cdf, u).clamp_(max=cdf.numel() - 1) + 1
        length, col = _random_columns(length, n, g)
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length, 0, out=rowptr[1:])
    val = torch.randn(col.numel(), dtype=torch.float64, device=DEV, generator=g)
    return m, n, rowptr.to(torch.int32), col, val


def _vector(n, seed, dtype):
    g = _gen(seed * 7 + 5)
    return (torch.rand(n, dtype=torch.float64, device=DEV, generator=g) * 2 - 1).to(XT[dtype])


def _handle(A, dtype, tune=True):
    m, n, rowptr, col, val = A
    M = smat.SpMatrix(m, n, rowptr, col, val.to(VT[dtype]), dtype)
    if tune:
        M.tune("learned")
    return M


def _load_model():
    if smat.smat_load_model(smat.MODEL_PATH) != smat.SMAT_OK:
        raise RuntimeError("the selector's model did not load")


def _many(case):
    return [(k, s, d) for k, s in (("grid3d", case["grid"]), ("uniform", case["uniform"]),
                                   ("powerlaw", case["powerlaw"]), ("blocks", case["blocks"])) for d in ("f64", "f32")]


def _batch(case):
    """Kinds and sizes of the batch's members: the grids of the hierarchy, then a fixed mixture."""
    got = [("grid27", max(4, case["top"] >> k)) for k in range(case["levels"])]
    for i in range(case["mixed"]):
        n = int(1000 * 1000 ** (((i * 7919 + 3) % 97) / 97.0))
        got.append((("uniform", n), ("powerlaw", n), ("blocks", n), ("grid3d", max(4, round(n ** (1 / 3)))))[i % 4])
    return got


def _spd(case):
    """shift*I + the 7-point Laplacian of a cubic grid (an implicit heat step)."""
    n, length, col = _stencil("grid3d", case["size"])
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length, 0, out=rowptr[1:])
    row = torch.repeat_interleave(torch.arange(n, device=DEV, dtype=torch.int32), length)
    val = torch.where(row == col, 6.0 + case["shift"], -1.0).to(torch.float64)
    return n, n, rowptr.to(torch.int32), col, val


def _spd_shift(case):
    # a shift that bfloat16 holds exactly, so that the solve's two matrices are the same one
    return {**case, "shift": float(torch.tensor(6.0 + case["shift"]).to(torch.bfloat16)) - 6.0}


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    s = {"op": op}
    _load_model()
    if op == "spmv":
        A = matrix(case["kind"], case["size"], seed)
        s["M"] = _handle(A, case["dtype"])
        s["x"] = _vector(A[1], seed, case["dtype"])
        s["b"] = _vector(A[0], seed + 1, case["dtype"]) if case["residual"] else None
        s["y"] = torch.empty(A[0], dtype=XT[case["dtype"]], device=DEV)
    elif op == "noalloc":
        m, n, rowptr, col, val = matrix(case["kind"], case["size"], seed)
        s.update(m=m, n=n, rowptr=rowptr, col=col, val=val.to(VT[case["dtype"]]), dtype=smat.DTYPES[case["dtype"]])
        s["x"] = _vector(n, seed, case["dtype"])
        s["b"] = _vector(m, seed + 1, case["dtype"]) if case["residual"] else None
        s["y"] = torch.empty(m, dtype=XT[case["dtype"]], device=DEV)
        s["alpha"] = np.array([-1.0 if case["residual"] else 1.0], np.float64 if case["dtype"] == "f64" else np.float32)
        s["beta"] = np.array([1.0 if case["residual"] else 0.0], s["alpha"].dtype)
    elif op == "many":
        s["mats"], s["xs"], s["ys"] = [], [], []
        for k, (kind, size, dtype) in enumerate(_many(case)):
            A = matrix(kind, size, seed * 31 + k // 2)
            s["mats"].append(_handle(A, dtype))
            s["xs"].append(_vector(A[1], seed * 31 + k, dtype))
            s["ys"].append(torch.empty(A[0], dtype=XT[dtype], device=DEV))
    elif op == "batch":
        mats, s["xs"], s["ys"] = [], [], []
        for k, (kind, size) in enumerate(_batch(case)):
            A = matrix(kind, size, seed * 31 + k)
            mats.append(_handle(A, case["dtype"]))
            s["xs"].append(_vector(A[1], seed * 31 + k, case["dtype"]))
            s["ys"].append(torch.empty(A[0], dtype=XT[case["dtype"]], device=DEV))
        s["batch"] = smat.Batch(mats)
        s["batch"].tune()
    elif op == "cg":
        A = _spd(_spd_shift(case))
        s["A64"], s["A32"] = _handle(A, "f64"), _handle(A, case["inner_dtype"])
        s["b"] = _vector(A[0], seed, "f64")
        s["x"] = torch.zeros(A[0], dtype=torch.float64, device=DEV)
        s["opts"] = {"rtol": 0.0, "max_outer": case["outer"], "max_inner": case["inner"], "inner_rtol": 0.0}
    elif op == "setup":
        m, n, rowptr, col, val = matrix(case["kind"], case["size"], seed)
        s.update(m=m, n=n, rowptr=rowptr, col=col, val=val.to(VT[case["dtype"]]), dtype=case["dtype"])
        s["x"] = _vector(n, seed, case["dtype"])
        s["variant"] = case["variant"]
    else:
        X, T = _samples(case, seed)
        start = torch.zeros(3, smat.SMAT_MLP_PARAMS, device=DEV)
        start[0] = _params()
        s.update(start=start, now=torch.empty_like(start), X=X, T=T, B=case["batch"], grad=torch.empty_like(start[0]),
                 loss=torch.empty(1, device=DEV), work=torch.empty(smat.smat_mlp_work_floats(case["batch"]), device=DEV))
    return s


def _params():
    """The trained selector's parameters: the model file's floats after its magic, version, mean and deviation."""
    return torch.from_numpy(np.fromfile(smat.MODEL_PATH, "<f4", offset=12)[24:]).to(DEV)


def _samples(case, seed):
    """Standardised features and soft targets that sum to one, as the training driver has them."""
    g = _gen(seed)
    X = torch.randn(case["batch"], 12, device=DEV, generator=g)
    T = torch.softmax(4.0 * torch.randn(case["batch"], 8, device=DEV, generator=g), 1)
    return X, T


def run(s):
    op = s["op"]
    if op == "spmv":
        if s["b"] is None:
            return s["M"].spmv(s["x"], s["y"])
        s["y"].copy_(s["b"])
        return s["M"].spmv(s["x"], s["y"], alpha=-1.0, beta=1.0)
    if op == "noalloc":
        if s["b"] is not None:
            s["y"].copy_(s["b"])
        st = smat.smat_spmv_csr_merge_noalloc(
            s["m"], s["n"], s["col"].numel(), s["rowptr"].data_ptr(), s["col"].data_ptr(), s["val"].data_ptr(), s["dtype"],
            s["alpha"].ctypes.data, s["x"].data_ptr(), s["beta"].ctypes.data, s["y"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        if st != smat.SMAT_OK:
            raise smat.SmatError(st, "smat_spmv_csr_merge_noalloc")
        return s["y"]
    if op == "many":
        return smat.spmv_many(s["mats"], s["xs"], s["ys"])
    if op == "batch":
        return s["batch"].spmv(s["xs"], s["ys"])
    if op == "cg":
        s["x"].zero_()
        info = smat.cg_mixed(s["A64"], s["A32"], s["b"], s["x"], **s["opts"])
        return {"x": s["x"], "outer": info["outer"], "inner": info["inner_total"]}
    if op == "setup":
        M = smat.SpMatrix(s["m"], s["n"], s["rowptr"], s["col"], s["val"], s["dtype"])
        if s["variant"] == "learned":   # the selector's own pick, with no timed trials
            M.tune("learned", conf_threshold=0.0, trial_extended=0)
        else:
            M.tune("fixed", variant=smat.VARIANT_NAMES.index(s["variant"]))
        y = M.spmv(s["x"])
        f = M.features()
        out = {"y": y, "variant": M.plan()["variant"],
               "features": [f[k] for k in ("max_rd", "min_rd", "empty_rows", "ndiags", "ntdiags", "s2")]}
        M.close()
        return out
    s["now"].copy_(s["start"])
    p, m, v = s["now"]
    stream = torch.cuda.current_stream().cuda_stream
    st = smat.smat_mlp_loss_grad(p.data_ptr(), s["X"].data_ptr(), s["T"].data_ptr(), s["B"], s["grad"].data_ptr(),
                                 s["loss"].data_ptr(), s["work"].data_ptr(), stream)
    st = st or smat.smat_mlp_adam(p.data_ptr(), s["grad"].data_ptr(), m.data_ptr(), v.data_ptr(), p.numel(), 1, 3e-3, 0.9,
                                  0.999, 1e-8, stream)
    if st != smat.SMAT_OK:
        raise smat.SmatError(st, "training step")
    return {"grad": s["grad"], "loss": s["loss"], "state": s["now"]}


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------

def _sizes(kind, size):
    """Rows and (expected) stored entries."""
    if kind == "grid2d":
        return size * size, 5 * size * size - 4 * size
    if kind == "grid3d":
        return size ** 3, 7 * size ** 3 - 6 * size ** 2
    if kind in ("box", "grid27"):
        r = 2 if kind == "box" else 1
        side = (2 * r + 1) * size - r * (r + 1)
        return size ** 3, side ** 3
    if kind == "blocks":
        return size, size // 8 * 64 + (size % 8) ** 2
    if kind == "uniform":
        return size, 16 * size
    cdf = _zipf_cdf(min(CAP, size))
    return size, int(size * (len(cdf) - cdf[:-1].sum()))


def _product(kind, size, dtype, residual=False):
    """Values, the column indices that no rule gives (random graphs), x and y."""
    m, nnz = _sizes(kind, size)
    t = 8 if dtype == "f64" else 4
    index = 4 * nnz + 4 * m if kind in ("uniform", "powerlaw") else 0
    return nnz * ESZ[dtype] + index + m * t * (3 if residual else 2), 2 * nnz


def work(case):
    op = case["op"]
    if op == "spmv":
        b, f = _product(case["kind"], case["size"], case["dtype"], case["residual"])
    elif op == "noalloc":
        m, nnz = _sizes(case["kind"], case["size"])
        b, f = _product(case["kind"], case["size"], case["dtype"], case["residual"])
        if case["kind"] not in ("uniform", "powerlaw"):
            b += 4 * nnz + 4 * m        # the caller's CSR arrays are what there is
    elif op == "many":
        b, f = map(sum, zip(*[_product(*c) for c in _many(case)]))
    elif op == "batch":
        b, f = map(sum, zip(*[_product(k, n, case["dtype"]) for k, n in _batch(case)]))
    elif op == "cg":
        n, nnz = _sizes("grid3d", case["size"])
        inner, outer = case["inner"] * case["outer"], case["outer"] + 1
        # inner: the values, p and d and the residual read and written; outer: the values, x, b and r
        b = inner * (nnz * ESZ[case["inner_dtype"]] + 6 * 4 * n) + outer * (nnz * 8 + 4 * 8 * n)
        f = inner * (2 * nnz + 10 * n) + outer * (2 * nnz + 4 * n)
    elif op == "setup":
        m, nnz = _sizes(case["kind"], case["size"])
        csr = nnz * (4 + ESZ[case["dtype"]]) + 4 * m
        p, f = _product(case["kind"], case["size"], case["dtype"])
        b = 2 * csr + p                 # the matrix in, the library's own copy of it, the product
    else:
        n = smat.SMAT_MLP_PARAMS
        b = 4 * (case["batch"] * 20 + n * 7)
        f = case["batch"] * 6 * (12 * 64 + 64 * 64 + 64 * 8) + 12 * n
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# exact: the same results in 64 bits, without the library
# ---------------------------------------------------------------------------

def _exact_product(A, dtype, x):
    """Each row's sum in pieces of 64 entries, then the pieces."""
    m, n, rowptr, col, val = A
    val = val.to(VT[dtype]).double()
    length = (rowptr[1:] - rowptr[:-1]).long()
    pieces = (length + 63) // 64
    first = torch.cumsum(pieces, 0) - pieces
    row = torch.repeat_interleave(torch.arange(m, device=DEV), length)
    at = torch.arange(col.numel(), device=DEV) - rowptr.long()[row]
    part = torch.zeros(int(pieces.sum()), dtype=torch.float64, device=DEV)
    part.index_add_(0, first[row] + at // 64, val * x.double()[col.long()])
    y = torch.zeros(m, dtype=torch.float64, device=DEV)
    return y.index_add_(0, torch.repeat_interleave(torch.arange(m, device=DEV), pieces), part)


def _exact_solve(A, b):
    """CG in 64 bits, restarted from the true residual until it no longer falls."""
    m, n, rowptr, col, val = A
    S = torch.sparse_csr_tensor(rowptr, col, val, (m, n))
    x = torch.zeros_like(b)
    for _ in range(3):
        r = b - S @ x
        p, rho, rho0 = r.clone(), r @ r, r @ r
        for _ in range(200):
            q = S @ p
            a = rho / (p @ q)
            x += a * p
            r -= a * q
            new = r @ r
            p = r + (new / rho) * p
            rho = new
            if float(rho) <= 1e-26 * float(rho0):
                break
    return x


def _exact_step(case, seed):
    params = _params().double().requires_grad_(True)
    X, T = (t.double() for t in _samples(case, seed))
    cut = torch.split(params, [768, 64, 4096, 64, 512, 8])
    h = torch.relu(X @ cut[0].view(64, 12).T + cut[1])
    h = torch.relu(h @ cut[2].view(64, 64).T + cut[3])
    z = h @ cut[4].view(8, 64).T + cut[5]
    loss = -(T * torch.log_softmax(z, 1)).sum() / case["batch"]
    g, = torch.autograd.grad(loss, params)
    m, v = 0.1 * g, 0.001 * g * g
    p = params.detach() - 3e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"grad": g, "loss": loss.detach().reshape(1), "state": torch.stack([p, m, v])}


def exact(case, seed):
    op = case["op"]
    if op in ("spmv", "noalloc"):
        A = matrix(case["kind"], case["size"], seed)
        y = _exact_product(A, case["dtype"], _vector(A[1], seed, case["dtype"]))
        return _vector(A[0], seed + 1, case["dtype"]).double() - y if case["residual"] else y
    if op == "many":
        got = []
        for k, (kind, size, dtype) in enumerate(_many(case)):
            A = matrix(kind, size, seed * 31 + k // 2)
            got.append(_exact_product(A, dtype, _vector(A[1], seed * 31 + k, dtype)))
        return got
    if op == "batch":
        got = []
        for k, (kind, size) in enumerate(_batch(case)):
            A = matrix(kind, size, seed * 31 + k)
            got.append(_exact_product(A, case["dtype"], _vector(A[1], seed * 31 + k, case["dtype"])))
        return got
    if op == "cg":
        A = _spd(_spd_shift(case))
        return {"x": _exact_solve(A, _vector(A[0], seed, "f64")), "outer": None, "inner": None}
    if op == "setup":
        A = matrix(case["kind"], case["size"], seed)
        return {"y": _exact_product(A, case["dtype"], _vector(A[1], seed, case["dtype"])), "variant": None,
                "features": None}
    return _exact_step(case, seed)
