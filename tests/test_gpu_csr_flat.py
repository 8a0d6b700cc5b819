"""CSR split evenly by stored entries (SMAT_V_CSR_MERGE and the product that
allocates nothing), at the edges of its chunks, tiles and rules: rows of many
tiles, runs of empty rows longer than a warp writes itself, ragged ends,
pointers without 32-byte alignment, several chunks per tile.  Against the
oracle, within the per-row bars the parity tests use."""
import ctypes

import numpy as np
import pytest

import paper_1210_2536_gb300 as smat
from paper_1210_2536_gb300 import synth
from helpers import TOL, assert_close_rows, reference, stored_values

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rows(lengths, n, seed):
    """Rows of the given lengths, columns evenly strided from a random start."""
    rng = np.random.default_rng(seed)
    L = np.asarray(lengths, np.int64)
    rp = np.concatenate([[0], np.cumsum(L)])
    step = np.maximum(n // np.maximum(L, 1), 1)
    start = (rng.random(L.size) * (n - (L - 1).clip(0) * step)).astype(np.int64)
    row = np.repeat(np.arange(L.size), L)
    col = start[row] + (np.arange(rp[-1]) - rp[row]) * step[row]
    return synth.CSR(L.size, n, rp.astype(np.int32), col.astype(np.int32), rng.standard_normal(int(rp[-1])))


def _cases():
    ones = np.ones(4000, int)
    yield "one_entry", _rows([1], 7, 0)
    yield "no_entries", _rows([0] * 5000, 7, 0)
    yield "chunk_edges", _rows([255, 1, 256, 257, 511, 1, 2, 3], 600, 1)
    yield "one_row_of_many_tiles", _rows([3, 40000, 5], 50000, 2)        # 157 carries of one row
    yield "rows_of_33_and_129_tiles", _rows([7, 33 * 256, 129 * 256 - 7, 0, 9], 40000, 3)
    yield "empty_ends", _rows([0] * 70 + [9] * 300 + [0] * 90, 900, 4)
    gap = np.concatenate([ones, np.zeros(4097 * 3, int), ones, np.zeros(200, int), [700], np.zeros(9000, int)])
    yield "gaps_past_the_warp_s_own", _rows(gap, 1000, 5)                # FLAT_MAX_ROWS + 1 and more
    yield "gap_at_the_limit", _rows(np.concatenate([[256], np.zeros(4095, int), [256, 0, 0]]), 1000, 6)
    yield "ragged_mix", _rows(np.random.default_rng(7).integers(0, 90, 5003), 4999, 7)


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name,A", list(_cases()), ids=[k for k, _ in _cases()])
def test_edges(name, A, dtype):
    vals, vals64 = stored_values(A, dtype)
    vals = np.ascontiguousarray(vals.view(np.int16) if dtype == "bf16" else vals)
    np_t = np.float64 if dtype == "f64" else np.float32
    ct = ctypes.c_double if dtype == "f64" else ctypes.c_float
    x = synth.uniform(1, 1, A.n).astype(np_t)
    xd = torch.from_numpy(x).to(DEV)
    M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, vals, dtype)
    rp = torch.from_numpy(A.rowptr).to(DEV)
    # columns and values of the allocation-free call: 32-byte aligned, and not
    arrays = []
    for off in (0, 1):
        ci = torch.zeros(A.nnz + 1 + off, dtype=torch.int32, device=DEV)[off:][:A.nnz + 1]
        vv = torch.zeros(A.nnz + 1 + off, dtype=torch.from_numpy(vals).dtype, device=DEV)[off:][:A.nnz + 1]
        ci[:A.nnz] = torch.from_numpy(A.colidx)
        vv[:A.nnz] = torch.from_numpy(vals)
        arrays.append((ci, vv))
    for alpha, beta in ((1.0, 0.0), (-2.0, 0.0), (-1.0, 1.0)):
        y0 = synth.uniform(2, 1, A.m).astype(np_t)
        start = np.full_like(y0, np.nan) if beta == 0 else y0
        ref, scale = reference(A, vals64, x, alpha, beta, y0 if beta != 0 else None)
        y = torch.from_numpy(start.copy()).to(DEV)
        M.spmv(xd, y, alpha, beta, variant=smat.SMAT_V_CSR_MERGE)
        assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} handle {alpha} {beta}")
        a, b = ct(alpha), ct(beta)
        for ci, vv in arrays:
            y = torch.from_numpy(start.copy()).to(DEV)
            st = smat.smat_spmv_csr_merge_noalloc(A.m, A.n, A.nnz, rp.data_ptr(), ci.data_ptr(), vv.data_ptr(),
                                                  smat.DTYPES[dtype], ctypes.addressof(a), xd.data_ptr(),
                                                  ctypes.addressof(b), y.data_ptr(),
                                                  torch.cuda.current_stream().cuda_stream)
            assert st == smat.SMAT_OK
            assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype],
                              f"{name} noalloc {alpha} {beta}")
    M.close()


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name,A", list(_cases()), ids=[k for k, _ in _cases()])
def test_every_row_takes_beta_once(name, A, dtype):
    # beta other than 0 and 1: a row written twice, or not at all, shows.  The
    # gaps case joins tiles of more than FLAT_MAX_ROWS rows with tiles that
    # hold short runs of empty rows.
    vals, vals64 = stored_values(A, dtype)
    vals = np.ascontiguousarray(vals.view(np.int16) if dtype == "bf16" else vals)
    np_t = np.float64 if dtype == "f64" else np.float32
    ct = ctypes.c_double if dtype == "f64" else ctypes.c_float
    x = synth.uniform(1, 1, A.n).astype(np_t)
    y0 = synth.uniform(2, 1, A.m).astype(np_t)
    xd, rp, ci, vv = (torch.from_numpy(t).to(DEV) for t in (x, A.rowptr, A.colidx, vals))
    M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, vals, dtype)
    N = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, vals, dtype)
    N.tune("fixed", variant=smat.SMAT_V_CSR_MERGE)
    for alpha, beta in ((2.0, -0.5), (1.0, 2.0), (1.5, -0.75)):
        ref, scale = reference(A, vals64, x, alpha, beta, y0)
        y = torch.from_numpy(y0.copy()).to(DEV)
        M.spmv(xd, y, alpha, beta, variant=smat.SMAT_V_CSR_MERGE)
        assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} {alpha} {beta}")
        y = torch.from_numpy(y0.copy()).to(DEV)
        N.spmv(xd, y, alpha, beta)
        assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} plan {alpha} {beta}")
        y = torch.from_numpy(y0.copy()).to(DEV)
        a, b = ct(alpha), ct(beta)
        st = smat.smat_spmv_csr_merge_noalloc(A.m, A.n, A.nnz, rp.data_ptr(), ci.data_ptr(), vv.data_ptr(),
                                              smat.DTYPES[dtype], ctypes.addressof(a), xd.data_ptr(),
                                              ctypes.addressof(b), y.data_ptr(),
                                              torch.cuda.current_stream().cuda_stream)
        assert st == smat.SMAT_OK
        assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} noalloc {alpha} {beta}")
    M.close(), N.close()


@pytest.mark.parametrize("name", ["gaps_past_the_warp_s_own", "ragged_mix"])
def test_first_product_while_capturing(name):
    # a relaxed capture may hold a handle's first CSR_MERGE product: what the
    # kernel needs to know of the rows is found beside the capture
    A = dict(_cases())[name]
    M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, A.val, "f64")
    x, y0 = synth.uniform(1, 1, A.n), synth.uniform(2, 1, A.m)
    xd, y = (torch.from_numpy(t).to(DEV) for t in (x, y0.copy()))
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        M.spmv(xd, y, 2.0, -0.5, variant=smat.SMAT_V_CSR_MERGE, stream=s)
    g.replay()
    torch.cuda.synchronize()
    ref, scale = reference(A, A.val, x, 2.0, -0.5, y0)
    assert_close_rows(y.cpu().numpy(), ref, scale, TOL["f64"], name)
    M.close()


def test_noalloc_several_chunks_per_tile():
    # 65536 tiles of one chunk hold 16.8 M entries: this matrix takes two per
    # tile, with rows that cross chunks and tiles
    A = _rows(np.tile([1, 300, 0, 17, 900, 2], 15000), 100000, 8)
    assert A.nnz > 65536 * 256
    x = synth.uniform(1, 1, A.n).astype(np.float32)
    vals = A.val.astype(np.float32)
    rp, ci, vv, xd = (torch.from_numpy(t).to(DEV) for t in (A.rowptr, A.colidx, vals, x))
    y = torch.full((A.m,), float("nan"), device=DEV)
    a, b = ctypes.c_float(1.0), ctypes.c_float(0.0)
    assert smat.smat_spmv_csr_merge_noalloc(A.m, A.n, A.nnz, rp.data_ptr(), ci.data_ptr(), vv.data_ptr(), smat.SMAT_F32,
                                            ctypes.addressof(a), xd.data_ptr(), ctypes.addressof(b), y.data_ptr(),
                                            torch.cuda.current_stream().cuda_stream) == smat.SMAT_OK
    ref, scale = reference(A, vals.astype(np.float64), x, 1.0, 0.0, None)
    assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL["f32"], "two chunks per tile")
