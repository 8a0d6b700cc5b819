"""COO, SPLIT and HYB products and their exported row indices, at the edges of
the 256-entry tiles, the staged sums (32 or 64 per warp) and the carries:
rows of one entry (256 ends in a tile), rows that end on a tile's last entry,
rows of many tiles, empty rows between, one tile only.  Against the oracle."""
import numpy as np
import pytest

import paper_1210_2536_gb300 as smat
from paper_1210_2536_gb300 import synth
from helpers import TOL, assert_close_rows, reference, stored_values

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rows(lengths, n, seed):
    rng = np.random.default_rng(seed)
    L = np.asarray(lengths, np.int64)
    rp = np.concatenate([[0], np.cumsum(L)])
    step = np.maximum(n // np.maximum(L, 1), 1)
    start = (rng.random(L.size) * (n - (L - 1).clip(0) * step)).astype(np.int64)
    row = np.repeat(np.arange(L.size), L)
    col = start[row] + (np.arange(rp[-1]) - rp[row]) * step[row]
    return synth.CSR(L.size, n, rp.astype(np.int32), col.astype(np.int32), rng.standard_normal(int(rp[-1])))


CASES = {
    "one_entry": [1], "one_tile": [100, 156], "tile_plus_one": [256, 1], "ones": [1] * 1000,
    "around_32_and_64_ends": [8] * 32 + [7] * 33 + [4] * 64 + [3] * 90 + [2] * 200,
    "ends_on_tiles": [256, 512, 255, 1, 128, 128, 768], "empty_between": [0, 0, 5, 0, 300, 0, 0, 1, 0] * 60,
    "many_tiles": [3, 256 * 40, 9, 0, 256 * 140 + 3, 5] + [2] * 50,
    "long_and_short": [1500, 3, 0, 9000, 20, 1] + [5] * 400 + [1024, 1023, 7],
}


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_products_and_exports(name, dtype):
    A = _rows(CASES[name], 40000, 11)
    vals, vals64 = stored_values(A, dtype)
    vals = np.ascontiguousarray(vals.view(np.int16) if dtype == "bf16" else vals)
    np_t = np.float64 if dtype == "f64" else np.float32
    M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, vals, dtype)
    M.tune("fixed", variant=smat.SMAT_V_CSR_SCALAR, keep_formats=1, fill_ratio_max=100000, bytes_cap=1e9)
    row = A.row_of_nnz()
    x = synth.uniform(1, 1, A.n).astype(np_t)
    xd = torch.from_numpy(x).to(DEV)
    built = 0
    for v, fmt in ((smat.SMAT_V_COO, smat.SMAT_FMT_COO), (smat.SMAT_V_SPLIT, smat.SMAT_FMT_SPLIT),
                   (smat.SMAT_V_HYB, smat.SMAT_FMT_HYB)):
        try:
            M.convert(fmt)
        except smat.SmatError as e:
            assert e.status == smat.SMAT_ERR_UNSUPPORTED and v != smat.SMAT_V_COO
            continue
        built += 1
        for alpha, beta in ((1.0, 0.0), (-2.0, 0.0), (-1.0, 1.0)):
            y0 = synth.uniform(2, 1, A.m).astype(np_t)
            y = torch.from_numpy(np.full_like(y0, np.nan) if beta == 0 else y0.copy()).to(DEV)
            M.spmv(xd, y, alpha, beta, variant=v)
            ref, scale = reference(A, vals64, x, alpha, beta, y0 if beta != 0 else None)
            assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} {v} {alpha} {beta}")
        if fmt == smat.SMAT_FMT_COO:
            assert np.array_equal(M.export(fmt)[0], row)
        else:
            p = M.export_parts(fmt)
            got = p["srow"] if fmt == smat.SMAT_FMT_SPLIT else p["coo_row"]
            length = np.diff(A.rowptr)[row]
            at = np.arange(A.nnz) - A.rowptr[row]
            keep = length < 1024 if fmt == smat.SMAT_FMT_SPLIT else at >= p["K"]
            assert np.array_equal(got, row[keep])
    assert built >= 1
    M.close()


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_every_row_takes_beta_once(name, dtype):
    # beta other than 0 and 1: a row written twice, or not at all, shows
    A = _rows(CASES[name], 40000, 11)
    vals, vals64 = stored_values(A, dtype)
    vals = np.ascontiguousarray(vals.view(np.int16) if dtype == "bf16" else vals)
    np_t = np.float64 if dtype == "f64" else np.float32
    M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, vals, dtype)
    M.tune("fixed", variant=smat.SMAT_V_CSR_SCALAR, keep_formats=1, fill_ratio_max=100000, bytes_cap=1e9)
    x = synth.uniform(1, 1, A.n).astype(np_t)
    y0 = synth.uniform(2, 1, A.m).astype(np_t)
    xd = torch.from_numpy(x).to(DEV)
    for v, fmt in ((smat.SMAT_V_COO, smat.SMAT_FMT_COO), (smat.SMAT_V_SPLIT, smat.SMAT_FMT_SPLIT),
                   (smat.SMAT_V_HYB, smat.SMAT_FMT_HYB)):
        try:
            M.convert(fmt)
        except smat.SmatError as e:
            assert e.status == smat.SMAT_ERR_UNSUPPORTED and v != smat.SMAT_V_COO
            continue
        for alpha, beta in ((2.0, -0.5), (1.0, 2.0), (1.5, -0.75)):
            y = torch.from_numpy(y0.copy()).to(DEV)
            M.spmv(xd, y, alpha, beta, variant=v)
            ref, scale = reference(A, vals64, x, alpha, beta, y0)
            assert_close_rows(y.cpu().numpy().astype(np.float64), ref, scale, TOL[dtype], f"{name} {v} {alpha} {beta}")
    M.close()
