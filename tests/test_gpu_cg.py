"""Mixed-precision CG: FP32/BF16 inner solves, FP64 residual and update.
The final residual is recomputed on the host by the oracle's FP64 SpMV."""
import contextlib
import ctypes
import threading
import time

import numpy as np
import pytest

import oracle
import paper_1210_2536_gb300 as smat
from paper_1210_2536_gb300 import synth
from helpers import stored_values

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def handles(A, inner="f32", tune=True):
    def mk(dt):
        vals, _ = stored_values(A, dt)
        if dt == "bf16":
            vals = vals.view(np.int16)
        M = smat.SpMatrix(A.m, A.n, A.rowptr, A.colidx, np.ascontiguousarray(vals), dt)
        if tune:
            M.tune("exhaustive", trial_reps=3)
        return M
    return mk("f64"), mk(inner)


def oracle_relres(A, x, b):
    r = b - oracle.spmv_csr(A.m, A.rowptr, A.colidx, A.val, x, threads=8)
    return float(np.linalg.norm(r) / np.linalg.norm(b))


@pytest.mark.parametrize("maker,inner", [(lambda: synth.poisson_2d_64(), "f32"),
                                         (lambda: synth.stencil3d7(20), "bf16"),
                                         (lambda: synth.stencil3d7(32), "f32")])
def test_cg_reaches_fp64_residual(maker, inner):
    A = maker()
    x_true = synth.uniform(0, 5, A.n)
    b = oracle.spmv_csr(A.m, A.rowptr, A.colidx, A.val, x_true, threads=8)
    A64, A32 = handles(A, inner)
    bd = torch.from_numpy(b).to(DEV)
    xd = torch.zeros(A.n, dtype=torch.float64, device=DEV)
    info = smat.cg_mixed(A64, A32, bd, xd, rtol=1e-10, max_inner=2000)
    assert info["converged"] and info["status"] == smat.SMAT_OK, info
    x = xd.cpu().numpy()
    rr = oracle_relres(A, x, b)
    assert rr <= 1e-10, rr
    assert abs(rr - info["relres"]) <= 0.05 * rr + 1e-16
    assert info["outer"] >= 2  # FP32 alone cannot reach 1e-10: refinement did the rest
    A64.close(), A32.close()


def test_graph_and_plain_launches_agree_bitwise():
    A = synth.stencil3d7(16)
    b = oracle.spmv_csr(A.m, A.rowptr, A.colidx, A.val, synth.uniform(1, 5, A.n))
    A64, A32 = handles(A, "f32")
    bd = torch.from_numpy(b).to(DEV)
    out = []
    for g in (1, 0):
        xd = torch.zeros(A.n, dtype=torch.float64, device=DEV)
        info = smat.cg_mixed(A64, A32, bd, xd, use_graph=g, rtol=1e-11)
        out.append((xd.cpu().numpy(), info["inner_total"]))
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][0].view(np.uint64), out[1][0].view(np.uint64))


def test_limits_and_degenerate_cases():
    A = synth.poisson_2d_64()
    b = oracle.spmv_csr(A.m, A.rowptr, A.colidx, A.val, synth.uniform(2, 5, A.n))
    A64, A32 = handles(A, "f32", tune=False)
    bd = torch.from_numpy(b).to(DEV)
    xd = torch.zeros(A.n, dtype=torch.float64, device=DEV)
    info = smat.cg_mixed(A64, A32, bd, xd, max_total_inner=5)
    assert info["status"] == smat.SMAT_ERR_NOT_CONVERGED and info["inner_total"] <= 5 and not info["converged"]
    # b = 0: x = 0 is returned at once
    xd.fill_(3.0)
    info = smat.cg_mixed(A64, A32, torch.zeros_like(bd), xd)
    assert info["converged"] and torch.count_nonzero(xd).item() == 0
    # an FP64 handle cannot be the inner operator
    st, _ = smat.smat_cg_mixed(A64.h, A64.h, bd.data_ptr(), xd.data_ptr(), None, 0)
    assert st == smat.SMAT_ERR_INVALID_ARG
    R = synth.CSR(3, 4, np.array([0, 1, 2, 3], np.int32), np.array([0, 1, 2], np.int32), np.ones(3))
    N64 = smat.SpMatrix(3, 4, R.rowptr, R.colidx, R.val, "f64")
    N32 = smat.SpMatrix(3, 4, R.rowptr, R.colidx, R.val.astype(np.float32), "f32")
    st, _ = smat.smat_cg_mixed(N64.h, N32.h, bd.data_ptr(), xd.data_ptr(), None, 0)
    assert st == smat.SMAT_ERR_INVALID_ARG
    for M in (A64, A32, N64, N32):
        M.close()


@pytest.mark.parametrize("n", [1, 3, 4095, 4097, 32767, 32769, 65539, 622592, 622595, 1400001])
def test_vector_kernel_sizes(n):
    """The vector kernel's launch shapes (one CTA, one cluster, registers over
    the whole GPU, streaming) at their edges and with n % 4 != 0, on
    tridiag(-1, 4, -1): eigenvalues in (2, 6), so a relative residual of
    1e-12 bounds the relative error by 3e-12 (plus rounding)."""
    i = np.arange(n)
    cols = np.stack([i - 1, i, i + 1], 1)
    ok = (cols >= 0) & (cols < n)
    val = np.broadcast_to(np.array([-1.0, 4.0, -1.0]), (n, 3))[ok].copy()
    rowptr = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    A = synth.CSR(n, n, rowptr, cols[ok].astype(np.int32), val)
    x_true = synth.uniform(3, 5, n)
    b = oracle.spmv_csr(n, A.rowptr, A.colidx, A.val, x_true, threads=8)
    A64, A32 = handles(A, tune=False)
    xd = torch.zeros(n, dtype=torch.float64, device=DEV)
    info = smat.cg_mixed(A64, A32, torch.from_numpy(b).to(DEV), xd, rtol=1e-12)
    assert info["converged"], info
    err = np.linalg.norm(xd.cpu().numpy() - x_true) / np.linalg.norm(x_true)
    assert err <= 4e-12, err
    A64.close(), A32.close()


def tridiagonal(n):
    i = np.arange(n)
    cols = np.stack([i - 1, i, i + 1], 1)
    ok = (cols >= 0) & (cols < n)
    val = np.broadcast_to(np.array([-1.0, 4.0, -1.0]), (n, 3))[ok].copy()
    rowptr = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    return synth.CSR(n, n, rowptr, cols[ok].astype(np.int32), val)


@pytest.mark.parametrize("graph", [1, 0])
@pytest.mark.parametrize("n", [40000, 1400001])
def test_grid_barriers_that_run_out_end_the_solve(n, graph):
    # the test hook keeps every grid barrier from being passed (vectors in
    # registers, and streamed).  The first waits for 6e8 cycles (0.3 s); the
    # other 39 of the chunk half a millisecond each, 20 ms in all, where they
    # would take 12 s if each waited for its limit.
    A = tridiagonal(n)
    b = oracle.spmv_csr(n, A.rowptr, A.colidx, A.val, synth.uniform(3, 5, n), threads=8)
    A64, A32 = handles(A, tune=False)
    bd = torch.from_numpy(b).to(DEV)
    xd = torch.zeros(n, dtype=torch.float64, device=DEV)
    opts = dict(rtol=1e-12, check_every=20, use_graph=graph)
    assert smat.cg_mixed(A64, A32, bd, xd, **opts)["converged"]
    good = xd.clone()
    xd.fill_(1.0)
    smat.lib().smat_test_stall_pipelines(1, 600_000_000)
    try:
        t0 = time.monotonic()
        with pytest.raises(smat.SmatError) as e:
            smat.cg_mixed(A64, A32, bd, xd, **opts)
        assert e.value.status == smat.SMAT_ERR_CUDA and time.monotonic() - t0 < 4.0
    finally:
        smat.lib().smat_test_stall_pipelines(0, 0)
    assert bool((xd == 1.0).all())            # no refinement step was taken
    xd.zero_()
    assert smat.cg_mixed(A64, A32, bd, xd, **opts)["converged"]
    assert torch.equal(xd, good)              # the context is usable, the solve reproducible
    A64.close(), A32.close()


@contextlib.contextmanager
def part_of_the_sms(count):
    """A green context of about `count` SMs, current inside the block."""
    cu = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        st = getattr(cu, name)(*args)
        assert st == 0, (name, st)

    torch.cuda.current_stream().synchronize()
    dev, groups = ctypes.c_int(), ctypes.c_uint(1)
    whole, part, rest = (ctypes.create_string_buffer(512) for _ in range(3))   # CUdevResource
    desc, green, ctx, old = (ctypes.c_void_p() for _ in range(4))
    call("cuDeviceGet", ctypes.byref(dev), 0)
    call("cuDeviceGetDevResource", dev, whole, 1)                              # CU_DEV_RESOURCE_TYPE_SM
    call("cuDevSmResourceSplitByCount", part, ctypes.byref(groups), whole, rest, 0, count)
    call("cuDevResourceGenerateDesc", ctypes.byref(desc), part, 1)
    call("cuGreenCtxCreate", ctypes.byref(green), desc, dev, 1)                # CU_GREEN_CTX_DEFAULT_STREAM
    call("cuCtxFromGreenCtx", ctypes.byref(ctx), green)
    call("cuCtxPushCurrent_v2", ctx)
    try:
        yield
    finally:
        call("cuCtxSynchronize")
        call("cuCtxPopCurrent_v2", ctypes.byref(old))
        call("cuGreenCtxDestroy", green)


@pytest.mark.parametrize("n", [20000, 40000, 1400001])
def test_context_with_part_of_the_sms(n):
    # the vector kernel waits for all of its CTAs: no more than the context's
    # SMs hold at once
    A = tridiagonal(n)
    x_true = synth.uniform(3, 5, n)
    b = oracle.spmv_csr(n, A.rowptr, A.colidx, A.val, x_true, threads=8)
    A64, A32 = handles(A, tune=False)
    bd = torch.from_numpy(b).to(DEV)
    xd = torch.zeros(n, dtype=torch.float64, device=DEV)
    with part_of_the_sms(16):
        info = smat.cg_mixed(A64, A32, bd, xd, stream=0, rtol=1e-12)
    assert info["converged"], info
    err = np.linalg.norm(xd.cpu().numpy() - x_true) / np.linalg.norm(x_true)
    assert err <= 4e-12, err
    A64.close(), A32.close()


def test_solves_on_several_threads():
    # each solve captures its iterations and frees its workspace, which waits
    # for the device: CUDA allows no such wait while another thread captures
    n, reps = 60000, 10
    A = tridiagonal(n)
    b = oracle.spmv_csr(n, A.rowptr, A.colidx, A.val, synth.uniform(3, 5, n), threads=8)
    bd = torch.from_numpy(b).to(DEV)
    pairs = [handles(A, tune=False) for _ in range(4)]
    xs = [[torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(reps)] for _ in pairs]
    first = torch.zeros(n, dtype=torch.float64, device=DEV)
    assert smat.cg_mixed(*pairs[0], bd, first, stream=0, rtol=1e-12)["converged"]
    torch.cuda.synchronize()
    status = [[] for _ in pairs]

    def work(k):
        for x in xs[k]:
            st, info = smat.smat_cg_mixed(pairs[k][0].h, pairs[k][1].h, bd.data_ptr(), x.data_ptr(), opts, 0)
            status[k].append(st)

    opts = smat.smat_cg_opts_default()
    opts.rtol = 1e-12
    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(pairs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert status == [[smat.SMAT_OK] * reps] * len(pairs), status
    assert all(torch.equal(x, first) for row in xs for x in row)
    for A64, A32 in pairs:
        A64.close(), A32.close()


def arrow(n):
    """A symmetric, diagonally dominant matrix with one full row and column."""
    i = np.arange(1, n)
    r = np.concatenate([[0], i, np.zeros(n - 1, int), i, i[1:], i[:-1]])
    c = np.concatenate([[0], i, i, np.zeros(n - 1, int), i[:-1], i[1:]])
    v = np.concatenate([np.full(n, 4.0), np.full(2 * (n - 1), -1e-3), np.full(2 * (n - 2), -1.0)])
    o = np.lexsort((c, r))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return synth.CSR(n, n, rowptr.astype(np.int32), c[o].astype(np.int32), v[o])


@pytest.mark.parametrize("variant", ["CSR_MERGE", "COO", "HYB", "SPLIT"])
def test_inner_plans_with_carries_on_a_handle_in_use(variant):
    # the inner handle's carries belong to the caller's stream already; the
    # solve's own stream needs some of its own before it captures, and leaves
    # none behind
    A = arrow(3000)
    x_true = synth.uniform(4, 5, A.n)
    b = oracle.spmv_csr(A.m, A.rowptr, A.colidx, A.val, x_true, threads=8)
    bd = torch.from_numpy(b).to(DEV)
    A64, A32 = handles(A, tune=False)
    for M in (A64, A32):
        M.tune("fixed", variant=getattr(smat, "SMAT_V_" + variant))
    x32 = torch.from_numpy(x_true.astype(np.float32)).to(DEV)
    before = A32.spmv(x32)
    A64.spmv(bd)
    for solve in range(3):
        xd = torch.zeros(A.n, dtype=torch.float64, device=DEV)
        info = smat.cg_mixed(A64, A32, bd, xd, rtol=1e-11, use_graph=int(solve < 2))
        assert info["converged"], info
        assert oracle_relres(A, xd.cpu().numpy(), b) <= 1.1e-11
    assert torch.equal(A32.spmv(x32), before)
    A64.close(), A32.close()
