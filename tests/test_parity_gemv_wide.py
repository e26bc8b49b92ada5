"""GPU parity of the dense products taken by sets of rows (few long rows, rows that
start at other offsets than x), by a thread per rows (column-major, very many rows)
and by windows shifted per column (column-major, columns off 16 bytes), against the
FP64 oracle: remainders of the 16-byte packs, every offset of A and x, the last
incomplete set, column splits, alpha / beta."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from checks import (assert_canary, assert_normwise_scaled, assert_reduced_sum, canary_buffer, host)

pytestmark = pytest.mark.gpu
STORAGES = ["f32", "f64", "bf16", "f16"]


def lak():
    import paper_1409_0669_gb300 as m
    return m


def off(t, k, pad):
    """The same values starting k elements into a buffer, NaN around them."""
    buf = torch.full((t.numel() + k + pad,), float("nan"), dtype=t.dtype)
    buf[k:k + t.numel()] = t
    return buf.cuda()[k:k + t.numel()]


def check(y, ref, abs_ref, n, storage, what):
    if storage in ("f32", "f64"):
        assert_normwise_scaled(host(y), ref, abs_ref, storage, what)
    else:
        assert_reduced_sum(host(y), ref, abs_ref, np.full(ref.size, n), storage, what)


def run_case(storage, layout, m, n, pad, ka, kx, alpha=1.0, beta=0.0):
    lda = (n if layout == "row" else m) + pad
    rows = m if layout == "row" else n
    A = synth.normal(rows * lda, m * 7 + n, storage)
    x = synth.uniform(n, n, storage)
    used = A.view(rows, lda)[:, :lda - pad]
    vals = used.contiguous() if layout == "row" else used.t().contiguous()
    if pad:
        A.view(rows, lda)[:, lda - pad:] = float("nan")
    last = (rows - 1) * lda + lda - pad                # the buffer ends with the last entry
    dA, dx = off(A[:last], ka, 0), off(x, kx, 0)
    buf, y = canary_buffer(m, dA.dtype, dA.device)
    y0 = synth.uniform(m, 3, storage)
    y.copy_(y0) if beta != 0 else y.fill_(float("nan"))
    lak().dense_gemv(dA, dx, y=y, m=m, n=n, lda=lda, layout=layout, alpha=alpha, beta=beta)
    torch.cuda.synchronize()
    ref = alpha * oracle.gemv(vals, x, m, n, n, "row")
    ab = abs(alpha) * oracle.gemv(np.abs(oracle.widen(vals)), np.abs(oracle.widen(x)), m, n, n, "row")
    if beta != 0:
        ref = ref + beta * oracle.widen(y0)
        ab = ab + np.abs(beta * oracle.widen(y0))
    check(y, ref, ab, n + 2, storage, f"{layout} {m}x{n} lda={lda} A+{ka} x+{kx}")
    assert_canary(buf, m)
    return dA, dx, y


ROW_SHAPES = [(1, 32768), (3, 16385), (5, 40003), (30, 33000), (128, 16391), (9, 150001),
              (1537, 3071), (1601, 2050), (700, 6007)]


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("shape", ROW_SHAPES, ids=str)
@pytest.mark.parametrize("ka,kx,pad", [(0, 0, 0), (1, 0, 0), (0, 1, 3), (3, 6, 1), (0, 0, 8)])
def test_row_sets(storage, shape, ka, kx, pad):
    run_case(storage, "row", *shape, pad, ka, kx)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("kx", range(8))
def test_row_sets_every_x_offset(storage, kx):
    run_case(storage, "row", 6, 32775, 0, 2, kx, alpha=-1.5, beta=0.5)


@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_row_sets_splits_without_workspace_and_repeated(storage):
    """Split columns: bit-equal over calls; without a workspace the columns stay
    unsplit and the result stays within the tolerance."""
    lk = lak()
    m, n = 7, 300_001
    dA, dx, y = run_case(storage, "row", m, n, 0, 0, 0)
    assert lk.dense_gemv_workspace(m, n, "row", storage) > 0
    for _ in range(5):
        assert torch.equal(lk.dense_gemv(dA, dx, m=m, n=n, lda=n, layout="row"), y)
    from paper_1409_0669_gb300 import _native
    z = torch.empty_like(y)
    st = _native.load().dense_gemv(z.data_ptr(), dA.data_ptr(), dx.data_ptr(), m, n, n,
                                   _native.LAYOUTS["row"], _native.DTYPES[storage], None, 0, None,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    ab = oracle.gemv(np.abs(host(dA)), np.abs(host(dx)), m, n, n, "row")
    assert_normwise_scaled(host(z), host(y), ab, storage)


def test_row_sets_carry_nan_and_inf():
    m, n = 4, 40001
    A = torch.ones(m, n, device="cuda")
    x = torch.ones(n, device="cuda")
    A[1, 17], A[2, n - 1] = float("inf"), float("nan")
    y = lak().dense_gemv(A, x)
    assert y[0] == n and y[1] == float("inf") and torch.isnan(y[2]) and y[3] == n


COL_SHAPES = {"f32": [(33, 9001), (1001, 1003), (2047, 300)], "f64": [(2001, 703), (3000, 901)],
              "bf16": [(2001, 301), (2303, 777)], "f16": [(2001, 301), (2303, 777)]}


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("ka,pad", [(0, 0), (0, 1), (1, 0), (1, 3), (3, 2), (5, 7), (1, 8)])
def test_columns_off_alignment(storage, shape, ka, pad):
    """Every offset of the first column and every period of the following ones; the
    last rows' window past the matrix; columns split over blocks."""
    shapes = COL_SHAPES[storage]
    m, n = shapes[shape % len(shapes)]
    if shape == 1:
        run_case(storage, "col", m, n, pad, ka, 2, alpha=-0.5, beta=2.0)
    else:
        run_case(storage, "col", m, n, pad, ka, 0)


def test_columns_off_alignment_repeat_and_small_workspace():
    """Split columns: bit-equal over calls; a workspace too small for the splits falls
    back to the other kernel's needs, and is refused below those as before."""
    lk = lak()
    m, n = 3001, 5000
    A = synth.normal(m * n, 1, "f32").cuda()
    x = synth.uniform(n, 2, "f32").cuda()
    y = lk.dense_gemv(A, x, m=m, n=n, lda=m, layout="col")
    for _ in range(5):
        assert torch.equal(lk.dense_gemv(A, x, m=m, n=n, lda=m, layout="col"), y)
    with pytest.raises(lk.LakError, match="LAK_EWORKSPACE"):
        lk.dense_gemv(A, x, m=m, n=n, lda=m, layout="col",
                      workspace=torch.zeros(256, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n", [1, 2, 3, 30])
@pytest.mark.parametrize("ka,extra,pad", [(0, 0, 0), (1, 5, 0), (0, 3, 2)])
def test_tall(storage, n, ka, extra, pad):
    per = {"f32": 4, "f64": 2, "bf16": 8, "f16": 8}[storage]
    m = 768 * 152 * per + extra
    if n == 30:
        run_case(storage, "col", m, n, pad, ka, 1, alpha=-1.0, beta=1.0)
    else:
        run_case(storage, "col", m, n, pad, ka, 0)
