"""The workspace of dense_gemv on few long rows, where it is optional: the caller's own is
used, the query covers any leading dimension, a smaller one gets fewer splits, a captured
call depends on no buffer that later calls replace, and scratch that the library makes for
a call on a given stream belongs to that stream."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from checks import assert_normwise_scaled, host

pytestmark = pytest.mark.gpu
COUNTERS = 65536


def lak():
    import paper_1409_0669_gb300 as m
    return m


def few_rows(m, n, lda, storage, seed=1):
    """(A, x, the oracle's A x, |A| |x|), A an m x n view of rows lda apart"""
    A = torch.full((m, lda), float("nan"), dtype=synth.torch_dtype(storage))
    A[:, :n] = synth.normal((m, n), seed, storage)
    x = synth.uniform(n, seed + 1, storage)
    full = A[:, :n].contiguous()
    ref = oracle.gemv(full, x, m, n, n, "row")
    absr = oracle.gemv(full.abs(), x.abs(), m, n, n, "row")
    return A.cuda()[:, :n], x.cuda(), ref, absr


def call(A, x, ws, nbytes):
    from paper_1409_0669_gb300 import _native
    y = torch.full((A.shape[0],), float("nan"), dtype=A.dtype, device="cuda")
    st = _native.load().dense_gemv(y.data_ptr(), A.data_ptr(), x.data_ptr(), A.shape[0], A.shape[1],
                                   A.stride(0), 0, _native.DTYPES[lak().storage_of(A)],
                                   ws.data_ptr() if nbytes else None, nbytes, None,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    return y


@pytest.mark.parametrize("storage, n, lda", [("f32", 1_048_577, 1_048_580), ("f64", 400_001, 400_002),
                                             ("f32", 300_000, 300_001), ("bf16", 700_003, 700_008),
                                             ("bf16", 700_000, 700_001), ("f64", 400_000, 400_001)])
def test_query_covers_any_leading_dimension(storage, n, lda):
    """The splits fill the GPU on the queried workspace, also where lda gives the rows
    another period than n does; less room gives fewer splits and the same sums."""
    m, es = 10, 8 if storage == "f64" else 4
    A, x, ref, absr = few_rows(m, n, lda, storage)
    need = lak().dense_gemv_workspace(m, n, "row", storage)
    assert need > COUNTERS
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")

    def splits(nbytes):
        ws[:COUNTERS] = 0
        ws[COUNTERS:] = 255                       # NaN: a sum that no split wrote
        y = call(A, x, ws, nbytes)
        assert_normwise_scaled(host(y), ref, absr, "f32" if storage != "f64" else "f64", storage) \
            if storage != "bf16" else np.testing.assert_allclose(host(y), ref, rtol=0.02, atol=2.0)
        assert (ws[:COUNTERS] == 0).all()
        words = ws[COUNTERS:COUNTERS + (need - COUNTERS) // (m * es) * m * es].view(-1, m * es)
        return int((words != 255).any(dim=1).sum())

    full = splits(need)
    sets_at_most = m                              # one row per set and block of a split
    assert full * sets_at_most >= 152 and full >= 2
    assert splits(COUNTERS + 5 * m * es) == 5
    assert splits(COUNTERS + 2 * m * es - 1) == 0
    assert splits(0) == 0


def test_the_callers_workspace_is_used():
    m = lak()
    A, x, ref, absr = few_rows(8, 300_000, 300_000, "f32")
    need = m.dense_gemv_workspace(8, 300_000, "row", "f32")
    key = (torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)
    kept = m._workspaces.pop(key, None)
    try:
        for run in (lambda w: m.dense_gemv(A, x, workspace=w),
                    lambda w: m.dense_gemv_trans(A.t(), x, workspace=w)):
            ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
            y = run(ws)
            assert (ws[:COUNTERS] == 0).all() and (ws[COUNTERS:] != 0).any()
            assert_normwise_scaled(host(y), ref, absr, "f32")
            assert key not in m._workspaces       # nothing made by the library
    finally:
        if kept is not None:
            m._workspaces[key] = kept


def test_captured_call_outlives_the_kept_workspace():
    """Capture without a call before it, replay after the stream's kept workspace was made,
    used, grown and its memory taken by other tensors."""
    m = lak()
    A, x, ref, absr = few_rows(8, 300_000, 300_000, "f32")
    big, xb, _, _ = few_rows(60, 400_000, 400_000, "f64")
    side = torch.cuda.Stream()
    key = (torch.cuda.current_device(), side.cuda_stream)
    m._workspaces.pop(key, None)
    y = torch.empty(8, device="cuda")
    torch.cuda.synchronize()
    for first in (True, False):                   # without, then with a kept workspace
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            m.dense_gemv(A, x, y)
        assert first == (key not in m._workspaces)
        with torch.cuda.stream(side):
            m.dense_gemv(A, x)                    # not on the graph's memory
            if not first:
                m.dense_gemv(big, xb)
            taken = [torch.full((1 << k,), 7, dtype=torch.uint8, device="cuda")
                     for k in range(14, 22) for _ in range(3)]
            for _ in range(3):
                y.fill_(float("nan"))
                graph.replay()
                assert_normwise_scaled(host(y), ref, absr, "f32")
        assert all((t == 7).all() for t in taken)
        del taken, graph


@pytest.mark.parametrize("handle", [False, True])
def test_scratch_of_a_given_stream(handle):
    """The first calls on another stream, while the current one is busy and the allocator
    has memory that is not zero: the scratch is filled on the stream that uses it."""
    m = lak()
    A, x, ref, absr = few_rows(8, 300_000, 300_000, "f32")
    want = m.vec_dot(x, x).item()
    out, y = torch.full((1,), float("nan"), device="cuda"), torch.full((8,), float("nan"), device="cuda")
    side = torch.cuda.Stream()
    m._workspaces.pop((torch.cuda.current_device(), side.cuda_stream), None)
    junk = [torch.full((1 << k,), 255, dtype=torch.uint8, device="cuda") for k in range(16, 22)]
    torch.cuda.synchronize()
    del junk
    torch.cuda._sleep(200_000_000)                # about 0.1 s
    stream = side.cuda_stream if handle else side
    m.vec_dot(x, x, out=out, stream=stream)
    m.dense_gemv(A, x, y, stream=stream)
    side.synchronize()
    assert torch.cuda.current_stream().query() is False
    with torch.cuda.stream(side):
        got, gy = out.item(), host(y)
    torch.cuda.synchronize()
    assert got == want
    assert_normwise_scaled(gy, ref, absr, "f32")
