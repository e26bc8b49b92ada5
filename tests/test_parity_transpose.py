"""The CSR transpose by stable partitioning against the oracle's stable counting sort
(bit-equal): every branch of its plan -- one and two partition passes, column blocks
that fit in shared memory and hub columns that do not, runs of empty rows, few entries
-- and the values carried along, in all storage types."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


def lak():
    import paper_1409_0669_gb300 as m
    return m


def make(kind):
    """(row_ptr, col_idx, n_cols)"""
    g = np.random.default_rng(5)
    if kind == "one entry":
        return np.array([0, 0, 1, 1]), np.array([6]), 7
    if kind == "one column":                      # nnz in one hub column, beyond shared memory
        m = 50_001
        return np.arange(m + 1), np.zeros(m, np.int64), 1
    if kind == "ragged":
        lens = g.integers(0, 30, 3001)
        n = 777
    elif kind == "empty rows":                    # runs of far more than 32 empty rows
        lens = np.where(g.random(40_000) < 0.01, g.integers(1, 200, 40_000), 0)
        n = 5000
    elif kind == "hub":                           # a third of the entries in one column
        lens = g.integers(0, 40, 20_000)
        n = 30_000
    elif kind == "powerlaw":
        rp, ci, _ = synth.powerlaw_csr(60_000, 50_000, 3)
        return rp.numpy(), ci.numpy(), 50_000
    elif kind == "wide":                          # more than 2048 blocks of 1024 columns
        lens = g.integers(0, 12, 150_000)
        n = 5_000_011
    elif kind == "wide and few":
        lens = g.integers(0, 3, 500)
        n = 2_097_153
    rp = np.concatenate([[0], np.cumsum(lens)])
    ci = g.integers(0, n, rp[-1])
    if kind == "hub":
        ci[g.random(ci.size) < 0.33] = 12_345
    return rp, ci, n


KINDS = ["one entry", "one column", "ragged", "empty rows", "hub", "powerlaw", "wide",
         "wide and few"]


@pytest.mark.parametrize("kind", KINDS)
def test_transpose_equals_the_oracle(kind):
    lk = lak()
    rp, ci, n = make(kind)
    rp, ci = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)) for a in (rp, ci))
    ocp, ori, operm = oracle.csr_to_csc(rp, ci, n)
    drp, dci = rp.cuda(), ci.cuda()
    cp, ri, perm = lk.csr_transpose(drp, dci, n)
    assert np.array_equal(cp.cpu().numpy(), ocp)
    assert np.array_equal(ri.cpu().numpy(), ori)
    assert np.array_equal(perm.cpu().numpy(), operm)
    for st in ("f32", "f64", "bf16", "f16"):
        v = synth.normal(ci.numel(), 4, st).cuda()
        for a, b in zip(lk.csr_transpose_vals(drp, dci, v, n), (cp, ri, perm, v[perm.long()])):
            assert torch.equal(a, b)


def test_least_workspace_gives_the_same():
    """The documented least workspace (no room for records) still serves the call."""
    lk = lak()
    from paper_1409_0669_gb300 import _native
    lib = _native.load()
    rp, ci, n = make("ragged")
    rp, ci = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in (rp, ci))
    want = lk.csr_transpose(rp, ci, n)
    got = [torch.empty_like(t) for t in want]
    ws = torch.empty(lib.csr_transpose_workspace(n), dtype=torch.uint8, device="cuda")
    assert ws.numel() < lib.csr_transpose_vals_workspace(n, ci.numel(), 0)
    args = [t.data_ptr() for t in got] + [rp.data_ptr(), ci.data_ptr(), rp.numel() - 1, n,
                                          ci.numel(), ws.data_ptr(), ws.numel()]
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.csr_transpose(*args, stream) == 0
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_empty_matrix_and_side_stream():
    lk = lak()
    rp = torch.zeros(5, dtype=torch.int32, device="cuda")
    none = torch.empty(0, dtype=torch.int32, device="cuda")
    cp, ri, perm, vt = lk.csr_transpose_vals(rp, none, torch.empty(0, device="cuda"), 9)
    assert cp.tolist() == [0] * 10 and ri.numel() == perm.numel() == vt.numel() == 0
    # on another stream: the scratch belongs to it
    rp, ci, n = make("ragged")
    rp, ci = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in (rp, ci))
    want = lk.csr_transpose(rp, ci, n)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    got = lk.csr_transpose(rp, ci, n, stream=side)
    side.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
