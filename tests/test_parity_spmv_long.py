"""GPU parity of csr_spmv on long rows (mean above 64) against the FP64 oracle: every
number of lanes per row, last warps with missing rows, empty rows, hub rows that a
warp takes one by one, columns that repeat."""
import numpy as np
import pytest
import torch

import oracle
import synth
from checks import assert_canary, assert_normwise_scaled, assert_reduced_sum, canary_buffer, host

pytestmark = pytest.mark.gpu


def lengths(kind, m, g):
    lo, hi = {"short": (66, 99), "mid": (101, 159), "long": (170, 310), "longest": (321, 700),
              "hubs": (60, 90), "gaps": (130, 200)}[kind]
    lens = g.integers(lo, hi + 1, m)
    if kind == "hubs":                              # one row in 50 is far longer
        lens[g.random(m) < 0.02] = 5003
        lens[0] = 4001
    if kind == "gaps":                              # a third of the rows are empty
        lens[g.random(m) < 0.33] = 0
        lens[-1] = 500
    return lens


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16", "f16"])
@pytest.mark.parametrize("kind", ["short", "mid", "long", "longest", "hubs", "gaps"])
@pytest.mark.parametrize("m", [1, 7, 33, 1001])
def test_long_rows(storage, kind, m):
    import paper_1409_0669_gb300 as lak
    g = np.random.default_rng(m)
    n = 6007
    rp = np.concatenate([[0], np.cumsum(lengths(kind, m, g))]).astype(np.int32)
    assert rp[-1] > 64 * m
    ci = g.integers(1, n, rp[-1]).astype(np.int32)
    rp, ci = torch.from_numpy(rp), torch.from_numpy(ci)
    v, x = synth.normal(ci.numel(), 3, storage), synth.uniform(n, 4, storage)
    ref = oracle.csr_spmv(rp, ci, v, x)
    absr = oracle.csr_spmv(rp, ci, np.abs(oracle.widen(v)), np.abs(oracle.widen(x)))
    dx = x.cuda()
    dx[0] = float("nan")                            # no entry reads column 0
    buf, y = canary_buffer(m, v.dtype, "cuda")
    off = torch.empty(ci.numel() + 1, dtype=torch.int32, device="cuda")[1:]
    off.copy_(ci)                                   # col_idx off 16 bytes
    lak.csr_spmv(rp.cuda(), off, v.cuda(), dx, y=y)
    torch.cuda.synchronize()
    if storage in ("f32", "f64"):
        assert_normwise_scaled(host(y), ref, absr, storage, f"{kind} {m}")
    else:
        assert_reduced_sum(host(y), ref, absr, np.diff(rp.numpy()).astype(np.float64), storage,
                           f"{kind} {m}")
    assert_canary(buf, m)


@pytest.mark.parametrize("storage", ["f32", "f64", "bf16"])
@pytest.mark.parametrize("m", [8191, 8193, 65537, 262145])
def test_lanes_by_rows(storage, m):
    """Row counts on both sides of the lines between the numbers of lanes per row."""
    import paper_1409_0669_gb300 as lak
    g = np.random.default_rng(m)
    lens = g.integers(60, 72, m)
    lens[[0, m // 2, m - 1]] = 4001, 0, 777         # hub rows and an empty one
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    assert rp[-1] > 64 * m
    ci = g.integers(0, 6007, rp[-1]).astype(np.int32)
    rp, ci = torch.from_numpy(rp), torch.from_numpy(ci)
    v, x = synth.normal(ci.numel(), 5, storage), synth.uniform(6007, 6, storage)
    ref = oracle.csr_spmv(rp, ci, v, x)
    absr = oracle.csr_spmv(rp, ci, np.abs(oracle.widen(v)), np.abs(oracle.widen(x)))
    buf, y = canary_buffer(m, v.dtype, "cuda")
    lak.csr_spmv(rp.cuda(), ci.cuda(), v.cuda(), x.cuda(), y=y)
    torch.cuda.synchronize()
    if storage == "bf16":
        assert_reduced_sum(host(y), ref, absr, np.diff(rp.numpy()).astype(np.float64), storage,
                           f"{m}")
    else:
        assert_normwise_scaled(host(y), ref, absr, storage, f"{m}")
    assert_canary(buf, m)
