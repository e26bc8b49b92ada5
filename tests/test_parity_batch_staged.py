"""GPU parity of the CSR batch where x is kept in shared memory against the FP64 oracle:
instances on both sides of the rule in one batch, several units per instance, rows that
cross steps, rows longer than a step, empty rows, a last block with missing rows, the
largest x that fits and one more, x off 16 bytes, row pointers that begin past the
array's start, and a replay from a CUDA graph."""
import numpy as np
import pytest
import torch

import oracle
import synth
from checks import assert_normwise, assert_reduced_sum, host

pytestmark = pytest.mark.gpu
FIT = {"f32": 51200, "bf16": 102400, "f16": 102400}      # values of x that fit


def matrix(kind, storage, g):
    """(row lengths, n, entries before row_ptr[0], elements by which x is off)"""
    if kind == "units":                                  # three units, the last one ragged
        return g.integers(17, 65, 9007), 9007, 0, 0
    if kind == "hubs":
        ln = g.integers(0, 40, 2003)
        ln[[0, 1000, 2002]] = 9001, 257, 5003
        return ln, 4099, 0, 1
    if kind == "long":
        return g.integers(97, 700, 101), 7001, 0, 0
    if kind == "gaps":
        ln = g.integers(60, 130, 1500)
        ln[g.random(1500) < 0.4] = 0
        ln[-40:] = 0
        return ln, 1501, 5, 3
    if kind == "widest":
        return g.integers(30, 65, 5000), FIT[storage], 0, 0
    if kind == "too_wide":
        return g.integers(30, 65, 5000), FIT[storage] + 1, 0, 0
    if kind == "small":                                  # too few entries
        return g.integers(5, 60, 300), 300, 0, 0
    assert kind == "pairs"                               # staged with 16-bit storage only
    return g.integers(0, 7, 13001), 13001, 0, 0


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
def test_staged_batch_vs_oracle(storage):
    from paper_1409_0669_gb300 import batch as B
    g = np.random.default_rng(5)
    kinds = ["units", "hubs", "long", "gaps", "widest", "too_wide", "small", "pairs"]
    made = []
    for i, kind in enumerate(kinds):
        ln, n, lead, off = matrix(kind, storage, g)
        rp = np.concatenate([[0], np.cumsum(ln)]).astype(np.int32)
        ci = g.integers(0, n, rp[-1]).astype(np.int32)
        v, x = synth.normal(int(rp[-1]), 10 + i, storage), synth.uniform(n, 30 + i, storage)
        rpt, cit = torch.from_numpy(rp), torch.from_numpy(ci)
        ref = oracle.csr_spmv(rpt, cit, v, x)
        absr = oracle.csr_spmv(rpt, cit, np.abs(oracle.widen(v)), np.abs(oracle.widen(x)))
        dc = torch.full((lead + ci.size,), 2 ** 30, dtype=torch.int32, device="cuda")
        dc[lead:] = cit.cuda()
        dv = torch.full((lead + ci.size,), float("nan"), dtype=v.dtype, device="cuda")
        dv[lead:] = v.cuda()
        dx = torch.full((n + off,), float("nan"), dtype=x.dtype, device="cuda")[off:]
        dx.copy_(x)
        made.append(((rpt.cuda() + lead, dc, dv, n), dx, ref, absr, ln.astype(np.float64)))
    count = 1200                                         # over 608 staged units in all storages
    order = [made[i % len(made)] for i in range(count)]
    ms = [m[4].size for m in order]
    starts = np.concatenate([[0], np.cumsum(np.array(ms) + 3)])
    out = torch.full((int(starts[-1]),), float("nan"), dtype=order[0][1].dtype, device="cuda")
    ys = [out[int(s):int(s) + m] for s, m in zip(starts, ms)]
    b = B.spmv_batch([m[0] for m in order], [m[1] for m in order], ys)
    plain = B.spmv_batch([m[0] for m in order], [m[1] for m in order], ys, cfg=(128, 0, 4, 0))
    assert b.info.table_bytes > plain.info.table_bytes   # some are staged
    b.run()
    torch.cuda.synchronize()
    first = out.clone()
    for i in list(range(len(made))) + [count - 1 - j for j in range(len(made))]:
        _, _, ref, absr, lens = order[i]
        y, what = host(ys[i]), f"{kinds[i % len(made)]} {i}"
        if storage == "f32":
            assert_normwise(y, ref, storage, what)
        else:
            assert_reduced_sum(y, ref, absr, lens, storage, what)
    for i in range(count):                               # equal instances: equal bits
        assert torch.equal(ys[i], ys[i % len(made)])
        assert torch.isnan(out[int(starts[i]) + ms[i]:int(starts[i + 1])]).all()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.run()
    for _ in range(2):
        out.fill_(float("nan"))
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.nan_to_num(out), torch.nan_to_num(first))
