"""The CSR transpose of patterns with far fewer entries than rows or columns, and with long
runs of empty rows, against the oracle's stable counting sort (bit-equal), and that its time
does not grow with the runs."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def lak():
    import paper_1409_0669_gb300 as m
    return m


def make(kind):
    """(row of every entry, number of rows, columns, number of columns)"""
    g = np.random.default_rng(11)
    if kind == "gap":                         # 10,000 rows at either end of 1.2 M
        r = np.concatenate([g.integers(0, 10_000, 700_000), 1_190_000 + g.integers(0, 10_000, 700_000)])
        m, n = 1_200_000, 40_000
    elif kind == "spread":                    # dense rows, then single entries far apart
        r = np.concatenate([g.integers(0, 20_000, 500_000), 20_000 + 300 * np.arange(1000)])
        m, n = 320_001, 3000
    elif kind == "empty ends":                # runs of empty rows before and after
        r, m, n = 400_000 + g.integers(0, 50, 900_000), 800_000, 300_000
    elif kind == "few entries":
        r, m, n = g.integers(0, 3_000_000, 1000), 3_000_000, 1000
    elif kind == "few entries, one row":      # a hub row among mostly empty ones
        r = np.concatenate([np.full(9001, 77_777), g.integers(0, 200_000, 501)])
        m, n = 200_000, 5000
    elif kind == "as many rows":              # either side of the rule on rows and entries
        r, m, n = g.integers(0, 100_000, 100_000), 100_000, 60_000
    elif kind == "one row more":
        r, m, n = g.integers(0, 100_001, 100_000), 100_001, 60_000
    elif kind == "two passes":                # 1024-column blocks in two passes
        r, m, n = g.integers(0, 90_000, 700_000), 90_000, 2_200_000
    elif kind == "blocks of 4096 columns":
        r, m, n = g.integers(0, 30_000, 300_000), 30_000, 1_300_000
    else:                                     # the same, a hub column beyond shared memory
        assert kind == "blocks of 4096 columns, hub"
        r, m, n = g.integers(0, 30_000, 300_000), 30_000, 6_000_000
    r.sort()
    ci = g.integers(0, n, r.size)
    if kind.endswith("hub"):
        ci[g.random(r.size) < 0.02] = 5_999_999
    return r, m, ci, n


KINDS = ["gap", "spread", "empty ends", "few entries", "few entries, one row", "as many rows",
         "one row more", "two passes", "blocks of 4096 columns", "blocks of 4096 columns, hub"]


@pytest.mark.parametrize("kind", KINDS)
def test_transpose_equals_the_oracle(kind):
    r, m, ci, n = make(kind)
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=m))])
    rp, ci = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)) for a in (rp, ci))
    want = oracle.csr_to_csc(rp, ci, n)
    vals = torch.arange(ci.numel(), dtype=torch.float32, device="cuda")
    cp, ri, perm, vt = lak().csr_transpose_vals(rp.cuda(), ci.cuda(), vals, n)
    for a, b in zip((cp, ri, perm), want):
        assert np.array_equal(a.cpu().numpy(), b)
    assert torch.equal(vt, vals[perm.long()])


@pytest.mark.parametrize("m, ends", [(10_000_000, 10_000_000), (16_000_000, 1000)])
def test_time_does_not_grow_with_the_empty_rows(m, ends):
    """1000 entries anywhere in 10 M rows, and 2 M in the first and the last thousand of
    16 M: tens of microseconds.  A walk through the empty rows took 19 and 175 ms."""
    g = torch.Generator(device="cuda").manual_seed(3)
    nnz = 1000 if ends == m else 2_000_000
    r = torch.randint(0, ends, (nnz,), device="cuda", generator=g)
    if ends < m:
        r[nnz // 2:] = m - 1 - r[nnz // 2:]
    rp = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(r, minlength=m), 0)
    ci = torch.randint(0, 50_000, (nnz,), device="cuda", generator=g).int()
    lk = lak()
    best = float("inf")
    for _ in range(4):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        lk.csr_transpose(rp, ci, 50_000)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    assert best < 3.0, f"{best:.2f} ms"
