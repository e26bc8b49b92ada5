"""The kernels for special shapes against the general kernels (an explicit configuration
names those): over many rows the root mean square of their errors is no larger.  References
are exact or nearly so: FP64 sums of FP32 values, and for FP64 integers whose products and
sums a 64-bit integer holds but a double does not.

Bound: with R rows of independent errors the mean square has a relative deviation of
sqrt(2 / R) at most 1 %, the ratio of two root mean squares 0.7 %; 4 % are more than five of
these."""
import pytest
import torch

pytestmark = pytest.mark.gpu
SLACK = 1.04
SMS = 152


def lak():
    import paper_1409_0669_gb300 as m
    return m


def gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def rms(y, exact):
    d = y.double() - exact if exact.dtype == torch.float64 else (y.long() - exact).double()
    return float(d.square().mean().sqrt())


def csr(lo, hi, m, seed=5):
    g = gen(seed)
    lens = torch.randint(lo, hi, (m,), device="cuda", generator=g)
    rp = torch.zeros(m + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum(lens, 0)
    ci = torch.randint(0, m, (int(rp[-1]),), device="cuda", generator=g).int()
    return rp, ci, torch.repeat_interleave(torch.arange(m, device="cuda"), lens)


@pytest.mark.parametrize("lo, hi, m", [(81, 82, 300_000), (66, 100, 270_000), (81, 82, 20_000),
                                       (105, 150, 70_000), (170, 256, 40_000)])
def test_long_rows_f64(lo, hi, m):
    rp, ci, row = csr(lo, hi, m)
    g = gen(6)
    # products of up to 2^54, 256 of them within 63 bits
    v = torch.randint(-2 ** 30, 2 ** 30, ci.shape, device="cuda", generator=g)
    x = torch.randint(-2 ** 24, 2 ** 24, (m,), device="cuda", generator=g)
    exact = torch.zeros(m, dtype=torch.int64, device="cuda").index_add_(0, row, v * x[ci.long()])
    args = (rp, ci, v.double(), x.double())
    err = rms(lak().csr_spmv(*args), exact)
    general = rms(lak().csr_spmv(*args, cfg=(64, 16 * SMS, 8, 0)), exact)
    assert 0 < err <= SLACK * general, (err, general)


@pytest.mark.parametrize("lo, hi, m", [(81, 82, 300_000), (105, 150, 100_000), (140, 181, 70_000),
                                       (400, 700, 20_000), (2000, 3000, 20_000)])
def test_long_rows_f32(lo, hi, m):
    rp, ci, row = csr(lo, hi, m)
    g = gen(6)
    v = torch.randn(ci.shape, device="cuda", generator=g)
    x = torch.rand(m, device="cuda", generator=g) * 2 - 1
    exact = torch.zeros(m, dtype=torch.float64, device="cuda").index_add_(
        0, row, v.double() * x.double()[ci.long()])
    err = rms(lak().csr_spmv(rp, ci, v, x), exact)
    general = rms(lak().csr_spmv(rp, ci, v, x, cfg=(128, 16 * SMS, 4, 0)), exact)
    assert 0 < err <= SLACK * general, (err, general)


def dense(m, n, layout):
    g = gen(7)
    A = torch.randn(m * n, device="cuda", generator=g)
    A = A.view(m, n) if layout == "row" else A.view(n, m).t()
    x = torch.rand(n, device="cuda", generator=g) * 2 - 1
    exact = torch.cat([A[r:r + 20_000].double() @ x.double() for r in range(0, m, 20_000)])
    return A, x, exact


@pytest.mark.parametrize("layout, m, n, general", [
    ("row", 20_000, 1500, (32, 32 * SMS, 8, 0)), ("row", 40_000, 1600, (32, 32 * SMS, 8, 0)),
    ("row", 20_000, 3001, (32, 32 * SMS, 8, 0)),
    ("col", 1_000_000, 8, (512, 0, 8, 0)), ("col", 2_000_000, 30, (512, 2 * SMS, 8, 1)),
    ("col", 500_000, 50, (512, 2 * SMS, 8, 1)), ("col", 1_000_000, 64, (512, 2 * SMS, 8, 1)),
    ("col", 999_983, 17, (512, 2 * SMS, 8, 1)), ("col", 700_001, 33, (512, 2 * SMS, 8, 1)),
    ("col", 30_001, 1000, (512, 2 * SMS, 8, 1))])
def test_dense_f32(layout, m, n, general):
    A, x, exact = dense(m, n, layout)
    err = rms(lak().dense_gemv(A, x), exact)
    ref = rms(lak().dense_gemv(A, x, cfg=general), exact)
    assert 0 < err <= SLACK * ref, (err, ref)


@pytest.mark.parametrize("m, n, general", [
    (1_000_000, 8, (128, 8 * SMS, 2, 1)), (700_001, 8, (512, 2 * SMS, 4, 0)),
    (2_000_000, 30, (128, 8 * SMS, 2, 1)), (500_000, 50, (128, 8 * SMS, 2, 1)),
    (250_001, 9, (512, 2 * SMS, 4, 0)), (130_001, 17, (512, 2 * SMS, 4, 0)),
    (30_001, 900, (128, 8 * SMS, 2, 1))])
def test_dense_columns_f64(m, n, general):
    g = gen(8)
    # sums as large as 63 bits hold, so that every addition rounds
    bits = 32 - n.bit_length()
    A = torch.randint(-2 ** 30, 2 ** 30, (n, m), device="cuda", generator=g)
    x = torch.randint(-2 ** bits, 2 ** bits, (n,), device="cuda", generator=g)
    exact = (A * x[:, None]).sum(0)
    Ad, xd = A.double().t(), x.double()
    err = rms(lak().dense_gemv(Ad, xd), exact)
    ref = rms(lak().dense_gemv(Ad, xd, cfg=general), exact)
    assert 0 < err <= SLACK * ref, (err, ref)
