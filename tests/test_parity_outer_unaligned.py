"""dense_outer on rows off the access width (odd leading dimensions, offset outputs),
bit-equal to the oracle's rounded products, nothing written beside the rows."""
import numpy as np
import pytest
import torch

import oracle
import synth
from checks import host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,m,n", [("f32", 1025, 1023), ("f32", 33, 40_001), ("f32", 20_003, 61),
                                         ("f64", 701, 803), ("bf16", 4099, 8191), ("f16", 8200, 4098)])
@pytest.mark.parametrize("pad,off", [(0, 0), (1, 0), (2, 3), (5, 1)])
def test_outer_unaligned(storage, m, n, pad, off):
    import paper_1409_0669_gb300 as lak
    dy, x = synth.uniform(m, 1, storage), synth.uniform(n, 2, storage)
    ld = n + pad
    buf = torch.full((off + m * ld + 16,), float("nan"), dtype=x.dtype, device="cuda")
    out = buf[off:off + m * ld].view(m, ld)[:, :n]
    lak.dense_outer(dy.cuda(), x.cuda(), out=out)
    torch.cuda.synchronize()
    rows = np.unique(np.r_[0, 1, m - 1, np.arange(0, m, max(1, m // 300))])
    ref = oracle.round_to(oracle.dense_outer(dy[rows], x).ravel(), storage)
    assert np.array_equal(host(out[rows].contiguous()).ravel(), ref)
    assert not torch.isnan(out).any()
    out.fill_(float("nan"))
    assert torch.isnan(buf).all()
