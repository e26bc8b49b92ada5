"""GPU parity of the vector operations on operands of unlike alignment around the sizes from
which they are read through shifted windows, with every remainder, with explicit launches,
and of the compensated inner product on either side of its own line."""
import numpy as np
import pytest
import torch

import oracle
import synth
from checks import assert_ulp, canary_buffer, host

pytestmark = pytest.mark.gpu


def lak():
    import paper_1409_0669_gb300 as m
    return m


def at(n, seed, storage, offset):
    return synth.uniform(n + offset, seed, storage).cuda()[offset:]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("cfg", [None, (32, 1, 16, 0), (64, 5, 8, 1), (512, 0, 16, 1)])
def test_updates_and_copy_at_the_line(storage, cfg):
    lk = lak()
    es = 4 if storage == "f32" else 2
    for operands, op in ((3, "axpy"), (2, "copy")):
        line = -(-(1 << 20) // (operands * es))              # the first size of a mebibyte
        for n in [line - 1] + [line + r for r in range(0, 17)]:
            for ox, oy, oz in ((0, 1, 2), (1, 0, 0), (3, 2, 1)):
                y, z = at(n, 1, storage, oy), at(n, 2, storage, oz)
                buf, _ = canary_buffer(n + ox, y.dtype, y.device)
                x = buf[64 + ox:64 + ox + n]
                what = f"{op} {storage} n={n} offsets {ox},{oy},{oz}"
                if op == "copy":
                    lk.vec_copy(x, y, cfg=cfg)
                    assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), what
                else:
                    lk.vec_axpy(x, y, z, 0.5, cfg=cfg)
                    ref = oracle.round_to(oracle.axpy(y.cpu(), z.cpu(), 0.5), storage)
                    if storage == "f32":
                        assert np.array_equal(host(x), ref), what
                    else:
                        assert_ulp(host(x), ref, storage, 1.0, what)
                assert torch.isnan(buf[:64 + ox]).all() and torch.isnan(buf[64 + ox + n:]).all(), what


@pytest.mark.parametrize("n", [16_777_215, 16_777_217])      # 64 MiB of two BF16 operands
def test_compensated_at_its_line(n):
    lk = lak()
    g = torch.Generator(device="cuda").manual_seed(3)
    b = (torch.rand(2 * n + 3, device="cuda", generator=g) * 2 - 1).bfloat16()
    x, y = b[:n], b[n + 3:]                                  # unlike alignment
    xd, yd = x.double(), y.double()
    got = float(lk.vec_dot_compensated(x, y))
    # products of 16-bit values are exact in FP64; its tree sum is good to 2^-48 here
    assert abs(got - float((xd * yd).sum())) <= 2.0 ** -44 * float((xd * yd).abs().sum())
