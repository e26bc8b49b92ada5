"""GPU parity of the vector operations on operands that share no alignment (slices at
odd offsets, read through shifted 16-byte windows) against the FP64 oracle: lengths
around the fewest packs the path takes, every offset, an output in place of one
operand."""
import numpy as np
import pytest
import torch

import oracle
import synth
from checks import assert_dot, assert_ulp, canary_buffer, host

pytestmark = pytest.mark.gpu
STORAGES = ["f32", "f64", "bf16", "f16"]
SIZES = [1, 7, 8, 17, 31, 32, 33, 39, 40, 41, 47, 63, 1023, 65_537, 700_001]


def lak():
    import paper_1409_0669_gb300 as m
    return m


def at(n, seed, storage, offset):
    """n values that start `offset` elements into an allocation of exactly that size."""
    return synth.uniform(n + offset, seed, storage).cuda()[offset:]


def check_update(got, ref, storage, what):
    ref = oracle.round_to(ref, storage)
    if storage in ("f32", "f64"):
        assert np.array_equal(got, ref), what
    else:
        assert_ulp(got, ref, storage, 1.0, what)


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n", SIZES)
def test_updates_and_copy(storage, n):
    lk = lak()
    per = {"f32": 4, "f64": 2, "bf16": 8, "f16": 8}[storage]
    for ox, oy, oz in ((0, 1, 0), (1, 0, 0), (per - 1, 1, per // 2), (0, per - 1, 1), (3, 3, 2)):
        y, z = at(n, 1, storage, oy), at(n, 2, storage, oz)
        what = f"{storage} n={n} offsets {ox},{oy},{oz}"
        ref = oracle.axpy(y.cpu(), z.cpu(), 0.5)
        buf, _ = canary_buffer(n + ox, y.dtype, y.device)
        x = buf[64 + ox:64 + ox + n]
        lk.vec_axpy(x, y, z, 0.5)
        check_update(host(x), ref, storage, what)
        x.fill_(0)
        lk.vec_axpby(x, 1.0, y, 0.5, z)
        check_update(host(x), ref, storage, what)
        x.fill_(0)
        s = lk.vec_axpy_norm2(x, y, z, 0.5)
        check_update(host(x), ref, storage, what)
        got = host(x)
        assert_dot(float(s), oracle.dot(x.cpu(), x.cpu()), got, got, storage, what)
        lk.vec_copy(x, y)
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), what
        assert torch.isnan(buf[:64 + ox]).all() and torch.isnan(buf[64 + ox + n:]).all(), what


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("n", SIZES)
def test_inner_products(storage, n):
    lk = lak()
    for ox, oy in ((0, 1), (1, 0), (5, 2), (2, 7)):
        x, y = at(n, 3, storage, ox), at(n, 4, storage, oy)
        ref = oracle.dot(x.cpu(), y.cpu())
        got = lk.vec_dot(x, y)
        assert_dot(float(got), ref, host(x), host(y), storage, f"{storage} n={n} {ox},{oy}")
        assert torch.equal(got, lk.vec_dot(x, y)) and torch.equal(got, lk.vec_dot_noalloc(x, y))
        if storage != "f64":
            c = float(lk.vec_dot_compensated(x, y))
            scale = np.abs(host(x) * host(y)).sum()
            assert abs(c - ref) <= 2.0 ** -44 * scale


@pytest.mark.parametrize("storage", STORAGES)
def test_in_place_and_explicit_shapes(storage):
    lk = lak()
    n = 10_007
    for cfg in (None, (32, 1, 16, 0), (64, 5, 8, 1), (512, 0, 16, 1)):
        x, z = at(n, 5, storage, 1), at(n, 6, storage, 2)
        ref = oracle.axpy(x.cpu(), z.cpu(), 0.5)
        lk.vec_axpy(x, x, z, 0.5, cfg=cfg)                    # x = y, z off its alignment
        check_update(host(x), ref, storage, f"in place, {cfg}")
        x, y = at(n, 7, storage, 1), at(n, 8, storage, 4)
        ref = oracle.axpy(y.cpu(), x.cpu(), 0.5)
        lk.vec_axpy(x, y, x, 0.5, cfg=cfg)                    # x = z
        check_update(host(x), ref, storage, f"in place of z, {cfg}")
