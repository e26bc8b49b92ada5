"""Which CSR batch plans give instances to the kernel that keeps x in shared memory (host
only): those for which the caller named no launch, neither with the plan nor as a default."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def nat():
    import __graft_entry__
    __graft_entry__._build_module().build()
    from paper_1409_0669_gb300 import _native
    _native.load()
    return _native


def info(nat, storage, cfg=None):
    d = (nat.CsrDesc * 400)(*[nat.CsrDesc(256, 512, 768, 1024, 1280, 20000, 20000, 680_000)] * 400)
    out = nat.BatchInfo()
    assert nat.load().lak_batch_plan(nat.OPS["spmv"], nat.DTYPES[storage], d, 400,
                                     ctypes.byref(cfg) if cfg else None, None, 0,
                                     ctypes.byref(out)) == 0
    return out


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16", "f64"])
def test_the_callers_default_names_the_launch(nat, storage):
    import paper_1409_0669_gb300 as lak
    lib = nat.load()
    mine = nat.LakCfg(128, 0, 4, 0)
    plain = info(nat, storage, mine).table_bytes
    # (two more prefix tables)
    assert (info(nat, storage).table_bytes > plain + 2 * 8 * 400) == (storage != "f64")
    before = set(lak._user_batch_defaults)
    try:
        lak.set_batch_default_cfg("spmv", storage, mine)
        got = info(nat, storage)
        assert got.cfg.as_tuple() == mine.as_tuple() and got.table_bytes == plain
        # an entry that the package ships only shapes the persistent launch
        assert lib.lak_set_batch_tuned_cfg(nat.OPS["spmv"], nat.DTYPES[storage],
                                           ctypes.byref(nat.LakCfg(512, 304, 8, 0))) == 0
        got = info(nat, storage)
        assert got.cfg.as_tuple() == (512, 304, 8, 0)
        assert (got.table_bytes > plain) == (storage != "f64")
        lak.set_batch_default_cfg("spmv", storage, None)             # back to the built-in shape
        got = info(nat, storage)
        assert got.cfg.as_tuple() == (64, 0, 4, 0)
        assert (got.table_bytes > plain) == (storage != "f64")
        for bad in (nat.LakCfg(48, 0, 4, 0), nat.LakCfg(64, -1, 4, 0)):
            assert lib.lak_set_batch_tuned_cfg(nat.OPS["spmv"], nat.DTYPES[storage],
                                               ctypes.byref(bad)) == nat.LAK_EINVAL
    finally:
        lib.lak_set_batch_default_cfg(nat.OPS["spmv"], nat.DTYPES[storage], None)
        lak._user_batch_defaults.clear()
        lak._user_batch_defaults.update(before)
