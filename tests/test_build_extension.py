"""The build of the Python extension (host only): it belongs to one torch, and the library is
built and the package works without it."""
import os
import subprocess
import sys
import types

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture()
def mod(tmp_path, monkeypatch):
    """The build script over a folder of its own, with compilers that only note their calls."""
    import __graft_entry__
    m = __graft_entry__._build_module()
    for name in ("OBJDIR", "LIB", "FAST", "FAST_STAMP"):
        monkeypatch.setattr(m, name, str(tmp_path / os.path.basename(getattr(m, name))))
    monkeypatch.setattr(m, "PKG", str(tmp_path))
    monkeypatch.setattr(m, "OBJDIR", str(tmp_path))
    m.calls = []

    def run(cmd, **kw):
        m.calls.append(cmd[0])
        if cmd[0] == "g++" and m.broken:
            return types.SimpleNamespace(returncode=1, stderr="no such header", stdout="")
        with open(cmd[cmd.index("-o") + 1], "w") as fh:
            fh.write("built")
        return types.SimpleNamespace(returncode=0, stderr="", stdout="")

    m.broken = False
    monkeypatch.setattr(m.subprocess, "run", run)
    return m


def test_another_torch_rebuilds(mod, monkeypatch):
    import torch
    assert mod.torch_version() == torch.__version__
    mod.build()
    assert os.path.exists(mod.FAST) and mod.up_to_date()
    n = len(mod.calls)
    mod.build()
    assert len(mod.calls) == n                    # nothing to do
    monkeypatch.setattr(mod, "torch_version", lambda: "9.9.9")
    assert not mod.up_to_date()
    mod.build()
    assert len(mod.calls) == 2 * n and mod.up_to_date()
    os.unlink(mod.FAST)
    assert not mod.up_to_date()


def test_the_library_is_built_without_the_extension(mod):
    mod.build()
    mod.broken = True
    with pytest.warns(UserWarning, match="no such header"):
        assert mod.build(force=True) == mod.LIB
    assert os.path.exists(mod.LIB) and not os.path.exists(mod.FAST)
    n = len(mod.calls)
    mod.build()                                   # the same sources and torch: not tried again
    assert len(mod.calls) == n
    mod.broken = False
    mod.build(force=True)
    assert os.path.exists(mod.FAST)


@pytest.mark.parametrize("state", ["another torch", "missing"])
def test_package_without_a_matching_extension(state):
    """Imported with an extension of another torch, or with none, the package takes the
    Python paths."""
    code = ("import sys, types\n"
            "m = types.ModuleType('paper_1409_0669_gb300._fast')\n"
            "m.torch_version = '0.0.0'\n"
            f"sys.modules['paper_1409_0669_gb300._fast'] = {'m' if state == 'another torch' else 'None'}\n"
            "import paper_1409_0669_gb300 as lak, paper_1409_0669_gb300.autograd as ag\n"
            "assert lak._fast is None and ag._fast is None\n"
            "assert lak.dense_gemv_workspace is not None\n")
    import __graft_entry__
    __graft_entry__._build_module().build()
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)
