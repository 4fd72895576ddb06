"""The build rules, with the compilers replaced by a recorder."""
import importlib.metadata
import importlib.util
import os

import pytest

from paper_2607_10071_b200 import build as fbuild


@pytest.fixture
def compiled(monkeypatch, tmp_path):
    """Outputs go to a folder of the test; the list holds what was asked of the compilers, by output file name."""
    done = []

    def run(cmd, check):
        out = cmd[cmd.index("-o") + 1]
        done.append(os.path.basename(out))
        open(out, "w").close()

    for name in ("LIB", "LIB_DEBUG_BOUNDS", "NATIVE", "NATIVE_RECORD"):
        monkeypatch.setattr(fbuild, name, str(tmp_path / os.path.basename(getattr(fbuild, name))))
    monkeypatch.setattr(fbuild.subprocess, "run", run)
    return done


def _without_torch(monkeypatch):
    find = importlib.util.find_spec
    monkeypatch.setattr(importlib.util, "find_spec", lambda name, *a: None if name == "torch" else find(name, *a))


def test_library_builds_without_pytorch(compiled, monkeypatch, capsys):
    _without_torch(monkeypatch)
    assert fbuild.build() == fbuild.LIB
    assert compiled == ["libflashbev.so"]
    assert "PyTorch is not installed" in capsys.readouterr().err
    with pytest.raises(RuntimeError, match="PyTorch is not installed"):
        fbuild.build_native()


def test_library_and_extension_build_with_pytorch(compiled):
    if fbuild.native_prerequisites():
        pytest.skip(fbuild.native_prerequisites())
    fbuild.build(force=True)
    assert compiled == ["libflashbev.so", os.path.basename(fbuild.NATIVE)]
    fbuild.build()                                 # up to date
    assert len(compiled) == 2


def test_extension_is_rebuilt_for_another_pytorch(compiled, monkeypatch):
    if fbuild.native_prerequisites():
        pytest.skip(fbuild.native_prerequisites())
    name = os.path.basename(fbuild.NATIVE)
    fbuild.build_native()
    fbuild.build_native()
    assert compiled == [name]
    version = importlib.metadata.version
    monkeypatch.setattr(importlib.metadata, "version", lambda p: "99.0" if p == "torch" else version(p))
    fbuild.build_native()
    fbuild.build_native()
    assert compiled == [name, name]
    os.remove(fbuild.NATIVE_RECORD)                # built by hand, or by an older rule: nothing says what with
    fbuild.build_native()
    assert compiled == [name, name, name]
