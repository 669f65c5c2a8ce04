"""What the build makes when one of its two files is missing or was made for something else, and the
binding without the marshalling extension."""
import os
import sys
import types

import pytest

from paper_2507_02659_b200 import binding, build


@pytest.fixture
def fake_build(tmp_path, monkeypatch):
    """The build with its outputs in a scratch folder and no compiler; which files it made, in order."""
    made = []
    monkeypatch.setattr(build, "LIB", str(tmp_path / "libomnidraft.so"))
    monkeypatch.setattr(build, "EXT", str(tmp_path / "_marshal.so"))
    monkeypatch.setattr(build, "EXT_FOR", str(tmp_path / "_build" / "marshal_built_for"))

    def run(cmd, **kw):
        out = cmd[cmd.index("-o") + 1]
        made.append(os.path.basename(out).split(".")[0])
        open(out, "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")
    monkeypatch.setattr(build.subprocess, "run", run)
    return made


def test_each_missing_or_stale_file_is_built(fake_build, monkeypatch):
    build.build()
    assert fake_build == ["libomnidraft", "_marshal"]
    build.build()
    assert len(fake_build) == 2
    os.remove(build.LIB)                                    # the extension alone is no reason to build nothing
    assert os.path.exists(build.build()) and fake_build[2:] == ["libomnidraft"]
    os.remove(build.EXT)
    build.build()
    assert fake_build[3:] == ["_marshal"]
    monkeypatch.setattr(build, "built_for", lambda: "python 3.99, torch 9")
    build.build()
    assert fake_build[4:] == ["_marshal"]


def test_a_host_without_a_compiler_for_the_extension(fake_build, monkeypatch, capsys):
    build.build()
    monkeypatch.setattr(build, "built_for", lambda: "python 3.99, torch 9")

    def run(cmd, **kw):
        raise FileNotFoundError("g++")
    monkeypatch.setattr(build.subprocess, "run", run)
    assert os.path.exists(build.build())
    assert not os.path.exists(build.EXT)                    # the one of another torch does not stay
    assert "in Python" in capsys.readouterr().err


@pytest.mark.parametrize("marshal", [None, types.SimpleNamespace(built_for="python 3.99, torch 9")])
def test_the_binding_without_the_extension(monkeypatch, marshal):
    build.build()
    monkeypatch.setitem(sys.modules, "paper_2507_02659_b200._marshal", marshal)
    if marshal is not None:
        monkeypatch.setattr(sys.modules["paper_2507_02659_b200"], "_marshal", marshal, raising=False)
    else:
        monkeypatch.delattr(sys.modules["paper_2507_02659_b200"], "_marshal", raising=False)
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_native", None)
    with pytest.warns(RuntimeWarning, match="_marshal is not usable"):
        assert binding.lib().od_version() >= 100
    assert binding._native.step(0, 0) is None and binding._native.cache_trim(0, 0) is None


def test_the_extension_belongs_to_this_python_and_torch():
    build.build()
    from paper_2507_02659_b200 import _marshal
    assert _marshal.built_for == build.built_for()
