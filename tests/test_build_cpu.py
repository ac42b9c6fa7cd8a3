"""The library does not need the extension module, and a module built from something else is not used (no GPU needed)."""
import pytest
import torch

from paper_2504_07878_b200 import binding, build


@pytest.mark.parametrize("error", [FileNotFoundError("g++"), RuntimeError("no Python.h"), ImportError("torch")])
def test_the_library_is_built_where_the_module_is_not(monkeypatch, capsys, error):
    calls = []

    def fail():
        calls.append("module")
        raise error

    monkeypatch.setattr(build, "build_library", lambda force, verbose: calls.append("library") or "the library")
    monkeypatch.setattr(build, "build_torch", fail)
    assert build.build(force=True) == "the library" and calls == ["library", "module"]
    assert "ctypes" in capsys.readouterr().err


def test_a_build_that_fails_leaves_no_old_module(monkeypatch, tmp_path):
    for name in ("TORCH_PATH", "TORCH_KEY"):
        monkeypatch.setattr(build, name, str(tmp_path / name))
        (tmp_path / name).write_text("old")
    monkeypatch.setattr(build, "TORCH_SOURCE", str(tmp_path / "none.cpp"))
    with pytest.raises(RuntimeError):
        build.build_torch()
    assert not list(tmp_path.iterdir())


def test_the_module_is_stale_when_anything_it_is_built_from_changes(monkeypatch, tmp_path):
    for name in ("TORCH_PATH", "TORCH_KEY"):
        monkeypatch.setattr(build, name, str(tmp_path / name))
    assert build.torch_is_stale()
    (tmp_path / "TORCH_PATH").write_text("")
    (tmp_path / "TORCH_KEY").write_text(build.torch_key())
    assert not build.torch_is_stale()
    (tmp_path / "include").mkdir()
    header = open(build.ROOT + "/include/tlr.h").read()
    (tmp_path / "include" / "tlr.h").write_text(header + "\n")
    with monkeypatch.context() as m:
        m.setattr(build, "ROOT", str(tmp_path))
        assert build.torch_is_stale()
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", "0.0")
        assert build.torch_is_stale()
    with monkeypatch.context() as m:
        m.setattr(build, "TORCH_FLAGS", build.TORCH_FLAGS + ["-g"])
        assert build.torch_is_stale()
    (tmp_path / "TORCH_PATH").unlink()
    assert build.torch_is_stale()


def test_a_module_built_for_another_torch_is_not_used(monkeypatch):
    build.build()
    for name in ("_native", "_extension"):
        monkeypatch.setattr(binding, name, None)
    assert "built-in" in repr(binding._native_route()) and binding._module()
    for name in ("_native", "_extension"):
        monkeypatch.setattr(binding, name, None)
    monkeypatch.setattr(torch, "__version__", "0.0")
    assert binding._native_route()(1, 2) is None and "built-in" not in repr(binding._native_route())
    assert not binding._module()
