"""The native marshalling is an aid: builds and imports do without it, and another interpreter's module is not taken (runs without a GPU)."""
import os
import sysconfig

import pytest


def _built():
    from paper_1803_09877_b200 import build
    build.build()
    from paper_1803_09877_b200 import binding
    return build, binding


def test_build_without_python_headers(monkeypatch, tmp_path, capsys):
    build, _ = _built()
    monkeypatch.setattr(build.sysconfig, "get_paths", lambda: {"include": str(tmp_path)})
    monkeypatch.setattr(build, "NATIVE", str(tmp_path / "module.so"))
    assert build.build() == build.LIB
    assert not (tmp_path / "module.so").exists() and "Python.h" in capsys.readouterr().err


def test_module_is_named_after_its_interpreter(monkeypatch):
    build, binding = _built()
    assert os.path.basename(build.NATIVE) == "_native" + sysconfig.get_config_var("EXT_SUFFIX") != "_native.so"
    assert binding._native.__file__ == build.NATIVE
    monkeypatch.setattr(binding.sysconfig, "get_config_var", lambda name: ".another-interpreter.so")
    assert binding._load_native() is binding._CtypesCalls


def test_module_that_cannot_be_loaded(monkeypatch, tmp_path):
    _, binding = _built()
    (tmp_path / ("_native" + sysconfig.get_config_var("EXT_SUFFIX"))).write_bytes(b"not a module")
    monkeypatch.setattr(binding, "_PKG", str(tmp_path))
    with pytest.warns(RuntimeWarning, match="ctypes"):
        assert binding._load_native() is binding._CtypesCalls


@pytest.mark.parametrize("name,count", [("encode", 3), ("locate", 4), ("decode", 4), ("decode_update", 4), ("locate_decode", 5)])
def test_ctypes_makes_the_same_calls(name, count):
    _, binding = _built()
    tail = (0.5, 7) if name == "decode_update" else (7,)                    # (scale,) stream handle
    for calls in (binding._CtypesCalls, binding._native):
        with pytest.raises(binding.DracoError, match="invalid argument"):
            getattr(calls, name)(*([None] * count), *tail)
        with pytest.raises(binding.DracoError, match="invalid argument"):
            getattr(calls, name)(None, *([4096] * (count - 1)), *tail)
        with pytest.raises(AttributeError):
            getattr(calls, name)(None, object(), *([None] * (count - 2)), *tail)
        with pytest.raises(TypeError):
            getattr(calls, name)(*([None] * count))
