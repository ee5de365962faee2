"""The native marshalling module is optional: without it (or without one for the installed torch) every call takes its Python form."""
import sys

import pytest
import torch

import paper_1910_06188_b200 as package
from paper_1910_06188_b200 import binding, build


@pytest.fixture
def no_module_loaded(monkeypatch):
    build.build()
    monkeypatch.setattr(binding, "_native_module", None)
    monkeypatch.delattr(package, "_q8_native", raising=False)
    monkeypatch.delitem(sys.modules, package.__name__ + "._q8_native", raising=False)


def _takes_the_python_form():
    with pytest.raises(TypeError, match="grad_out must be a CUDA tensor"):  # (what the Python form says of a CPU tensor)
        binding.q8_ste_backward(torch.ones(4))


def test_calls_run_without_the_native_module(no_module_loaded, monkeypatch):
    monkeypatch.setitem(sys.modules, package.__name__ + "._q8_native", None)  # the import fails
    with pytest.warns(RuntimeWarning, match="marshalled in Python"):
        _takes_the_python_form()
    _takes_the_python_form()  # (says so once)


def test_the_library_is_built_where_the_native_module_cannot_be(monkeypatch, tmp_path):
    build.build()
    monkeypatch.setattr(build, "NATIVE", str(tmp_path / "missing.so"))
    for command in (["false"], [str(tmp_path / "no-such-compiler")]):
        monkeypatch.setattr(build, "_native_command", lambda: command)
        with pytest.warns(RuntimeWarning, match="was not built"):
            assert build.build() == build.LIB


def test_a_module_for_another_torch_is_rebuilt_and_not_used(no_module_loaded, monkeypatch):
    assert build._native_is_current()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not build._native_is_current()
    with pytest.warns(RuntimeWarning, match="built for torch"):
        _takes_the_python_form()
