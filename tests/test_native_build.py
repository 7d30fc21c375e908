"""The extension module of the binding belongs to one torch and one Python: another one makes build() compile it again, and
makes the binding refuse it (no GPU)."""
import pytest
import torch

from paper_2511_23225_b200 import binding, build


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def compiled(monkeypatch, tmp_path):
    """Whether build_native() calls the compiler, which is stood in for."""
    calls = []
    monkeypatch.setattr(build.subprocess, "check_call", lambda cmd: calls.append(cmd))
    monkeypatch.setattr(build.os, "replace", lambda a, b: None)
    real = open
    monkeypatch.setattr("builtins.open", lambda f, mode="r", *a, **k: real(tmp_path / "written", mode) if "w" in mode else real(f, mode, *a, **k))
    build.build_native()
    return len(calls)


def test_an_up_to_date_module_is_left_alone(monkeypatch, tmp_path):
    assert compiled(monkeypatch, tmp_path) == 0


def test_another_torch_compiles_it_again(monkeypatch, tmp_path):
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    assert compiled(monkeypatch, tmp_path) == 1


def test_another_python_compiles_it_again(monkeypatch, tmp_path):
    monkeypatch.setattr(build.sysconfig, "get_config_var", lambda name: ".cpython-0.so")
    assert compiled(monkeypatch, tmp_path) == 1


def test_the_binding_refuses_a_module_built_for_another_torch(monkeypatch):
    monkeypatch.setattr(binding, "_native_module", None)
    assert binding._native().BUILT_FOR == build.native_target()
    monkeypatch.setattr(binding, "_native_module", None)
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    with pytest.raises(RuntimeError, match="built for"):
        binding._native()
