"""What the build compiles, and when (no compiler runs here)."""
import os
import subprocess

import pytest

from paper_2505_19115_b200 import build


@pytest.mark.parametrize("force", [False, True])
def test_the_c_library_is_built_where_the_extension_module_cannot_be(tmp_path, monkeypatch, force):
    compiled = []

    def no_module(*args, **kw):
        raise subprocess.CalledProcessError(1, "g++")
    monkeypatch.setattr(build, "OUT", str(tmp_path / "libnvfp4.so"))
    monkeypatch.setattr(build, "_compile", lambda out, *args, **kw: compiled.append(out) or out)
    monkeypatch.setattr(build, "build_calls", no_module)
    with pytest.raises(subprocess.CalledProcessError):
        build.build(force=force)
    assert compiled == [build.OUT]


def test_the_extension_module_is_built_again_for_another_pytorch_or_python(tmp_path, monkeypatch):
    import sysconfig
    import torch
    compiled = []

    def compile_module(cmd):
        compiled.append(cmd[0])
        open(build.CALLS_OUT, "w").close()
    monkeypatch.setattr(build, "CALLS_OUT", str(tmp_path / "_calls.so"))
    monkeypatch.setattr(build, "CALLS_BUILT_FOR", str(tmp_path / "_calls.so.built_for"), raising=False)
    monkeypatch.setattr(subprocess, "check_call", compile_module)
    build.build_calls()
    build.build_calls()
    assert len(compiled) == 1                               # built, and fresh
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    build.build_calls()
    build.build_calls()
    assert len(compiled) == 2
    variables = sysconfig.get_config_var
    monkeypatch.setattr(sysconfig, "get_config_var", lambda name: "cpython-399" if name == "SOABI" else variables(name))
    build.build_calls()
    build.build_calls()
    assert len(compiled) == 3
    os.remove(build.CALLS_BUILT_FOR)                        # a module of unknown origin
    build.build_calls()
    assert len(compiled) == 4
