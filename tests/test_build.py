"""What the build compiles, and when (no compiler runs here)."""
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
