"""The C++ half of the binding: found for this Python and this torch only, missed aloud, and never in the library's way."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2302_01425_b200 import binding, build


def test_the_file_belongs_to_one_python_and_one_torch():
    name = os.path.basename(build.bind_path())
    assert sys.implementation.cache_tag in name and torch.__version__ in name
    assert build.build_bind() == build.bind_path() and os.path.exists(build.bind_path())
    module, reason = binding._load_native(build.bind_path())
    assert reason is None and hasattr(module, "fwd_ex")


def test_what_cannot_be_loaded_gives_its_reason(tmp_path):
    assert binding._load_native(str(tmp_path / "none.so")) == (None, "not built")
    bad = tmp_path / "_tk_bind.so"
    bad.write_bytes(b"not a library")
    module, reason = binding._load_native(str(bad))
    assert module is None and reason and reason != "not built"


def test_a_missing_half_is_reported_once_per_load(monkeypatch):
    build.build()
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "_native_missing", "undefined symbol: x")
    monkeypatch.setattr(binding, "_lib", None)
    with pytest.warns(RuntimeWarning, match="undefined symbol: x"):
        binding.load()


@pytest.mark.parametrize("fails", [False, True])
def test_the_library_is_built_before_the_binding_and_without_it(tmp_path, monkeypatch, fails):
    built = []

    def run(cmd, check):
        assert check
        if fails and cmd[0] == "g++":
            raise subprocess.CalledProcessError(1, cmd)
        built.append(cmd[0])
        open(cmd[cmd.index("-o") + 1], "w").close()

    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setattr(build, "LIB", str(tmp_path / "libtk.so"))
    monkeypatch.setattr(build, "bind_path", lambda: str(tmp_path / "bind.so"))
    if fails:
        with pytest.warns(RuntimeWarning, match="ctypes"):
            assert build.build(force=True) == build.LIB
        assert built == ["nvcc"]
    else:
        assert build.build(force=True) == build.LIB
        assert built == ["nvcc", "g++"]
    assert os.path.exists(build.LIB)
