"""When the extension module of the autograd integration is compiled again (nothing is compiled here)."""
import os
import subprocess

import pytest
import torch

from paper_2110_15362_b200 import build


@pytest.fixture
def module(tmp_path, monkeypatch):
    """A module that looks built, and a compiler that writes an empty file."""
    path = tmp_path / "_autograd.so"
    path.write_bytes(b"")
    built = []

    def compile_(command):
        built.append(command)
        open(command[command.index("-o") + 1], "w").close()

    monkeypatch.setattr(build, "AUTOGRAD_PATH", str(path))
    monkeypatch.setattr(build, "AUTOGRAD_BUILT_FOR", str(tmp_path / "_autograd.built_for"), raising=False)
    monkeypatch.setattr(subprocess, "check_call", compile_)
    return tmp_path, built


@pytest.mark.parametrize("built_for", [None, "", "2.0.0", "this"])
def test_a_module_for_another_torch_is_built_again(module, built_for):
    tmp, built = module
    if built_for is not None:
        (tmp / "_autograd.built_for").write_text(torch.__version__ if built_for == "this" else built_for)
    assert build.build_autograd() == str(tmp / "_autograd.so")
    assert len(built) == (built_for != "this")
    assert build.autograd_built_for() == torch.__version__
    build.build_autograd()                                           # and then it stands
    assert len(built) == (built_for != "this")
    os.utime(tmp / "_autograd.so", (1, 1))                           # older than its source
    build.build_autograd()
    assert len(built) == (built_for != "this") + 1


def test_a_failed_build_is_not_taken_for_done(module, monkeypatch):
    tmp, built = module

    def fail(command):
        raise subprocess.CalledProcessError(1, command)

    monkeypatch.setattr(subprocess, "check_call", fail)
    for _ in range(2):
        with pytest.raises(subprocess.CalledProcessError):
            build.build_autograd()
    assert build.autograd_built_for() == ""
