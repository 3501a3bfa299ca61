"""Building and loading the library and its native binding (no GPU needed)."""
import os
import subprocess

import pytest
import torch

from paper_2605_19561_b200 import build, torq


@pytest.mark.parametrize("what", ["library", "binding"])
def test_a_file_appears_complete_or_not_at_all(monkeypatch, tmp_path, what):
    """The compiler writes beside the final name, under a name of this process; a failed build leaves nothing."""
    final = str(tmp_path / "out.so")
    monkeypatch.setattr(build, "LIB_PATH", final)
    monkeypatch.setattr(build, "binding_path", lambda: final)
    make = {"library": build.build_library, "binding": build.build_binding}[what]
    code = 1

    def compiler(cmd, **_):
        out = cmd[cmd.index("-o") + 1]
        assert out != final and os.path.dirname(out) == str(tmp_path) and str(os.getpid()) in os.path.basename(out)
        assert not os.path.exists(final)
        open(out, "w").write("x")
        return subprocess.CompletedProcess(cmd, code, "", "")

    monkeypatch.setattr(build.subprocess, "run", compiler)
    with pytest.raises(RuntimeError):
        make(force=True)
    assert os.listdir(tmp_path) == []
    code = 0
    assert make(force=True) == final
    assert os.listdir(tmp_path) == ["out.so"]


def test_a_binding_of_another_torch_is_not_used(monkeypatch):
    build.build_binding()
    assert not build.needs_binding()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build.needs_binding()


def test_the_library_loads_where_the_binding_cannot_be_built(monkeypatch):
    def no_compiler(*a, **k):
        raise FileNotFoundError("g++")

    monkeypatch.setattr(build, "build_binding", no_compiler)
    monkeypatch.setattr(torq, "_lib_handle", None)
    assert torq.torq_scales_bytes(128, 128) == 512
    with pytest.warns(UserWarning, match="native binding"):
        assert torq._layer_native() is None
