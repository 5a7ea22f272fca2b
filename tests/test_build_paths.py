"""Where the build finds the toolkit (CPU only)."""
from types import SimpleNamespace

import pytest

from paper_2402_18668_b200 import build as b


@pytest.mark.parametrize("how", ["NVCC", "PATH", "link"])
def test_extension_takes_the_headers_of_its_compiler(tmp_path, monkeypatch, how):
    root = tmp_path / "toolkit"
    (root / "bin").mkdir(parents=True)
    (root / "include").mkdir()
    (root / "include" / "cuda_runtime_api.h").touch()
    nvcc = root / "bin" / "nvcc"
    nvcc.touch(mode=0o755)
    monkeypatch.delenv("NVCC", raising=False)
    if how == "PATH":
        monkeypatch.setattr(b, "_nvcc", lambda: "nvcc")
        monkeypatch.setenv("PATH", str(root / "bin"))
    else:
        if how == "link":
            (tmp_path / "bin").mkdir()
            (tmp_path / "bin" / "nvcc").symlink_to(nvcc)
            nvcc = tmp_path / "bin" / "nvcc"
        monkeypatch.setenv("NVCC", str(nvcc))
    monkeypatch.setattr(b, "OBJ", tmp_path)
    monkeypatch.setattr(b, "NATIVE", tmp_path / "_native.so")
    commands = []

    def run(cmd, **kw):
        commands.append(cmd)
        return SimpleNamespace(returncode=0, stdout="", stderr="")
    monkeypatch.setattr(b.subprocess, "run", run)
    monkeypatch.setattr(b.os, "replace", lambda *a: None)
    b.build_native()
    assert str(root / "include") in commands[-1] and "/usr/local/cuda/include" not in commands[-1]
