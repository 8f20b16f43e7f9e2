"""When the library and its extensions are rebuilt, and what a failed build leaves behind (no GPU needed)."""
import subprocess

import pytest
import torch

from paper_2608_15522_b200 import build


def test_extension_of_another_pytorch_is_rebuilt(monkeypatch):
    """The allocating extension is bound to the PyTorch that it was compiled against, which file times do not tell."""
    build.build_library()
    assert not build._stale()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build._stale()


def test_a_failed_compilation_leaves_no_compiler_running(monkeypatch, tmp_path):
    """A compiler that fails at once beside one that takes a second."""
    fails, runs = tmp_path / "fails", tmp_path / "runs"
    fails.write_text("#!/bin/sh\nexit 1\n")
    runs.write_text("#!/bin/sh\nexec sleep 1\n")
    fails.chmod(0o755)
    runs.chmod(0o755)
    started = []

    def start(cmd):
        started.append(subprocess.Popen([str(cmd)], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True))
        return started[-1]

    monkeypatch.setattr(build, "_nvcc", lambda: str(fails))
    monkeypatch.setattr(build, "_start_host_builds", lambda: [("a.cc", start(fails)), ("b.cc", start(runs))])
    with pytest.raises(RuntimeError, match="failed on"):
        build.build_library(force=True)
    ended = [p.poll() is not None for p in started]
    for p in started:
        p.wait()
    assert ended == [True, True]
