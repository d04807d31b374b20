"""The library's build is reproducible: nvcc's split compilation divides a file among
threads, and which kernels got more registers' worth of spills changed from build to
build (a stand-alone data VJP kernel of 72 or 80 registers, 4 % apart)."""
import types

from paper_2401_09283_gb300 import build


def test_no_compile_command_depends_on_threads(monkeypatch, tmp_path):
    seen = []

    def run(cmd, **kw):
        seen.append(cmd)
        if "-o" in cmd:
            open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stderr="", stdout="")

    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setitem(build.VARIANTS, "release", (str(tmp_path), str(tmp_path / "lib.so"), []))
    build.build_library(force=True)
    compiled = [c for c in seen if "-c" in c]
    assert len(compiled) == len(build.SOURCES)
    assert not [a for c in compiled for a in c if "split-compile" in a or a == "-t" or "threads" in a]
