"""The in-tree build recompiles a source when any header beside it changes (.h and .cuh), and only then.  The compiler
is replaced by a stand-in that writes the output file and notes the source."""
import os
import types

import pytest

import paper_2507_18282_gb300.build as B


@pytest.mark.parametrize("header", ["ew_a.h", "ew_b.cuh"])
def test_header_change_recompiles(tmp_path, monkeypatch, header):
    src = tmp_path / "csrc"
    src.mkdir()
    for name in ("k.cu", "ew_a.h", "ew_b.cuh"):
        (src / name).write_text("")
        os.utime(src / name, (1000, 1000))
    monkeypatch.setattr(B, "CSRC", str(src))
    monkeypatch.setattr(B, "BUILD", str(tmp_path / "build"))
    monkeypatch.setattr(B, "LIB", str(tmp_path / "build" / "libew.so"))
    monkeypatch.setattr(B, "_nvcc", lambda: "nvcc")
    compiled = []

    def fake(cmd, **kw):
        if "-c" in cmd:
            compiled.append(os.path.basename(cmd[cmd.index("-c") + 1]))
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(B.subprocess, "run", fake)
    B.build()
    assert compiled == ["k.cu"]
    B.build()
    assert compiled == ["k.cu"]
    obj = os.path.join(B.BUILD, "k.cu.o")
    t = os.path.getmtime(obj)
    os.utime(src / header, (t + 10, t + 10))
    B.build()
    assert compiled == ["k.cu", "k.cu"]
