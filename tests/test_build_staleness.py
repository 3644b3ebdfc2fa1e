"""The build decides what is out of date: the extension is compiled again when it was built for another PyTorch version."""
import importlib.metadata
import subprocess
import types

from paper_2508_20407_b200 import build


def test_extension_follows_the_pytorch_version(monkeypatch, tmp_path):
    compiled = []

    def run(cmd, **kwargs):                       # nothing is compiled here, only the files appear: the decisions are looked at
        compiled.append(cmd[0])
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    for name, path in (("OBJ", tmp_path), ("LIB", tmp_path / "lib.so"), ("FASTCALL", tmp_path / "ext.so")):
        monkeypatch.setattr(build, name, str(path))
    monkeypatch.setattr(subprocess, "run", run)

    def extension_compiled():
        compiled.clear()
        build.build()
        return "g++" in compiled

    monkeypatch.setattr(importlib.metadata, "version", lambda name: "2.0")
    assert extension_compiled()
    assert not extension_compiled()
    monkeypatch.setattr(importlib.metadata, "version", lambda name: "2.1")
    assert extension_compiled()
    assert not extension_compiled()
