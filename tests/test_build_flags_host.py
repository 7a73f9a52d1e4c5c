"""How the library is compiled: the flags of every translation unit."""

import os
import subprocess
import types

from paper_2305_05055_gb300 import build


def test_device_code_is_not_packed(tmp_path, monkeypatch):
    """Packed device code would be unpacked inside the first call that needs it."""
    cmds = []

    def fake_run(cmd, **kw):
        cmds.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build, "OUT", str(tmp_path))
    monkeypatch.setattr(build, "LIB", os.path.join(str(tmp_path), "libcpma.so"))
    monkeypatch.setattr(build, "nvcc", lambda: "nvcc")
    monkeypatch.setattr(subprocess, "run", fake_run)
    build.build(force=True)
    units = [c for c in cmds if "-c" in c]
    assert len(units) == len(build.UNITS)
    assert all("--no-compress" in c for c in units)
