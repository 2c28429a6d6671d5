"""The build without what only the extension module needs."""
import os
import subprocess
import sysconfig

import pytest

from paper_1709_04060_b200 import build


def test_extension_is_named_for_its_interpreter():
    assert os.path.basename(build.FASTCALL) == "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX")


@pytest.mark.parametrize("fault", ["no compiler", "no headers"])
def test_build_goes_on_without_the_extension(monkeypatch, tmp_path, capsys, fault):
    run = subprocess.run

    def gcc_fails(cmd, **kw):
        if cmd[0] == "gcc":
            if fault == "no compiler":
                raise FileNotFoundError("gcc")
            if kw.get("check"):
                raise subprocess.CalledProcessError(1, cmd)
            return subprocess.CompletedProcess(cmd, 1, "", "Python.h: No such file or directory")
        return run(cmd, **kw)

    build.build()                                    # the library itself is up to date from here on
    stale = tmp_path / os.path.basename(build.FASTCALL)
    stale.write_bytes(b"made from an older source")
    os.utime(stale, (0, 0))
    monkeypatch.setattr(build, "FASTCALL", str(stale))
    monkeypatch.setattr(subprocess, "run", gcc_fails)
    assert build.build() == build.LIB
    assert not stale.exists()
    assert "ctypes" in capsys.readouterr().err
