"""What the build needs, without building."""
import subprocess

import pytest

from paper_1603_05279_b200 import build as b


def test_the_library_does_not_wait_for_the_python_binding(monkeypatch):
    """libxnor.so is compiled before, and whether or not, the torch extension beside it can be."""
    made = []

    def run(cmd, check):
        if b.PYEXT in cmd:
            raise subprocess.CalledProcessError(1, cmd)
        made.append(cmd[cmd.index("-o") + 1])

    monkeypatch.setattr(subprocess, "run", run)
    for bounds_check, lib in ((False, b.LIB), (True, b.LIB_CHECK)):
        monkeypatch.setattr(b, "up_to_date", lambda lib: False)
        monkeypatch.setattr(b, "build_pyext", lambda force=False: run([b.PYEXT], check=True))
        with pytest.raises(subprocess.CalledProcessError):
            b.build(force=True, bounds_check=bounds_check)
        assert made[-1] == lib
