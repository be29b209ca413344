"""The native argument marshalling is optional: the library builds and loads
without it, calls then take the Python path, and a module that was built for
another Python or torch is not loaded. (No GPU: no kernel is launched.)"""
import os
import subprocess
import sys
import sysconfig

import pytest
import torch

from paper_2401_13660_gb300 import build as b
from paper_2401_13660_gb300 import mbscan as mb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def elsewhere(tmp_path, monkeypatch):
    """A build into a folder of its own, without compilers: every command writes its -o file."""
    monkeypatch.setattr(b, "BUILD", str(tmp_path))
    monkeypatch.setattr(b, "LIB", str(tmp_path / "libmbscan.so"))
    monkeypatch.setattr(b, "BINDING", str(tmp_path / os.path.basename(b.BINDING)))
    ran = []

    def run(cmd, **kw):
        ran.append(os.path.basename(cmd[0]))
        if cmd[0] == "g++" and broken:
            return subprocess.CompletedProcess(cmd, 1, "", "no such header")
        with open(cmd[cmd.index("-o") + 1], "w"):
            return subprocess.CompletedProcess(cmd, 0, "", "")
    broken = [True]
    monkeypatch.setattr(b.subprocess, "run", run)
    return ran, broken


def test_the_library_builds_where_the_binding_does_not(elsewhere):
    ran, broken = elsewhere
    with pytest.warns(UserWarning, match="no such header"):
        assert b.build() == b.LIB
    assert os.path.exists(b.LIB) and not os.path.exists(b.BINDING)
    ran.clear()
    b.build()
    assert not ran   # not tried again for every process
    broken.clear()
    b.build(force=True)
    assert os.path.exists(b.BINDING) and b.up_to_date()
    os.remove(b.BINDING)
    assert not b.up_to_date()   # rebuilt, not an error


def test_the_name_tells_python_and_torch(monkeypatch, tmp_path):
    assert sysconfig.get_config_var("SOABI") in os.path.basename(b.BINDING)
    assert b.torch_dir() == os.path.dirname(torch.__file__)
    (tmp_path / "version.py").write_text("__version__ = '1.0'")
    monkeypatch.setattr(b, "torch_dir", lambda: str(tmp_path))
    assert b.binding_path() != b.BINDING


@pytest.mark.parametrize("found", [None, b"not a module"])
def test_calls_go_through_python_without_it(found, tmp_path):
    b.build()
    path = tmp_path / "_mbcall.so"
    if found:
        path.write_bytes(found)
    code = f"""
import warnings
import torch
from paper_2401_13660_gb300 import build, mbscan as mb
build.BINDING = {str(path)!r}
with warnings.catch_warnings(record=True) as w:
    warnings.simplefilter("always")
    mb.load_library(build_if_needed=False)
assert len(w) == 1 and "marshalled in Python" in str(w[0].message)
t = torch.zeros(1, 1, 8)
try:   # the Python path's own check
    mb.mb_step(t, t, torch.zeros(1, 1, 16), torch.zeros(1, 1, 15), torch.zeros(8, 16), t, torch.zeros(1, 8, 16))
except ValueError as e:
    assert "C: torch.float32 (1, 1, 15)" in str(e)
    print("ok")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT)
    assert r.stdout.strip() == "ok", r.stderr


def test_it_is_loaded_here():
    b.build()
    assert type(mb._native()).__name__ == "module"
