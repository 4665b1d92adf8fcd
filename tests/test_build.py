"""The build: what counts as up to date, and what a failing compiler leaves behind."""
import subprocess
import sys

import pytest
import torch

from paper_2602_24082_b200 import build as B


def test_a_module_built_for_another_torch_or_python_is_not_up_to_date(monkeypatch):
    B.build()
    started = []
    monkeypatch.setattr(B.subprocess, "Popen", lambda cmd, **kw: started.append(cmd))
    assert B._start_ext(False) is None and not started
    here = B.ext_path()
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".post1")
    assert B.ext_path() != here and B._start_ext(False) is not None
    assert started[-1][started[-1].index("-o") + 1] == B.ext_path()
    monkeypatch.undo()
    monkeypatch.setattr(B.sysconfig, "get_config_var", lambda name: ".cpython-399-x86_64-linux-gnu.so")
    monkeypatch.setattr(B.subprocess, "Popen", lambda cmd, **kw: started.append(cmd))
    assert B._start_ext(False) is not None and len(started) == 2


def test_no_compiler_is_left_running_behind_one_that_fails():
    run = lambda code: subprocess.Popen([sys.executable, "-c", code], stdout=subprocess.PIPE,
                                        stderr=subprocess.STDOUT, text=True)
    procs = [(["first"], run("raise SystemExit(3)")), (["second"], run("import time; time.sleep(1)"))]
    with pytest.raises(RuntimeError, match="compiler failed: first$"):
        B._finish(procs, False)
    assert [p.poll() for _, p in procs] == [3, 0]
