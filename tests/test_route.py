"""The rules that choose a solver (csrc/route.h), compiled with the host C++
compiler."""
from __future__ import annotations

import subprocess

from test_host_parts import _compile


def test_lines_between_the_solvers(tmp_path_factory):
    exe = _compile(tmp_path_factory, "route_check")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
