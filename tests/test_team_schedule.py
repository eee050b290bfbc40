"""The exchange buffers of the team evolver (host logic, no GPU).

team_schedule.h says which buffer each step of team.cu writes and reads;
tests/team_schedule_check.cpp compiles it with the host compiler and checks
that no two accesses of a buffer, one of them a write, are left unordered by
the barriers and arrivals of the exchange (see its header).
"""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_team_exchange_buffers(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    exe = tmp_path / "team_schedule_check"
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1103_1399_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "team_schedule_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
