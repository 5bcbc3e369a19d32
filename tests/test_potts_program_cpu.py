"""tests/host/potts_check.cpp, compiled with g++ against the planner and program builder:
the chains of Potts programs with and without small runs (no GPU)."""
import subprocess

import pytest

from test_host_cpu import _build_check


@pytest.mark.timeout(300)
def test_potts_programs_without_runs_keep_their_tiles(tmp_path):
    exe = _build_check(tmp_path, "potts_check")
    r = subprocess.run([exe], capture_output=True, text=True, timeout=240)
    assert r.returncode == 0, r.stdout + r.stderr
    last = r.stdout.strip().splitlines()[-1].split()
    assert int(last[1]) == 30 and int(last[3]) > 100 and last[5] == "0"
