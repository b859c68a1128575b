"""LSLU_PROJ_TIMING's phase times of the projected solve, for a problem of each of the two
bidiagonalisations (registers up to 63 columns, shared memory above): every phase has run,
and together they take no longer than the call."""
import os
import re
import subprocess
import sys

import pytest

from paper_2409_05239_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("k", [20, 63, 64])
def test_every_phase_is_timed(k):
    build.build()
    env = dict(os.environ, LSLU_PROJ_TIMING="1")
    cmd = [sys.executable, "-m", "paper_2409_05239_gb300.solve_once", "--workload", "ct32",
           "--value-type", "f64", "--K", str(k), "--repeat", "3"]
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = r.stderr.splitlines()
    total = [x for x in lines if x.startswith(f"lslu projected k={k}:")]
    parts = [x for x in lines if "bidiag sections:" in x]
    assert len(total) == len(parts) == 3
    phases = [float(x) for x in re.findall(r"(-?[\d.]+) us", total[-1])]
    sections = [float(x) for x in re.findall(r" (-?[\d.]+)(?:,| us)", parts[-1])]
    assert len(phases) == 5 and len(sections) == 4
    assert all(0.0 < x < 1e5 for x in phases + sections), (phases, sections)
    assert sum(sections) <= phases[0] + 0.3  # printed to 0.1
