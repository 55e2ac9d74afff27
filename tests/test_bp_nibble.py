"""The expand sweep's distance test on nibble rows (csrc/bp_nibble.h) against
plain sums of distances, compiled here with g++ (tests/bp_nibble_check.cpp)."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]


def test_nibble_rows_equal_plain_sums(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = tmp_path / "bp_nibble_check"
    subprocess.run([gxx, "-O2", "-std=c++17", f"-I{ROOT / 'paper_1304_4661_gb300' / 'csrc'}",
                    str(ROOT / "tests" / "bp_nibble_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok ")
