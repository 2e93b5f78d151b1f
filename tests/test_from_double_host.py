"""Host (CPU) check of the float64 to fixed-point conversion at the end of its range:
tests/from_double_check.cpp."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


def test_from_double_reaches_its_bound(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "from_double_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", str(ROOT / "paper_2407_13012_gb300" / "csrc"),
                    str(ROOT / "tests" / "from_double_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip().endswith("OK")
