"""The end-of-solve rule of the device-side conjugate gradients, compiled for the host (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_thread_of_a_launch_decides_alike(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "cg_state_checks")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2202_03655_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "cg_state_checks.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    lines = out.stdout.strip().splitlines()
    assert out.returncode == 0 and len(lines) == 14 and all(l.startswith("ok") for l in lines), out.stdout
