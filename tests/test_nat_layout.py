"""Host-side invariants of the natural-order staging layout (nat_word in
paper_2103_01767_gb300/csrc/team_fft.cuh) for all five FFT tiles: tests/nat_layout_check.cu,
compiled with nvcc for the host and run here (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not on PATH")
def test_natural_layout(tmp_path):
    exe = tmp_path / "nat_layout_check"
    subprocess.run(["nvcc", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2103_01767_gb300", "csrc"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "nat_layout_check.cu")], check=True, capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    lines = r.stdout.strip().splitlines()
    assert len(lines) == 5 and all(line.endswith(": 0 failed checks") for line in lines), r.stdout + r.stderr
    assert r.returncode == 0
