"""When an engine's delivery mode may change and what the tuner's last turns
decide, compiled on the host with g++ (the header has no CUDA dependency)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_switch_steps_and_verdict(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    exe = str(tmp_path / "turns_test")
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror",
                    "-I", os.path.join(ROOT, "paper_2211_15963_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "turns_test.cc"), "-o", exe],
                   check=True, capture_output=True, timeout=300)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
