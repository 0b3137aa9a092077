"""What the launchers keep per device (shared-memory opt-ins, SM counts), on the CPU against a fake runtime."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1312_2880_gb300", "csrc")


def test_state_belongs_to_the_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("CUDA headers not found")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path / "device_state")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + CSRC, "-I" + include,
                    os.path.join(HERE, "device_state.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_no_launcher_keeps_a_flag_or_a_count_for_the_whole_process(name):
    text = open(os.path.join(CSRC, name)).read()
    assert not re.findall(r"static\s+(?:bool|int)\s+\w+\s*(?:\[\d*\]\s*)?=", text)
