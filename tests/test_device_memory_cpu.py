"""The memory the library keeps, what it takes host memory for and its side streams (csrc/device_memory.cu,
csrc/internal.h), compiled for the host against a fake of the CUDA calls: failing calls and odd address ranges without a device."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("device_memory") / "checks")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-DACCERL_KEEP_IDLE_MS=250", "-x", "c++", os.path.join(HERE, "device_memory_checks.cpp"), "-o", out,
                           "-I/usr/local/cuda/include", "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(ROOT, "paper_2211_15023_b200", "csrc")])
    return out


@pytest.mark.parametrize("check", ["reach", "busy", "pageable", "hungry", "idle", "in_use", "trim", "side"])
def test_device_memory(program, check):
    r = subprocess.run([program, check], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
