"""The device reductions run on the host, thread by thread (tests/native): what a CTA announces to the
others has to be stored by then, in any order in which its threads may have run, and a sum that FP64
adds exactly has to come out exactly."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cuda_include():
    for cand in (os.environ.get("CUDA_HOME"), "/usr/local/cuda"):
        if cand and os.path.exists(os.path.join(cand, "include", "cuda_runtime.h")):
            return os.path.join(cand, "include")
    pytest.skip("no CUDA headers")


def run_native(name, tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    exe = os.path.join(tmp_path, name)
    src = os.path.join(ROOT, "tests", "native", name + ".cpp")
    inc = [os.path.join(ROOT, "paper_1002_1505_gb300", "csrc"), os.path.join(ROOT, "include"), cuda_include()]
    cmd = ["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-o", exe, src] + ["-I" + i for i in inc]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-3000:]
    return subprocess.run([exe], capture_output=True, text=True, timeout=120)


def test_sums_keep_the_bits_of_fp64(tmp_path):
    res = run_native("reduction_bits", tmp_path)
    assert res.returncode == 0, res.stdout


def test_slot_is_stored_before_it_is_announced(tmp_path):
    res = run_native("reduction_order", tmp_path)
    assert res.returncode == 0, res.stdout
