"""The network's launches on a process's second device (tests/native/two_devices.cpp): a kernel's opt-in
to more than 48 KB of shared memory holds for one device only.  Runs without a GPU."""
import os
import subprocess

import pytest

from paper_1002_1505_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("tensor_cores", ["1", "0"])
def test_every_device_is_opted_in(tmp_path, tensor_cores):
    obj = os.path.join(build.OUT_DIR, "unet.o")
    newest = max(os.path.getmtime(os.path.join(build.SRC, f)) for f in os.listdir(build.SRC))
    if not os.path.exists(obj) or os.path.getmtime(obj) < newest:
        os.makedirs(build.OUT_DIR, exist_ok=True)
        build._compile("unet.cu")
    exe = os.path.join(tmp_path, "two_devices")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    cmd = ["g++", "-std=c++17", "-O1", "-w", "-o", exe, os.path.join(ROOT, "tests", "native", "two_devices.cpp"), obj,
           "-I" + cuda, "-I" + os.path.join(ROOT, "include")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-3000:]
    env = dict(os.environ, DDA_UNET_TC=tensor_cores)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=120, env=env)
    assert res.returncode == 0, res.stdout
