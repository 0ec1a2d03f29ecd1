"""Accuracy of the compile-time FP32 transforms, run on the host (tests/native/fft_accuracy.cpp)."""
from test_native_reductions import run_native


def test_transforms_lose_no_accuracy_to_their_split(tmp_path):
    res = run_native("fft_accuracy", tmp_path)
    assert res.returncode == 0, res.stdout
