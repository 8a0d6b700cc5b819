"""Shared memory limits are raised on every device a kernel is launched on: the
launch code against a small stand-in for the CUDA runtime with two devices."""
import os
import subprocess

from paper_1210_2536_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_second_device_gets_its_limits(tmp_path):
    cc = _build.nvcc()
    objs = []
    for name in ("mlp", "staged"):
        objs.append(str(tmp_path / f"{name}.o"))
        subprocess.check_call([cc] + _build.NVCC_FLAGS + ["-c", os.path.join(_build.CSRC, f"{name}.cu"), "-o", objs[-1]])
    exe = str(tmp_path / "fake_devices")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(cc))), "include")
    subprocess.check_call(["g++", "-std=c++17", "-I", inc, "-I", _build.INCLUDE, "-I", _build.CSRC,
                           os.path.join(HERE, "fake_devices.cpp"), *objs, "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
