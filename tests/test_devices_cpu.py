"""Launches of one process on two devices, checked on the host against stand-ins for the CUDA
runtime's functions (two_devices.cu, fake_cudart.cpp): the shared-memory allowance of a kernel and the sizes taken
from the number of multiprocessors belong to a device, not to the process."""
import glob
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1412_2629_gb300 import build as B
    B.build()
    objects = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    if not all(map(os.path.exists, objects)):
        B.build(force=True)
    out = str(tmp_path_factory.mktemp("devices") / "two_devices")
    cuda = os.path.dirname(os.path.dirname(B.nvcc()))
    lib = [d for d in (os.path.join(cuda, "lib64"), *glob.glob(os.path.join(cuda, "targets", "*", "lib")))
           if os.path.exists(os.path.join(d, "libcudart.so"))]
    cmd = [B.nvcc(), *B.ARCH, "-O1", "-std=c++17", "-I" + B.INCLUDE, "-I" + B.CSRC, os.path.join(HERE, "two_devices.cu"),
           os.path.join(HERE, "fake_cudart.cpp"), *objects, "-cudart", "shared", "-Xlinker", "-rpath," + lib[0], "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("mode", ["map", "no-map"])
def test_launches_on_two_devices(program, mode):
    r = subprocess.run([program, mode], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
