"""Builds tests/device/split_check.cu against the kernels' headers."""
import ctypes
import os
import subprocess

from paper_1807_00370_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp_dir):
    so = os.path.join(str(tmp_dir), "split_check.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-o", so,
                    os.path.join(HERE, "device", "split_check.cu")], check=True)
    lib = ctypes.CDLL(so)
    lib.split_value_host.restype = ctypes.c_double
    lib.mixed_step_cost_host.restype = ctypes.c_double
    return lib
