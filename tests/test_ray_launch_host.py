"""The ray tracer's launches (raytrace.cu) when several threads trace disks of different sizes: the shared-memory limit of a
kernel belongs to the process, so no launch may leave it below another's need."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_0902_3092_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    so = str(tmp_path_factory.mktemp("raylaunch") / "raylaunch.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           os.path.join(HERE, "hostshim", "ray_launch_shim.cu"), "-o", so])
    return C.CDLL(so)


@pytest.mark.parametrize("prec,sizes", [(32, [60, 1400, 2000, 5000, 8500]), (64, [60, 700, 1500, 4200])])
@pytest.mark.parametrize("nlam", [1, 40, 100, 256])
def test_launches_leave_the_limit_to_each_other(shim, prec, sizes, nlam):
    need = C.c_longlong()
    for a in sizes:
        limit = shim.host_ray_limit(prec, a, nlam, 48 * 1024, C.byref(need))
        assert need.value <= limit <= 227 * 1024
        for b in sizes:  # another thread's launch between this one's limit and its launch
            assert shim.host_ray_limit(prec, b, nlam, limit, C.byref(C.c_longlong())) >= need.value, (a, b)
