"""The cluster solve's launches (cgcluster.cuh) when several threads plan and launch solves of different boxes: the
shared-memory limit of a kernel belongs to the process, so no thread may lower it under another's launch."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0902_3092_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    so = str(tmp_path_factory.mktemp("cgplan") / "cgplan.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I", CSRC, os.path.join(HERE, "hostshim", "cg_plan_shim.cu"), "-o", so])
    return C.CDLL(so)


BOXES = [(1, 1), (3, 40), (20, 30), (33, 20), (120, 32), (400, 30), (64, 60), (16, 150), (200, 90), (30, 1000), (60, 2000), (300, 400)]


def test_another_threads_plan_takes_no_memory_from_a_launch(shim):
    for a in BOXES:
        assert shim.host_cg_solve(*a, 0, 0) == 0  # alone
        for b in BOXES:
            assert shim.host_cg_solve(*a, *b) == 0, (a, b)
