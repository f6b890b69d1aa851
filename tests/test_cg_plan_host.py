"""The cluster solve's launches (cgcluster.cuh) when several threads plan and launch solves of different boxes: the
shared-memory limit of a kernel belongs to the process, so no thread may lower it under another's launch."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
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


@pytest.mark.parametrize("nr,nt", [(1, 1), (1, 40), (40, 1), (37, 53), (300, 200), (700, 400)])
@pytest.mark.parametrize("share", [0.0, 0.002, 0.3, 1.0])
def test_box_of_the_unknown_cells(shim, nr, nt, share):
    """The smallest box; of a region too large for any plan, some box that has none either."""
    rng = np.random.default_rng(nr + nt)
    for _ in range(5):
        mask = np.where(rng.random((nr, nt)) < share, 2, rng.integers(0, 2, (nr, nt))).astype(np.int8)
        mask[: rng.integers(0, nr), :] %= 2
        mask[:, : rng.integers(0, nt)] %= 2
        i, j = np.nonzero(mask == 2)
        want = [i.min(), i.max() + 1, j.min(), j.max() + 1] if i.size else [0, 0, 0, 0]
        got = (C.c_int * 4)()
        nc = shim.host_cg_box(mask.ctypes.data_as(C.c_void_p), nr, nt, got)
        if (want[1] - want[0]) * (want[3] - want[2]) <= 131072:
            assert list(got) == want
        else:
            assert nc == 0
