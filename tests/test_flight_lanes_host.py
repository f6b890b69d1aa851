"""Every lane of a flight's pass (flight.cuh), those past the flight's last crossing among them, reads the face
tables only where they are: the results do not depend on what lies in front of and behind them."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_flight_host import CSRC, CUDA_INC, GRIDS, HERE, _rays


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not found")
    so = str(tmp_path_factory.mktemp("flight") / "flight_lanes.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CUDA_INC, "-I", CSRC,
                           "-I", os.path.join(HERE, "hostshim"), os.path.join(HERE, "hostshim", "flight_lanes_shim.cpp"),
                           "-o", so])
    return C.CDLL(so)


@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_lanes_read_inside_the_tables(shim, grid):
    rf, tf = GRIDS[grid]
    nr, nt = len(rf) - 1, len(tf) - 1
    n = 300
    p, u, cell = _rays(rf / rf[0], tf, n, np.random.default_rng(8))
    ptr = lambda a, t: a.ctypes.data_as(C.POINTER(t))  # noqa: E731
    rf_c, tf_c = np.ascontiguousarray(rf, np.float64), np.ascontiguousarray(tf, np.float64)
    out = []
    for pad, kind in ((0.25, 1), (7.0, 0), (float("nan"), -1)):
        o = np.zeros((n, 32, 5), np.float32)
        shim.host_flight_lanes(nr, nt, ptr(rf_c, C.c_double), ptr(tf_c, C.c_double), n, ptr(p, C.c_float),
                               ptr(u, C.c_float), ptr(cell, C.c_int), C.c_float(pad), kind, ptr(o, C.c_float))
        out.append(o)
    for o in out[1:]:
        assert np.array_equal(out[0], o, equal_nan=True)
