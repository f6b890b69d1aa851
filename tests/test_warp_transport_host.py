"""The transport with one packet per warp (run_packet_warp, fly_warp, interact_now, mrw_chain_now of transport.cuh) with 32 lanes
on the host, each a coroutine that meets the others at every warp operation."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_0902_3092_gb300 import disks

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not found")
    out = tmp_path_factory.mktemp("warp") / "libwarptransport.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CUDA_INC,
                           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_0902_3092_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "hostshim", "warp_transport_shim.cpp"), "-o", str(out)])
    return C.CDLL(str(out))


def run(lib, d, n, seed, nmin=20, exit_dir=0, mueller=None, keep_j=False, late=None):
    op, nc = d.opacity, d.nr * d.ntheta
    out = {k: np.zeros(nc, np.uint64) for k in ("tally", "visits", "nabs")}
    out["sed"], out["cnt"] = np.zeros(op.nlam * 10, np.uint64), np.zeros(8, np.uint64)
    out["j"] = np.zeros(nc * op.nlam) if keep_j else None
    arrs = [np.ascontiguousarray(x, np.float64) for x in
            (d.r_faces_cm, d.theta_faces, d.rho.ravel(), op.lam_edges_um, op.kappa_abs, op.kappa_sca, op.g)]
    mu = None if mueller is None else np.ascontiguousarray(mueller, np.float64)
    P = lambda x: None if x is None else x.ctypes.data_as(C.c_void_p)  # noqa: E731
    out["parted"] = lib.host_warp_transport(
        C.c_int(d.nr), C.c_int(d.ntheta), P(arrs[0]), P(arrs[1]), P(arrs[2]), C.c_int(op.nlam), P(arrs[3]), P(arrs[4]),
        P(arrs[5]), P(arrs[6]), C.c_double(d.star.T_K), C.c_double(d.star.R_cm), C.c_uint64(n), C.c_uint64(seed), C.c_int(1),
        C.c_double(2.0), C.c_int(nmin), C.c_int(exit_dir), C.c_int(0 if mu is None else mu.shape[-1]), P(mu), None, P(late),
        P(out["tally"]), P(out["visits"]), P(out["nabs"]), P(out["sed"]), P(out["j"]), P(out["cnt"]))
    return out


@pytest.mark.parametrize("form", ["nongray", "nongray_j", "nongray_polarized", "gray_j_outward"])
def test_lanes_agree_on_a_tally_that_other_packets_change(lib, form):
    """What a warp does next may depend on a cell's tally, which other packets' deposits change between two loads of it: all
    lanes have to go by one load. Here the loads of lanes 1 .. 31 find other values than lane 0's (hundreds of packet energies
    where it finds few): the lanes stay together, and nothing changes."""
    d = disks.config_nongray(16, 16, 1e5) if form.startswith("nongray") else disks.config_thick_gray(30, 20, 1e4)
    kw = dict(nmin=3, keep_j="_j" in form, exit_dir=1 if form.endswith("outward") else 0,
              mueller=disks.rayleigh_mueller(d.opacity.nlam, 31) if form.endswith("polarized") else None)
    n = 300
    a = run(lib, d, n, 5, **kw)
    assert a["parted"] == 0 and a["cnt"][0] == n and a["cnt"][6] == n and a["cnt"][4] > 20 and a["cnt"][7] == 0
    late = np.full(d.nr * d.ntheta, 700 * 65536, np.uint64)
    b = run(lib, d, n, 5, late=late, **kw)
    assert b["parted"] == 0
    for k in ("tally", "visits", "nabs", "sed", "cnt"):
        assert np.array_equal(a[k], b[k]), k
    if a["j"] is not None:
        assert np.array_equal(a["j"], b["j"])


def test_counters_of_a_long_run_do_not_wrap(lib):
    """A warp that makes a run's packets one after another passes 2^32 crossings."""
    each, times = (700_000_000, 90_000_000, 80_000_000, 3), 60
    cnt, at = np.zeros(64, np.uint64), np.zeros(5, np.int32)
    lib.host_counter_places(at.ctypes.data_as(C.c_void_p))
    lib.host_counters(C.c_int(times), *(C.c_uint(x) for x in each), cnt.ctypes.data_as(C.c_void_p))
    assert [int(cnt[i]) for i in at] == [times] + [times * x for x in each]
