"""A packet's flight through 32 cells at a time (flight.cuh), compiled for the host and run lane by lane,
against the cells a ray crosses from every root of every face in FP64, on grids with thin rim shells, a
refined midplane, few cells, and an odd number of polar cells, for rays from the star, from cells at any
depth, along the axis and in the midplane."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_0902_3092_gb300 import disks

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_0902_3092_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not found")
    so = str(tmp_path_factory.mktemp("flight") / "flight.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CUDA_INC, "-I", CSRC,
                           "-I", os.path.join(HERE, "hostshim"), os.path.join(HERE, "hostshim", "flight_shim.cpp"),
                           "-o", so])
    return C.CDLL(so)


def _uniform_theta(nt):
    t = np.linspace(0.0, np.pi, nt + 1)
    t[-1] = np.pi
    return t


GRIDS = {
    "rim": (disks.rim_refined_r_faces(0.1, 100.0, 60), disks.midplane_refined_theta_faces(40)),
    "log": (disks.log_r_faces(0.1, 100.0, 100), disks.midplane_refined_theta_faces(60)),
    "thick": (disks.rim_refined_r_faces(0.1, 100.0, 200), disks.midplane_refined_theta_faces(120)),
    "odd": (disks.log_r_faces(0.1, 100.0, 33), _uniform_theta(7)),
    "one": (disks.log_r_faces(0.1, 100.0, 1), _uniform_theta(1)),
    "two": (disks.log_r_faces(0.1, 10.0, 2), _uniform_theta(2)),
}


def _rays(rf, tf, n, rng):
    """Points (unit: inner radius) in random cells, isotropic directions; then special rays."""
    nr, nt = len(rf) - 1, len(tf) - 1
    ir, it = rng.integers(0, nr, n), rng.integers(0, nt, n)
    r = rf[ir] + (rf[ir + 1] - rf[ir]) * rng.uniform(0.05, 0.95, n)
    th = tf[it] + (tf[it + 1] - tf[it]) * rng.uniform(0.05, 0.95, n)
    ph = rng.uniform(0, 2 * np.pi, n)
    p = np.stack([r * np.sin(th) * np.cos(ph), r * np.sin(th) * np.sin(ph), r * np.cos(th)], 1)
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    k = n // 5
    u[:k] = p[:k] / np.linalg.norm(p[:k], axis=1, keepdims=True)   # radially out
    u[k:2 * k] = -u[k:2 * k] * 0 - p[k:2 * k] / np.linalg.norm(p[k:2 * k], axis=1, keepdims=True) + 0.02 * u[k:2 * k]
    u[k:2 * k] /= np.linalg.norm(u[k:2 * k], axis=1, keepdims=True)  # nearly at the star
    u[2 * k:2 * k + 5] = [0, 0, 1]
    u[2 * k + 5:2 * k + 10] = [0, 0, -1]
    u[2 * k + 10:2 * k + 20, 2] = 0
    u[2 * k + 10:2 * k + 20] /= np.linalg.norm(u[2 * k + 10:2 * k + 20], axis=1, keepdims=True)
    return np.ascontiguousarray(p, np.float32), np.ascontiguousarray(u, np.float32), \
        np.ascontiguousarray(np.stack([ir, it], 1), np.int32)


def _reference(rf, tf, p, u):
    """Path length per cell from all crossings of the ray with all faces (FP64, the faces as the kernels
    hold them: rounded to FP32)."""
    nr, nt = len(rf) - 1, len(tf) - 1
    f32 = lambda x: np.asarray(x, np.float32).astype(np.float64)  # noqa: E731
    rf, C2, S2 = np.sqrt(f32(rf * rf)), f32(np.cos(tf) ** 2), f32(np.sin(tf) ** 2)
    tf = np.where(np.abs(tf - np.pi / 2) < 1e-12, np.pi / 2, np.arctan2(np.sqrt(S2), np.sign(np.pi / 2 - tf) * np.sqrt(C2)))
    p, u = p.astype(np.float64), u.astype(np.float64)
    b, r2, uu = p @ u, p @ p, u @ u
    eps = 2.0 ** -24
    s = [0.0]
    # rounding of a root of A s^2 + 2 B s + C by the rounding of its terms (absolute values a, b, c):
    # eps (a s^2 + 2 b s + c) / |2 (A s + B)|; it moves path length between the cells on both sides of the face
    tol_r, tol_t = np.zeros(nr + 2), np.zeros(nt + 2)

    def add(tol, k, x, A, B, a, bb, c):
        if x > 0 and np.isfinite(x):
            s.append(x)
            with np.errstate(divide="ignore"):
                e = eps * (a * x * x + 2 * bb * x + c) / abs(2 * (A * x + B))
            tol[k:k + 2] += min(8 * e, np.sqrt(c) + x)

    for k, R in enumerate(rf):
        d = b * b - uu * (r2 - R * R)
        if d >= 0:
            for x in ((-b - np.sqrt(d)) / uu, (-b + np.sqrt(d)) / uu):
                add(tol_r, k, x, uu, b, 1.0, np.sqrt(r2), r2 + R * R)
    for k, (t, cc, ss) in enumerate(zip(tf[1:-1], C2[1:-1], S2[1:-1])):
        A = cc * (u[0] ** 2 + u[1] ** 2) - ss * u[2] ** 2
        B = cc * (p[0] * u[0] + p[1] * u[1]) - ss * p[2] * u[2]
        Cc = cc * (p[0] ** 2 + p[1] ** 2) - ss * p[2] ** 2
        d = B * B - A * Cc
        if abs(t - np.pi / 2) < 1e-12:
            if u[2] != 0:
                add(tol_t, k + 1, -p[2] / u[2], 0.0, 0.5 * u[2], 0.0, abs(u[2]), abs(p[2]) + 1e-30)
        elif d >= 0:
            q = -(B + np.copysign(np.sqrt(d), B))
            for x in ([q / A] if A != 0 else []) + ([Cc / q] if q != 0 else []):
                add(tol_t, k + 1, x, A, B, 1.0, np.sqrt(r2), r2)
    s = np.unique([x for x in s if x >= 0 and np.isfinite(x)])
    m, L = 0.5 * (s[1:] + s[:-1]), np.diff(s)
    x = p[None, :] + m[:, None] * u[None, :]
    r = np.linalg.norm(x, axis=1)
    ir = np.searchsorted(rf, r, side="right") - 1
    it = np.clip(np.searchsorted(tf, np.arccos(np.clip(x[:, 2] / r, -1, 1)), side="right") - 1, 0, nt - 1)
    out = np.zeros((nr, nt))
    ok = (ir >= 0) & (ir < nr)
    np.add.at(out, (ir[ok], it[ok]), L[ok])
    # column and row sums shift by the roundings of their faces, on top of the positions' own
    base = 8 * eps * (L.sum() + np.sqrt(r2) + 1.0)
    return out, r2, tol_r[1:-1] + base, tol_t[1:-1] + base


@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_flight_cells_match_all_face_roots(shim, grid):
    rf_cm, tf = GRIDS[grid]
    rf = rf_cm / rf_cm[0]
    nr, nt = len(rf) - 1, len(tf) - 1
    n = 300
    p, u, cell = _rays(rf, tf, n, np.random.default_rng(5))
    p = np.concatenate([p, np.zeros((50, 3), np.float32)])  # from the star, through the cavity
    us = np.random.default_rng(6).standard_normal((50, 3))
    us /= np.linalg.norm(us, axis=1, keepdims=True)
    u = np.ascontiguousarray(np.concatenate([u, us.astype(np.float32)]))
    it = np.clip(np.searchsorted(tf, np.arccos(us[:, 2]), side="right") - 1, 0, nt - 1)
    cell = np.ascontiguousarray(np.concatenate([cell, np.stack([np.full(50, -1), it], 1)]).astype(np.int32))
    n += 50
    length = np.zeros((n, nr, nt))
    entries = np.zeros((n, nr, nt), np.int64)
    passes = np.zeros(n, np.int32)
    off = np.zeros(n)
    ptr = lambda a, t: a.ctypes.data_as(C.POINTER(t))  # noqa: E731
    rf_c, tf_c = np.ascontiguousarray(rf_cm, np.float64), np.ascontiguousarray(tf, np.float64)
    rc = shim.host_flights(nr, nt, ptr(rf_c, C.c_double), ptr(tf_c, C.c_double), n, ptr(p, C.c_float),
                           ptr(u, C.c_float), ptr(cell, C.c_int), ptr(length, C.c_double), ptr(entries, C.c_longlong),
                           ptr(passes, C.c_int), ptr(off, C.c_double))
    assert rc == 0
    # a pass ends inside the cell it names, to the roundings of the position (three, each 2^-24 of the radius)
    # and of the faces' tables
    assert off.max() <= 4 * 2.0 ** -24, off.max() * 2.0 ** 24
    for k in range(n):
        ref, r2, tol_r, tol_t = _reference(rf, tf, p[k], u[k])
        scale = max(1.0, np.sqrt(r2))
        # shells and polar rows separately: misassignments at a corner cancel in them
        for ax, tol in ((1, tol_r), (0, tol_t)):
            a, b = length[k].sum(ax), ref.sum(ax)
            assert np.all(np.abs(a - b) <= tol), (grid, k, ax, (np.abs(a - b) / tol).max())
        assert abs(length[k].sum() - ref.sum()) <= 64 * 2.0 ** -24 * (ref.sum() + scale), (grid, k)
        # every cell with a sizeable path was entered (the first one was not)
        big = ref > 1e-3 * scale
        ent = entries[k].copy()
        if cell[k, 0] >= 0:
            ent[cell[k, 0], cell[k, 1]] += 1
        assert np.all(ent[big] >= 1), (grid, k)
