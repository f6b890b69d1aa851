"""The ray tracer's warp layout at its edges, against the FP64 oracle: bins per lane (1 to 256 bins, a full last lane and
one bin past it), rays per warp (1 to 20,000 rays: a lone ray, one past a warp's 32, many), optically thin and
thick dust (the segment's thin, thick and mixed branches), and visibilities in one part and in several. Tolerances are
test_gpu_raytrace.py's, for the reasons given there."""
import math

import numpy as np
import pytest

from test_gpu_raytrace import M, PC, RT, close_to, setup  # noqa: F401  (fixtures)
from paper_0902_3092_gb300 import disks

pytestmark = pytest.mark.gpu


def _disk(nlam, tau):
    return disks.make_disk(disks.log_r_faces(0.1, 100.0, 20), disks.midplane_refined_theta_faces(16), disks.paper_star(),
                           disks.gray_opacity(nlam), tau)


def _some(rays, n):
    k = np.linspace(0, rays.n - 1, n).astype(int)
    return type(rays)(rays.p[k].copy(), rays.q[k].copy(), rays.w[k].copy())


@pytest.mark.parametrize("nlam,tau,n", [(1, 30.0, 1), (31, 0.01, 33), (32, 1e5, 32), (33, 30.0, 200), (64, 1e5, 31),
                                        (65, 0.01, 65), (96, 30.0, 500), (100, 1e5, 129), (129, 30.0, 100),
                                        (192, 1e5, 40), (224, 30.0, 40), (256, 30.0, 40), (12, 30.0, 20000)])
def test_image_for_bins_and_rays(M, oracle, RT, nlam, tau, n):  # noqa: F811
    d = _disk(nlam, tau)
    g, T = setup(M, oracle, d)
    rays = _some(disks.polar_rays(d.r_faces_cm, n_sub=4, n_phi=224, n_inner=4), n)
    incl = 0.9
    g.set_rays(incl, 140 * PC, rays)
    look = np.unique(np.linspace(0, n - 1, min(n, 500)).astype(int))
    I_or = RT.image(d, T, incl, rays.p[look], rays.q[look])
    for prec, tol in ((64, 1e-9), (32, 3e-4)):
        out = g.raytrace(precision=prec, want_image=True)
        assert close_to(out["I"][look], I_or, tol), (prec, np.max(np.abs(out["I"][look] - I_or) / (I_or.max(0) + 1e-300)))
    g.close()


@pytest.mark.parametrize("n,n_vis", [(1, 1), (257, 1), (5000, 3), (300, 700)])
def test_visibilities_in_parts(M, oracle, RT, n, n_vis):  # noqa: F811
    d = _disk(40, 30.0)
    g, T = setup(M, oracle, d)
    rays = _some(disks.polar_rays(d.r_faces_cm, n_sub=2, n_phi=128, n_inner=4), n)
    dist = 140 * PC
    g.set_rays(math.pi / 4, dist, rays)
    I_or = RT.image(d, T, math.pi / 4, rays.p, rays.q)
    Fs = RT.star_flux(d, math.pi / 4, dist)
    k = np.arange(n_vis)
    bins, B, PA = list(k % 40), list(1e3 + 37.0 * k), list(0.01 * k)
    for prec, tol in ((64, 1e-9), (32, 2e-5)):
        g.raytrace(precision=prec)
        got = g.visibilities(bins, B, PA, with_star=True)
        for j in np.unique(np.linspace(0, n_vis - 1, 5).astype(int)):
            ref = RT.visibility(rays.p, rays.q, rays.w, I_or[:, bins[j]], dist, RT.bin_centre_cm(d, bins[j]), B[j], PA[j],
                                F_star=Fs[bins[j]])
            assert abs(got[j] - ref) < tol, (prec, j, got[j] - ref)
    g.close()
