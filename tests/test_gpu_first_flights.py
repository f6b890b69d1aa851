"""First flights found at once (k_star_flights) against the packets' marches: a gray plain run with the tail
kernel takes them, the repeatable form (tail_warps = -1) marches. Same packets, same random blocks, each dropped
after its first interaction (an event cap of 1): the same cells up to the packets whose flight ends within a
rounding of a face."""
import numpy as np
import pytest

from paper_0902_3092_gb300 import disks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    return mcrt


def _disk(nr, nt, tau, hole=False):
    tf = np.linspace(0.0, np.pi, nt + 1) if nt % 2 else disks.midplane_refined_theta_faces(nt)
    tf[-1] = np.pi
    d = disks.make_disk(disks.log_r_faces(0.1, 100.0, nr), tf, disks.paper_star(), disks.gray_opacity(13), tau, h1_au=0.2)
    if hole:  # dust-free shells inside and at both ends of the disk
        d.rho[: nr // 5] = 0.0
        d.rho[nr // 2: nr // 2 + 2] = 0.0
        d.rho[-1] = 0.0
    return d


@pytest.mark.parametrize("nr,nt,tau,hole,n", [(1, 1, 3.0, False, 5000), (2, 3, 0.0, False, 1000), (31, 8, 10.0, False, 1),
                                              (32, 7, 10.0, False, 33), (33, 20, 300.0, True, 200_000),
                                              (40, 40, 100.0, False, 1_000_000), (200, 60, 1000.0, False, 300_000)])
def test_first_flights_match_marches(M, nr, nt, tau, hole, n):
    d = _disk(nr, nt, max(tau, 1e-30), hole)
    out = []
    for tail in (0, -1):
        g = M.Disk.from_model(d)
        for part in range(2):  # the second run adds to the first one's tallies
            st = g.run_photons(n, seed=11, first_id=part * n, n_total=2 * n, tail_warps=tail, max_events=1)
            assert st["packets"] == n and st["escaped"] + st["capped"] == n and st["error_flags"] == 0
        out.append((g.tallies(), g.sed().sum(axis=0), st["crossings"]))
        g.close()
    (a, sa, ca), (b, sb, cb) = out
    # a march rounds its position and optical depth about once per shell, 2^-24 of them each: of the flights,
    # up to nr x 2^-23 end on the other side of a face (16 times that allowed, and two packets)
    slack = 2 + 16 * 2 * n * nr * 2.0 ** -23
    for x, y in zip(a, b):
        scale = 65536.0 if x is a[0] else 1.0
        moved = np.abs(x.astype(float) - y.astype(float)).sum() / 2 / scale
        assert moved <= slack * (nr + 1 if x is a[1] else 1), (moved, slack)
    assert abs(ca - cb) <= slack * (nr + 1)
    assert np.abs(sa - sb).sum() <= 2 * slack * d.star.L / (2 * n)
