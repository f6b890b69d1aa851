"""The escape spectrum of a non-gray run by its bins against that of (almost) one packet after another, the method's order:
the packets that a run has in flight at once may not move it further than the transport kernel's packets in lanes did.

Bound: the mean over 16 seeds of the bins' differences, rms over the bins, in units of one run's Poisson error. With 100 packets
in lanes it is 0.24, with 100 in warps 0.48, of which 0.12 is the noise of the mean (32 seeds: 0.09): halfway, 0.37."""
import numpy as np
import pytest

from paper_0902_3092_gb300 import disks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    return mcrt


def test_spectrum_stays_near_one_packet_after_another(M):
    n = 300_000
    d = disks.make_disk(disks.log_r_faces(0.1, 100.0, 60), disks.midplane_refined_theta_faces(40), disks.paper_star(),
                        disks.powerlaw_opacity(60), 1e5)
    g = M.Disk.from_model(d)
    out = []
    for cap in (0, 12):
        s = []
        for k in range(16):
            g.reset()
            st = g.run_photons(n, seed=500 + k, mrw=True, gamma=2.0, max_events=10 ** 6, max_in_flight=cap)
            assert st["error_flags"] == 0 and st["escaped"] + st["capped"] == n
            s.append(g.sed().sum(axis=1) * n / d.star.L)
        out.append(np.array(s))
    g.close()
    a, b = out
    sel = b.mean(0) >= 20
    assert sel.sum() >= 40
    shift = (a - b).mean(0)[sel] / np.sqrt(b.mean(0)[sel])
    assert np.sqrt(np.mean(shift ** 2)) <= 0.37, shift
