"""Non-gray temperatures and Rosseland means by the lanes of a warp (k_temperature, k_kappaR) against the oracle, at bin counts
around the warp's width and cell counts that do not fill the last warp."""
import numpy as np
import pytest

import mcstate as S
from paper_0902_3092_gb300 import disks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    return mcrt


@pytest.mark.parametrize("nr,nt,nlam", [(1, 2, 2), (3, 4, 31), (5, 2, 32), (9, 6, 33), (13, 10, 64), (11, 8, 65), (7, 14, 100)])
def test_temperatures_match_oracle(M, oracle, nr, nt, nlam):
    d = disks.make_disk(disks.log_r_faces(0.1, 100.0, nr), disks.midplane_refined_theta_faces(nt), disks.paper_star(),
                        disks.powerlaw_opacity(nlam), 1e4, h1_au=0.3)
    n_total = 10 ** 7
    tally, visits = S.random_tallies(d, nr + nlam, n_total)
    g = M.Disk.from_model(d)
    g.restore(S.blob(d, tally, visits, n_total))
    T, _, _ = g.temperatures()
    g.close()
    r = oracle.Run(d)
    r.tally[:] = tally
    r.n_total = n_total
    To, _ = r.temperatures()
    on = To > 0
    assert np.array_equal(T > 0, on)
    # sums of up to 100 bins of FP64 tail integrals (each exact to a few 2^-53 of the whole integral), a Newton root
    assert np.all(np.abs(T[on] / To[on] - 1) < 1e-12)
