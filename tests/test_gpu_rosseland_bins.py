"""Rosseland means by the lanes of a warp (k_kappaR) at bin counts around the warp's width: the PDA of a non-gray disk whose
conductances need them, against the oracle's direct solve on the exact means."""
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


@pytest.mark.parametrize("nlam", [2, 31, 32, 33, 64, 65, 100])
def test_pda_on_rosseland_means(M, oracle, nlam):
    nr, nt = 23, 22  # 506 cells: the last block's last warp has 26
    d = disks.make_disk(disks.log_r_faces(0.1, 100.0, nr), disks.midplane_refined_theta_faces(nt), disks.paper_star(),
                        disks.powerlaw_opacity(nlam), 1e6)
    tally, visits = S.state_for(d, S.wanted_T(d), S.midplane_band(d))
    g = M.Disk.from_model(d)
    g.restore(S.blob(d, tally, visits, 10 ** 6))
    n_pda, _ = g.solve_pda()
    T = g.temperatures(M.T_PDA)[0]
    r = oracle.Run(d)
    r.tally[:] = tally
    r.n_total = 10 ** 6
    To_mc, eo = r.temperatures()
    To, mask, _, _ = oracle.solve_pda(d, To_mc, tally, visits, eo)
    assert n_pda == int(mask.sum()) > 20
    # the parity tolerance of the PDA (its residual is 1e-12 of the right-hand side, the means are exact to some 1e-15)
    assert np.max(np.abs(T[mask] / To[mask] - 1)) < 1e-6
    # and the means matter: with one mean for all cells the solution is another one
    op = d.opacity
    flat = np.full(d.rho.shape, float(np.mean(op.kappa_abs + (1 - op.g) * op.kappa_sca)))
    g.solve_pda(kappa_R=flat)
    if nlam > 2:
        assert np.max(np.abs(g.temperatures(M.T_PDA)[0][mask] / To[mask] - 1)) > 1e-4
    g.close()
