"""The line-preconditioned one-launch conjugate gradient (cgcluster.cuh) at the edges of its shapes: columns per lane
(1, 2, 3, 5, 7, 9; a full last lane and one column past it), rows per warp, one CTA, CTAs of unequal rows, one row, one
column, holes, and couplings along theta up to 300 times those along r. The solution's scaled FP64 residual is what the
solver promises: at most 1e-8 of the right-hand side's (its acceptance at the rounding floor). Two solves give the
same bits: every sum of the inner solve has a fixed order."""
import numpy as np
import pytest

from test_gpu_pda_cluster import M, _system  # noqa: F401  (M is a fixture)

pytestmark = pytest.mark.gpu


def _residual(mask, Cr, Ct, x):
    r, deg = np.zeros_like(x), np.zeros_like(x)
    d = Cr[:-1] * (x[1:] - x[:-1])
    r[:-1] += d
    r[1:] -= d
    deg[:-1] += Cr[:-1]
    deg[1:] += Cr[:-1]
    d = Ct[:, :-1] * (x[:, 1:] - x[:, :-1])
    r[:, :-1] += d
    r[:, 1:] -= d
    deg[:, :-1] += Ct[:, :-1]
    deg[:, 1:] += Ct[:, :-1]
    un = mask == 2
    return np.linalg.norm(r[un] / np.sqrt(deg[un]))


@pytest.mark.parametrize("nr,nt,holes,stretch", [
    (3, 9, False, 300.0), (3, 290, False, 1.0), (90, 3, False, 300.0), (7, 34, True, 30.0), (34, 35, True, 300.0),
    (34, 66, False, 1.0), (34, 67, True, 30.0), (35, 98, False, 300.0), (35, 99, True, 1.0), (130, 162, False, 300.0),
    (100, 163, True, 30.0), (37, 226, True, 300.0), (200, 227, False, 30.0), (226, 290, True, 300.0), (227, 290, False, 1.0),
    (520, 30, True, 300.0), (1010, 34, False, 30.0), (700, 66, True, 300.0), (600, 90, False, 300.0)])
def test_line_preconditioned_solve(M, nr, nt, holes, stretch):  # noqa: F811
    import torch
    mask, Cr, Ct, u = _system(nr, nt, holes, nr * 1000 + nt)
    Ct = Ct * stretch
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(a.ravel().copy()).to(dev) for a in (mask, Cr, Ct)]
    out = []
    for _ in range(2):
        x = torch.from_numpy(u.ravel().copy()).to(dev)
        torch.cuda.synchronize()
        assert M.pda_solve_static(nr, nt, *(a.data_ptr() for a in t), x.data_ptr()) > 0
        out.append(x.cpu().numpy().reshape(nr, nt))
    assert _residual(mask, Cr, Ct, out[0]) <= 1e-8 * _residual(mask, Cr, Ct, u)  # (u is 0 on the unknown cells)
    assert np.array_equal(out[0], out[1])
    fixed = mask != 2
    assert np.array_equal(out[0][fixed], u[fixed])
