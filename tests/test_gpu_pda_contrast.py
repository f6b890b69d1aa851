"""Diffusion systems whose neighbouring cells differ by up to 1e8 and 1e12 in D, more than the float scalars of the cluster's
inner solve carry: the solve ends, below its acceptance level (a scaled residual of 1e-8 of the right-hand side's), as with the
tile kernels' FP64 sums."""
import numpy as np
import pytest

from test_gpu_pda_cluster import M  # noqa: F401  (a fixture)
from test_gpu_pda_lines import _residual

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nr,nt,decades,stretch,kw", [
    (40, 40, 6, 1.0, {}), (40, 40, 6, 1.0, dict(inner_tol=1e-3)), (120, 30, 6, 1.0, {}),
    (64, 200, 4, 100.0, {}), (64, 200, 4, 100.0, dict(inner_tol=1e-7)), (200, 64, 4, 0.01, dict(inner_tol=1e-3)),
    (12, 11, 6, 0.01, {}), (40, 40, 0.5, 1.0, dict(max_outer=1, tol=1e-4))])
def test_solve_of_a_system_of_high_contrast(M, nr, nt, decades, stretch, kw):  # noqa: F811
    import torch
    rng = np.random.default_rng(nr * nt)
    D = 10.0 ** rng.uniform(-decades, decades, (nr, nt))
    mask = np.full((nr, nt), 1, np.int8)
    mask[1:-1, 1:-1] = 2
    Cr, Ct = np.zeros((nr, nt)), np.zeros((nr, nt))
    Cr[:-1] = 2 / (1 / D[:-1] + 1 / D[1:])
    Ct[:, :-1] = stretch * 2 / (1 / D[:, :-1] + 1 / D[:, 1:])
    u = np.where(mask == 1, rng.uniform(1e8, 1e9, (nr, nt)), 0.0)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(a.ravel().copy()).to(dev) for a in (mask, Cr, Ct)]
    x = torch.from_numpy(u.ravel().copy()).to(dev)
    torch.cuda.synchronize()
    assert M.pda_solve_static(nr, nt, *(a.data_ptr() for a in t), x.data_ptr(), **kw) > 0
    x = x.cpu().numpy().reshape(nr, nt)
    assert _residual(mask, Cr, Ct, x) <= max(1e-8, kw.get("tol", 0.0)) * _residual(mask, Cr, Ct, u)
    assert np.array_equal(x[mask == 1], u[mask == 1])
