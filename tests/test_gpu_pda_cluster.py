"""The one-launch conjugate gradient of small PDA systems (cgcluster.cuh) through mcrt_pda_solve_static against a
sparse direct solve, at the edges of its plans: one cell, one row, one column, rows that do not divide among the
CTAs, every cells-per-thread count, the largest box and the first one beyond it (tile kernels), and a region with
holes and fixed cells inside."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    pytest.importorskip("torch")
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    return mcrt


def _system(nr, nt, holes, seed):
    rng = np.random.default_rng(seed)
    D = 10.0 ** rng.uniform(-1, 1, (nr, nt))
    mask = np.full((nr, nt), 1, np.int8)
    mask[1:-1, 1:-1] = 2
    if holes:
        mask[rng.random((nr, nt)) < 0.1] = 1
        mask[rng.random((nr, nt)) < 0.05] = 0
    Cr, Ct = np.zeros((nr, nt)), np.zeros((nr, nt))
    on = mask > 0
    Cr[:-1] = np.where(on[:-1] & on[1:], 2 / (1 / D[:-1] + 1 / D[1:]), 0.0)
    Ct[:, :-1] = np.where(on[:, :-1] & on[:, 1:], 2 / (1 / D[:, :-1] + 1 / D[:, 1:]), 0.0)
    # an unknown cell without a conducting face makes the system singular
    deg = Cr + Ct
    deg[1:] += Cr[:-1]
    deg[:, 1:] += Ct[:, :-1]
    mask[(mask == 2) & (deg == 0)] = 0
    u = np.where(mask == 1, rng.uniform(1e8, 1e9, (nr, nt)), 0.0)
    return mask, Cr, Ct, u


def _direct(mask, Cr, Ct, u):
    import scipy.sparse as sp
    import scipy.sparse.linalg as sl
    nr, nt = mask.shape
    n = nr * nt
    idx = np.arange(n).reshape(nr, nt)
    i = np.concatenate([idx[:-1].ravel(), idx[:, :-1].ravel()])
    j = np.concatenate([idx[1:].ravel(), idx[:, 1:].ravel()])
    c = np.concatenate([Cr[:-1].ravel(), Ct[:, :-1].ravel()])
    L = sp.coo_matrix((np.concatenate([c, c]), (np.concatenate([i, j]), np.concatenate([j, i]))), shape=(n, n)).tocsr()
    A = sp.diags(np.asarray(L.sum(1)).ravel()) - L
    un = (mask == 2).ravel()
    b = -(A[un][:, ~un] @ u.ravel()[~un])
    x = u.ravel().copy()
    x[un] = sl.spsolve(A[un][:, un].tocsc(), b)
    return x


@pytest.mark.parametrize("nr,nt,holes", [(3, 3, False), (3, 2500, False), (2500, 3, False), (35, 102, False), (66, 66, False),
                                         (67, 66, True), (19, 300, False), (132, 131, True), (260, 263, False),
                                         (200, 322, True), (362, 362, False), (400, 327, True), (4, 20000, False)])
def test_one_launch_cg_matches_direct_solve(M, nr, nt, holes):
    import torch
    mask, Cr, Ct, u = _system(nr, nt, holes, nr * 1000 + nt)
    ref = _direct(mask, Cr, Ct, u)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(a.ravel().copy()).to(dev) for a in (mask, Cr, Ct)]
    out = []
    for _ in range(2):
        x = torch.from_numpy(u.ravel().copy()).to(dev)
        torch.cuda.synchronize()
        it = M.pda_solve_static(nr, nt, *(a.data_ptr() for a in t), x.data_ptr())
        assert it > 0
        out.append(x.cpu().numpy())
    # the residual of the scaled system ends below 1e-12 of its right-hand side; its condition is at most about
    # (grid side)^2 times the contrast of D: 1e5 x 1e2
    assert np.max(np.abs(out[0] / np.where(ref != 0, ref, 1.0) - (ref != 0))) < 1e-12 * 1e7 / 10
    fixed = (mask != 2).ravel()
    assert np.array_equal(out[0][fixed], u.ravel()[fixed])
    if nr * nt < 100_000:  # one cluster: sums in a fixed order
        assert np.max(np.abs(out[0] / np.where(ref != 0, out[1], 1.0) - (ref != 0))) < 1e-12
