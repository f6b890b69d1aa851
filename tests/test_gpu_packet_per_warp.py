"""Non-gray runs and batches with one packet per warp (transport_warp_kernel) against the forms with a packet per lane: which runs
take which, gray models among non-gray ones, the tail of a run in lanes, and the edges of the kernel's range."""
import numpy as np
import pytest

from paper_0902_3092_gb300 import disks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    return mcrt


def _disk(nr, nt, tau, nlam=24, gray=False, g=0.6):
    tf = np.linspace(0.0, np.pi, nt + 1) if nt < 16 else disks.midplane_refined_theta_faces(nt)
    tf[-1] = np.pi
    op = disks.gray_opacity(nlam) if gray else disks.powerlaw_opacity(nlam, g=g)
    return disks.make_disk(disks.log_r_faces(0.1, 100.0, nr), tf, disks.paper_star(), op, tau, h1_au=0.2)


@pytest.mark.parametrize("tau,with_gray,cap,warps", [
    (1e3, False, 0, 33),          # 100,000 packets / 3000
    (1e5, False, 0, 11),          # an optically thick disk: a third of them
    (1e3, False, 1, 1),
    (1e3, False, 2000, 2000),
    (1e3, False, 19_456, 2432),   # 8 x 152 x 16 allowed: the warps that the device holds
    (1e3, False, 19_457, None),   # more of them in lanes
    (1e3, True, 9728, 2432),      # with a gray disk 4 x 152 x 16
    (1e3, True, 9729, None),
    (1e3, False, 100_000, None),
])
def test_packets_allowed_in_flight_decide_between_warps_and_lanes(M, tau, with_gray, cap, warps):
    gs = [M.Disk.from_model(_disk(20, 20, tau)), M.Disk.from_model(_disk(20, 20, 30.0, gray=with_gray))]
    B = M.Batch(gs, [60_000, 40_000], mrw=True, gamma=2.0, max_events=10 ** 6, block_size=128, max_in_flight=cap)
    c = B.config()
    if warps is None:  # whole blocks of 128 lanes
        assert c["block_size"] == 128 and c["grid"] == -(-min(cap, 100_000) // 128)
    else:
        assert c["block_size"] == 32 and c["grid"] == warps
    st = B.run(seed=3)
    for g, s, n in zip(gs, st, (60_000, 40_000)):
        assert s["packets"] == n and s["escaped"] + s["capped"] == n and s["error_flags"] == 0
        assert int(g.tallies()[0].sum()) == s["deposit_sum"]
    B.close()  # (before its disks)
    for g in gs:
        g.close()


def _agree(a, b, what):
    """Two sets of 8 runs agree in the mean: z from their own scatter, Student's t with 14 degrees of freedom per value (variance
    1.17; one of a few hundred values passes 6 once in a hundred tests). Paired random numbers make it smaller."""
    a, b = np.array(a), np.array(b)
    v = (a.var(0, ddof=1) + b.var(0, ddof=1)) / 8
    ok = (v > 0) & (a.mean(0) > 0) & (b.mean(0) > 0)
    z = (a.mean(0) - b.mean(0))[ok] / np.sqrt(v[ok])
    assert z.size >= 8, what
    assert np.sqrt(np.mean(z ** 2)) < 1.5 and np.abs(z).max() < 6, (what, z)


@pytest.mark.parametrize("tau,mrw,g,sources", [(100.0, False, 0.0, False), (100.0, False, 0.5, True), (3e3, True, 0.0, False)])
def test_gray_models_of_a_mixed_batch(M, tau, mrw, g, sources):
    """A gray model that shares a batch with non-gray dust (its packets then have a warp each) has the temperatures and the spectrum of
    a run of its own in lanes with as many packets in flight."""
    d = _disk(24, 20, tau, nlam=8, gray=True)
    d.opacity.g[:] = g
    n = 200_000
    a, other, b = M.Disk.from_model(d), M.Disk.from_model(_disk(16, 16, 100.0)), M.Disk.from_model(d)
    if sources:
        L = disks.viscous_sources(d)
        L *= d.star.L / L.sum()
        a.set_sources(L)
        b.set_sources(L)
    kw = dict(mrw=mrw, gamma=2.0, max_events=10 ** 6)
    B = M.Batch([a, other], [n, n // 4], **kw)
    assert B.config()["block_size"] == 32
    runs = []
    for k in range(8):
        for x in (a, other, b):
            x.reset()
        s = B.run(seed=9 + k)[0]
        assert s["escaped"] == n and s["error_flags"] == 0
        st = b.run_photons(n, seed=9 + k, tail_warps=-1, max_in_flight=96, **kw)
        assert abs(s["events"] / st["events"] - 1) < 0.02
        runs.append([(x.temperatures()[0], x.tallies()[2], x.sed().sum(axis=1)) for x in (a, b)])
    B.close()
    nabs = np.mean([r[1][1] for r in runs], axis=0).reshape(d.nr, d.ntheta)
    hot = nabs >= 200
    _agree([r[0][0][hot] for r in runs], [r[1][0][hot] for r in runs], "temperatures")
    _agree([r[0][2] for r in runs], [r[1][2] for r in runs], "spectrum")
    for x in (a, other, b):
        x.close()


@pytest.mark.parametrize("keep_j", [False, True])
def test_tail_of_a_run_in_lanes(M, keep_j):
    """A run that may have more packets in flight than go in warps: its tail (one packet per warp) against the form whose
    packets all stay in lanes, 20,000 in flight in both."""
    d = _disk(30, 20, 300.0)
    n = 400_000
    g = M.Disk.from_model(d)
    if keep_j:
        g.keep_mean_intensity()
    out = []
    for tail in (0, -1):
        runs = []
        for k in range(8):
            g.reset()
            st = g.run_photons(n, seed=40 + k, mrw=True, gamma=2.0, max_events=10 ** 6, tail_warps=tail, max_in_flight=20_000)
            assert st["escaped"] == n and st["error_flags"] == 0
            assert int(g.tallies()[0].sum()) == st["deposit_sum"]
            nabs = g.tallies()[2].reshape(d.nr, d.ntheta)
            runs.append((g.sed().sum(axis=1), np.where(nabs >= 200, g.temperatures()[0], 0.0),
                         g.mean_intensity().sum(axis=(0, 1)) if keep_j else 0))
        out.append(runs)
    g.close()
    for i, what in enumerate(("spectrum", "temperatures", "mean intensity")[:3 if keep_j else 2]):
        a, b = (np.array([r[i] for r in runs]) for runs in out)
        on = (np.concatenate([a, b]) > 0).all(axis=0)
        _agree(a[:, on], b[:, on], what)


@pytest.mark.parametrize("nr,nt,nlam,n,cap,sources,keep_j", [
    (1, 1, 1, 1, 0, False, False), (1, 1, 2, 5000, 0, False, False), (1, 9, 33, 5000, 1, False, True),
    (9, 1, 31, 5000, 7, True, False), (40, 3, 100, 3000, 0, True, True), (2, 2, 12, 30_000, 100_000, False, False)])
def test_edges(M, nr, nt, nlam, n, cap, sources, keep_j):
    """Few cells, bins and packets, one packet at a time, sources: every packet escapes, and the tallies, the absorbed and the escaped
    energy close. (One bin, or nt = 1 of a uniform disk: gray or not, whatever the opacity says.)"""
    d = _disk(nr, nt, 20.0, nlam=nlam)
    g = M.Disk.from_model(d)
    Ls = 0.0
    if sources:
        L = np.where(d.rho > 0, 1.0, 0.0)
        L *= 0.5 * d.star.L / L.sum()
        Ls = L.sum()
        g.set_sources(L)
    if keep_j:
        g.keep_mean_intensity()
    st = g.run_photons(n, seed=2, mrw=True, gamma=2.0, nmin=3, max_events=10 ** 6, max_in_flight=cap)
    assert st["packets"] == n and st["escaped"] == n and st["error_flags"] == 0
    tally, visits, nabs = g.tallies()
    assert int(tally.sum()) == st["deposit_sum"] and int(nabs.sum()) == st["absorptions"]
    assert abs(g.sed().sum() / (d.star.L + Ls) - 1) < 1e-12
    T = g.temperatures()[0]
    assert np.all(np.isfinite(T)) and np.array_equal(T.ravel() > 0, (tally.ravel() > 0) & (d.rho.ravel() > 0))
    if keep_j:
        assert np.isfinite(g.mean_intensity()).all()
    g.close()
