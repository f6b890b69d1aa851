"""Workloads of the library through its public entry points, for timing and for comparing results.

A case is a dict of plain values; its "kind" names one way the library is used:

  plain    gray plain Monte Carlo step: reset, transport, temperatures, escape spectrum; "repeat": the
           bitwise repeatable form of the run (no tail kernel)
  thick    the same with the modified random walk on a very thick gray disk (optionally with the PDA)
  nongray  the same with wavelength-dependent, anisotropically scattering dust
  scatter  a step that keeps the mean-intensity tally, then the ray-traced SED with scattered light
  polar    polarized transport with a Rayleigh Mueller matrix: broad-band Stokes parameters by inclination
  batch    several non-gray disks in one prepared batch
  pda      temperatures and diffusion solve of a Monte Carlo state read from a checkpoint
  grad     differentiable PDA: temperatures and the gradients of a weighted sum of them
  static   the allocation-free PDA solve on the caller's device buffers
  rays     ray-traced SED and N-band visibilities of a disk with known temperatures
  hydro    one vertical-structure update from known temperatures

What a transport step returns: the escape spectrum, and, of a repeatable run, the temperatures and the
integer tallies. By default the nearly empty cells hold the deposits of single packets whose paths depend
on when the tail kernel takes them over (and, with non-gray dust, on the order in which the GPU
interleaves packets), so the temperature array of such a run says little about another run of the same code.
"""
import math
import struct

import numpy as np
import torch

from paper_0902_3092_gb300 import disks, mcrt
from paper_0902_3092_gb300.pda_torch import pda_temperature

EUNIT = 65536
PC_CM = 3.0856775814913673e18
KB, HP, CL = 1.380649e-16, 6.62607015e-27, 2.99792458e10
SIGMA = disks.SIGMA_SB


def listed():
    return [
        # a small optically thin-to-moderate disk, the ordinary first run of a user (40 x 40 gray, tau 100)
        dict(name="plain_40x40_1e6", kind="plain", nr=40, nt=40, tau=100.0, n=1_000_000, repeat=False),
        # a quick look at the thick disk: few packets, the call waits for its longest ones
        dict(name="thick_200x120_1e6", kind="thick", nr=200, nt=120, tau=1e6, n=1_000_000, gamma=2.0, pda=False),
        # the production run of the thick disk with MRW and PDA (the benchmark step)
        dict(name="thick_200x120_1e8", kind="thick", nr=200, nt=120, tau=1e6, n=100_000_000, gamma=2.0, pda=True),
        # wavelength-dependent dust with g = 0.6 at tau 1e5: the ordinary disk model
        dict(name="nongray_100x60_1e6", kind="nongray", nr=100, nt=60, nlam=100, tau=1e5, n=1_000_000),
        # scattered-light SED: path-length tally kept in the run, then ray tracing with it
        dict(name="scatter_60x40_1e6", kind="scatter", nr=60, nt=40, tau=1e4, n=1_000_000, nphi=32),
        # broad-band polarization against inclination of a disk of small particles
        dict(name="polar_60x40_1e6", kind="polar", nr=60, nt=40, tau=1e3, n=1_000_000),
        # a parameter sweep of uneven non-gray disks replayed from one graph
        dict(name="batch_6", kind="batch", models=6, lo=30, hi=80, tau=1e3, n=1_200_000),
        # post-processing of a saved run: non-gray temperatures and the diffusion solve on the 400 x 200 disk
        dict(name="pda_400x200", kind="pda", nr=400, nt=200, gray=False, tau=1e6, half=0.15),
        # inverse problem step on the 400 x 200 disk: solve and adjoint through autograd
        dict(name="grad_400x200", kind="grad", nr=400, nt=200, gray=False, tau=1e6, half=0.05),
        # embedded use: small assembled system, no allocation
        dict(name="static_40x40", kind="static", nr=40, nt=40),
        # SED and visibilities of the thick disk at 45 degrees (104,448 rays, 100 bins)
        dict(name="rays_200x120", kind="rays", nr=200, nt=120, gray=True, nlam=100, tau=1e6, nsub=4, nphi=128,
             incl=45.0, image=False),
        # vertical-structure update of the thick disk
        dict(name="hydro_200x120", kind="hydro", nr=200, nt=120, tau=1e6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _ilog(rng, lo, hi):
    return int(round(_log(rng, lo, hi)))


def draw(rng):
    kind = rng.choice(["plain", "thick", "nongray", "scatter", "polar", "batch", "pda", "grad", "static", "rays",
                       "hydro"])
    c = dict(kind=kind)
    if kind == "plain":
        c.update(nr=_ilog(rng, 12, 150), nt=2 * _ilog(rng, 6, 60), tau=_log(rng, 10, 1e3), n=_ilog(rng, 1e5, 2e7),
                 repeat=rng.random() < 0.5)
    elif kind == "thick":
        c.update(nr=_ilog(rng, 60, 300), nt=2 * _ilog(rng, 20, 90), tau=_log(rng, 1e4, 1e6), n=_ilog(rng, 5e5, 5e7),
                 gamma=rng.choice([2.0, 4.0, 10.0]), pda=False)
    elif kind == "nongray":
        c.update(nr=_ilog(rng, 30, 150), nt=2 * _ilog(rng, 12, 40), nlam=rng.randint(24, 150), tau=_log(rng, 1e2, 1e5),
                 n=_ilog(rng, 2e5, 1.2e6))
    elif kind == "scatter":
        c.update(nr=_ilog(rng, 20, 100), nt=2 * _ilog(rng, 10, 30), tau=_log(rng, 30, 1e4), n=_ilog(rng, 2e5, 2e6),
                 nphi=rng.randint(16, 64))
    elif kind == "polar":
        c.update(nr=_ilog(rng, 20, 100), nt=2 * _ilog(rng, 10, 30), tau=_log(rng, 30, 1e3), n=_ilog(rng, 2e5, 2e6))
    elif kind == "batch":
        c.update(models=rng.randint(2, 8), lo=20, hi=rng.randint(40, 120), tau=_log(rng, 1e2, 1e3),
                 n=_ilog(rng, 6e5, 2e6))
    elif kind == "pda":
        c.update(nr=_ilog(rng, 24, 1500), nt=2 * _ilog(rng, 12, 500), gray=rng.random() < 0.5, tau=1e6,
                 half=rng.uniform(0.06, 0.15))
        if not c["gray"]:  # the non-gray tables are used on ordinary grids
            c.update(nr=min(c["nr"], 400), nt=min(c["nt"], 200))
    elif kind == "grad":
        c.update(nr=_ilog(rng, 40, 400), nt=2 * _ilog(rng, 16, 100), gray=rng.random() < 0.5, tau=1e6,
                 half=rng.uniform(0.06, 0.12))
    elif kind == "static":
        c.update(nr=_ilog(rng, 12, 400), nt=_ilog(rng, 11, 300))
    elif kind == "rays":
        c.update(nr=_ilog(rng, 20, 400), nt=2 * _ilog(rng, 8, 100), gray=rng.random() < 0.5, nlam=rng.randint(12, 200),
                 tau=_log(rng, 30, 1e6), nsub=rng.randint(1, 4), nphi=_ilog(rng, 12, 128), incl=rng.uniform(0.0, 88.0),
                 image=rng.random() < 0.3)
    else:
        c.update(nr=_ilog(rng, 24, 800), nt=2 * _ilog(rng, 12, 150), tau=_log(rng, 1e3, 1e6))
    return c


# ------------------------------------------------------------------------------------------ models
def _model(c):
    """The disk of a case."""
    kind = c["kind"]
    if kind == "plain":
        return disks.config_plain_gray(c["nr"], c["nt"], c["tau"])
    if kind == "polar":  # one broad band: the emission bins of gray dust would only spread Q and U thin
        return disks.make_disk(disks.log_r_faces(0.1, 100.0, c["nr"]), disks.midplane_refined_theta_faces(c["nt"]),
                               disks.paper_star(), disks.gray_opacity(1), c["tau"])
    if kind in ("thick", "scatter", "hydro"):
        return disks.config_thick_gray(c["nr"], c["nt"], c["tau"])
    if kind == "nongray":
        return disks.make_disk(disks.log_r_faces(0.1, 100.0, c["nr"]), disks.midplane_refined_theta_faces(c["nt"]),
                               disks.paper_star(), disks.powerlaw_opacity(c["nlam"]), c["tau"])
    nlam = c.get("nlam", 100)
    op = disks.gray_opacity(nlam) if c["gray"] else disks.powerlaw_opacity(nlam)
    rf = disks.rim_refined_r_faces(0.1, 100.0, c["nr"]) if kind == "rays" and c["gray"] and c["nr"] >= 40 \
        else disks.log_r_faces(0.1, 100.0, c["nr"])
    return disks.make_disk(rf, disks.midplane_refined_theta_faces(c["nt"]), disks.paper_star(), op, c["tau"])


def _volumes(d):
    rf, tf = d.r_faces_cm, d.theta_faces
    return (2 * math.pi / 3) * (rf[1:] ** 3 - rf[:-1] ** 3)[:, None] * (np.cos(tf[:-1]) - np.cos(tf[1:]))[None, :]


def _temperature_field(d, seed):
    """A smooth field (K), falling with radius and warmer away from the midplane, with waves of the seed."""
    rng = np.random.default_rng(seed)
    rc, tc = disks.cell_centres(d.r_faces_cm, d.theta_faces)
    T = 400.0 * (rc[:, None] / disks.AU_CM) ** -0.5 * (1 + 0.3 * np.cos(tc)[None, :] ** 2)
    x = np.log(rc / rc[0]) / math.log(rc[-1] / rc[0])
    for k in range(1, 4):
        T = T * (1 + 0.03 * np.sin(2 * math.pi * (k * x[:, None] + rng.random())) * np.cos(k * tc[None, :] + rng.random()))
    return T


def _state(d, seed, half):
    """Tallies and entry counts of a finished run: counting noise on the tallies of a smooth temperature
    field, and a band around the midplane that no packet entered."""
    rng = np.random.default_rng(seed + 1)
    rc, tc = disks.cell_centres(d.r_faces_cm, d.theta_faces)
    op, n_total = d.opacity, 10 ** 6
    band = (d.rho > 0) & (np.abs(tc - math.pi / 2)[None, :] < half) & (np.arange(d.nr)[:, None] >= 3)
    ext = np.minimum(np.diff(d.r_faces_cm)[:, None], rc[:, None] * np.diff(d.theta_faces)[None, :])
    thick = d.rho * float(np.max(op.kappa_abs + (1 - op.g) * op.kappa_sca)) * ext >= 1.0
    q = 4 * op.kappa_abs[0] * SIGMA * _temperature_field(d, seed) ** 4
    t = np.floor(q * d.rho * _volumes(d) * n_total * EUNIT / d.star.L) + 1 + 1000 * EUNIT
    t = np.where(thick & ~band, t * (1 + 0.01 * rng.standard_normal(t.shape)), 0)
    tally = np.floor(t).astype(np.uint64)
    visits = np.where(band, 0, 10_000).astype(np.uint64)
    return tally, visits, n_total


def _light_state(d, seed):
    """Tallies that give every dusty cell heavy enough to hold one count a smooth temperature."""
    q = 4 * d.opacity.kappa_abs[0] * SIGMA * _temperature_field(d, seed) ** 4
    n_total = 10 ** 9
    tally = np.where(d.rho > 0, np.floor(q * d.rho * _volumes(d) * n_total * EUNIT / d.star.L), 0).astype(np.uint64)
    return tally, np.full(tally.shape, 10_000, np.uint64), n_total


def _blob(d, tally, visits, n_total):
    """Checkpoint image of a Monte Carlo state (the format Disk.checkpoint writes)."""
    hdr = struct.pack("<7Qd", 0x4D43525443484B31, 1, d.nr, d.ntheta, d.opacity.nlam, n_total, 0, 0.0)
    hdr = hdr[:48] + struct.pack("<d", float(n_total)) + hdr[56:]
    return hdr + tally.tobytes() + visits.tobytes() + bytes(8 * (d.nr * d.ntheta + 10 * d.opacity.nlam))


def _batch_models(c, seed):
    rng = np.random.default_rng(c["models"] * 1000 + c["hi"])  # the sweep; the seed draws the packets
    ds, w = [], []
    for m in range(c["models"]):
        nr, nt = int(rng.integers(c["lo"], c["hi"] + 1)), 2 * int(rng.integers(c["lo"] // 2, c["hi"] // 2 + 1))
        beta = float(rng.uniform(1 / 7, 3 / 7))
        tau = float(c["tau"] ** rng.uniform(0.6, 1.0))
        ds.append(disks.make_disk(disks.log_r_faces(0.1, 100.0, nr), disks.midplane_refined_theta_faces(nt),
                                  disks.paper_star(), disks.powerlaw_opacity(), tau, p=1.0 + beta))
        w.append(rng.uniform(0.5, 2.0))
    return ds, [int(c["n"] * x / sum(w)) for x in w]


def _static_system(c, seed):
    """Mask, face conductances and boundary values of a diffusion region on the whole grid but its rim, with
    a smooth diffusion coefficient over four decades (numpy, FP64)."""
    nr, nt = c["nr"], c["nt"]
    rng = np.random.default_rng(seed)
    x, y = np.linspace(0, 1, nr)[:, None], np.linspace(0, 1, nt)[None, :]
    a, b = rng.random(2)
    D = 10.0 ** (2 * np.sin(2 * math.pi * (x + a)) * np.cos(math.pi * (y + b)) + 0.1 * rng.standard_normal((nr, nt)))
    Cr, Ct = np.zeros((nr, nt)), np.zeros((nr, nt))
    Cr[:-1] = 1.0 / (0.5 / D[:-1] + 0.5 / D[1:])
    Ct[:, :-1] = 1.0 / (0.5 / D[:, :-1] + 0.5 / D[:, 1:])
    mask = np.full((nr, nt), 2, np.int8)
    mask[0] = mask[-1] = 1
    mask[:, 0] = mask[:, -1] = 1
    u = np.where(mask == 1, (100.0 + 50.0 * np.cos(6 * x + a) * np.sin(5 * y + b)) ** 4, 0.0)
    return mask, Cr, Ct, u


def _vis_bins(d):
    """Bins of the N band (8-13 um)."""
    lc = np.sqrt(d.opacity.lam_edges_um[:-1] * d.opacity.lam_edges_um[1:])
    b = np.nonzero((lc > 8.0) & (lc < 13.0))[0]
    return b if b.size else np.array([d.opacity.nlam // 2])


def _rays(d, c):
    return disks.polar_rays(d.r_faces_cm, n_sub=c.get("nsub", 1), n_phi=c["nphi"], n_inner=4 * c.get("nsub", 1))


class _Bag:
    pass


def prepare(case, seed):
    c, s = case, _Bag()
    s.case, s.seed, kind = c, int(seed) + 1, c["kind"]
    if kind == "static":
        mask, Cr, Ct, u = _static_system(c, seed)
        dev = torch.device("cuda")
        s.mask, s.Cr, s.Ct, s.u0 = (torch.from_numpy(a.ravel()).to(dev) for a in (mask, Cr, Ct, u))
        return s
    if kind == "batch":
        ds, npk = _batch_models(c, seed)
        s.disks = [mcrt.Disk.from_model(d) for d in ds]
        s.batch = mcrt.Batch(s.disks, npk, mrw=True, gamma=2.0, max_events=10 ** 6, block_size=128)
        return s
    d = _model(c)
    s.disk = mcrt.Disk.from_model(d)
    if kind == "scatter":
        s.disk.keep_mean_intensity()
        s.disk.set_rays(math.pi / 4, 140 * PC_CM, _rays(d, c))
    elif kind == "polar":
        s.disk.set_mueller(disks.rayleigh_mueller(d.opacity.nlam, 181))
    elif kind in ("pda", "grad"):
        s.blob = _blob(d, *_state(d, seed, c["half"]))
        if kind == "grad":
            s.disk.restore(s.blob)
            dev, rng = torch.device("cuda"), np.random.default_rng(seed + 7)
            s.log_rho = torch.from_numpy(np.log(np.where(d.rho > 0, d.rho, 1.0))).to(dev).requires_grad_()
            op = d.opacity
            s.kappa = torch.from_numpy(np.full(d.rho.shape, float(op.kappa_abs[0])) *
                                       (1 + 0.2 * rng.random(d.rho.shape))).to(dev).requires_grad_()
            s.w = torch.from_numpy(rng.random(d.rho.shape)).to(dev)
    elif kind == "rays":
        s.disk.restore(_blob(d, *_light_state(d, seed)))
        s.disk.temperatures()
        s.disk.set_rays(math.radians(c["incl"]), 140 * PC_CM, _rays(d, c))
        s.bins = _vis_bins(d)
    elif kind == "hydro":
        s.disk.restore(_blob(d, *_light_state(d, seed)))
        s.disk.temperatures()
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "plain":
        s.disk.reset()
        s.disk.run_photons(c["n"], seed=s.seed, tail_warps=-1 if c["repeat"] else 0)
        T, sed = s.disk.temperatures()[0], s.disk.sed()
        return {"T": T, "tallies": list(s.disk.tallies()), "sed": sed} if c["repeat"] else {"sed": sed}
    if kind == "thick":
        s.disk.reset()
        s.disk.run_photons(c["n"], seed=s.seed, mrw=True, gamma=c["gamma"], max_events=10 ** 6)
        if c["pda"]:
            s.disk.solve_pda()
            s.disk.temperatures(mcrt.T_PDA)
        return {"sed": s.disk.sed()}
    if kind == "nongray":
        s.disk.reset()
        s.disk.run_photons(c["n"], seed=s.seed, mrw=True, gamma=2.0, max_events=10 ** 6)
        s.disk.temperatures()
        return {"sed": s.disk.sed()}
    if kind == "scatter":
        s.disk.reset()
        s.disk.run_photons(c["n"], seed=s.seed, mrw=True, gamma=2.0, max_events=10 ** 6)
        o = s.disk.raytrace(scattering=True)
        s.disk.temperatures()
        return {"F": o["F"].astype(np.float32), "sed": s.disk.sed()}
    if kind == "polar":
        s.disk.reset()
        s.disk.run_photons(c["n"], seed=s.seed, mrw=True, gamma=2.0, max_events=10 ** 6)
        I, Q, U = s.disk.sed_stokes()
        return {"I": I, "Q": Q, "U": U}
    if kind == "batch":
        for g in s.disks:
            g.reset()
        s.batch.run(seed=s.seed)
        return {"sed": [g.sed() for g in s.disks]}
    if kind == "pda":
        s.disk.restore(s.blob)
        T = s.disk.temperatures()[0]
        s.disk.solve_pda()
        return {"T_mc": T, "T": s.disk.temperatures(mcrt.T_PDA)[0]}
    if kind == "grad":
        s.log_rho.grad = s.kappa.grad = None
        T = pda_temperature(s.disk, s.log_rho, s.kappa)
        (s.w * T).sum().backward()
        return {"T": T.detach(), "g_log_rho": s.log_rho.grad, "g_kappa": s.kappa.grad}
    if kind == "static":
        u = s.u0.clone()
        mcrt.pda_solve_static(c["nr"], c["nt"], s.mask.data_ptr(), s.Cr.data_ptr(), s.Ct.data_ptr(), u.data_ptr())
        return {"u": u}
    if kind == "rays":
        # the trace is FP32; its results come widened to doubles
        o = s.disk.raytrace(want_image=c["image"])
        v = s.disk.visibilities(s.bins, 1e4, 0.4)
        out = {"F": o["F"].astype(np.float32), "F_star": o["F_star"], "vis": v.astype(np.float32)}
        if c["image"]:
            out["I"] = o["I"].astype(np.float32)
        return out
    return {"rho": s.disk.hydrostatic_density(which=mcrt.T_MC)}


# ------------------------------------------------------------------------------------------ work
def work(case):
    c = case
    kind = c["kind"]
    if kind in ("plain", "thick", "nongray", "scatter", "polar", "batch"):
        # every packet crosses about one face per cell row on its way (nr of them), and in a thick disk
        # makes of order 100 interactions; a crossing needs four face distances (about 100 operations),
        # an interaction a random block and a direction (about 60)
        cells = c["models"] * c["hi"] ** 2 if kind == "batch" else c["nr"] * c["nt"]
        rows = c["hi"] if kind == "batch" else c["nr"]
        inter = 1 if kind == "plain" or c["tau"] <= 1e3 else 10 * math.log10(c["tau"] / 1e3)
        return {"bytes": 40.0 * cells, "flops": c["n"] * (100.0 * rows + 60.0 * inter)}
    n = c["nr"] * c["nt"]
    if kind == "hydro":
        return {"bytes": 24.0 * n, "flops": 60.0 * n}
    if kind == "rays":
        rays = c["nphi"] * c["nsub"] * (c["nr"] + 4)
        # a ray crosses about nr / 2 shells twice over; an exponential and a few operations per bin
        seg = rays * 0.8 * c["nr"]
        return {"bytes": 4.0 * c["nlam"] * (n + rays) + 24.0 * rays, "flops": seg * 10.0 * c["nlam"]}
    # the diffusion region (about a tenth to the whole grid): iterations of the order of its longer side,
    # about 20 operations each; bytes: the state read and the solution written
    frac = 1.0 if kind == "static" else 0.25
    iters = 3.0 * max(c["nr"], c["nt"])
    return {"bytes": 40.0 * n, "flops": 20.0 * frac * n * iters * (2 if kind == "grad" else 1)}


# ------------------------------------------------------------------------------------------ exact values
def _tails(x):
    """G3 = int_x^inf t^3/(e^t - 1), G4 = int_x^inf t^4 e^t/(e^t - 1)^2 (torch, FP64)."""
    x = x.clamp(max=700.0)
    g3, g4 = torch.zeros_like(x), torch.zeros_like(x)
    xl = x.clamp(min=0.9)
    e1 = torch.exp(-xl)
    e = e1.clone()
    for n in range(1, 48):
        g3 += e * (xl ** 3 / n + 3 * xl ** 2 / n ** 2 + 6 * xl / n ** 3 + 6.0 / n ** 4)
        g4 += e * (xl ** 4 + 4 * xl ** 3 / n + 12 * xl ** 2 / n ** 2 + 24 * xl / n ** 3 + 24.0 / n ** 4)
        e = e * e1
    # below 0.9: t/(e^t - 1) = sum B_k t^k / k!; G4 = 4 G3 + x^4/(e^x - 1)
    bern = [1.0, -0.5, 1 / 6, 0.0, -1 / 30, 0.0, 1 / 42, 0.0, -1 / 30, 0.0, 5 / 66, 0.0, -691 / 2730, 0.0, 7 / 6, 0.0,
            -3617 / 510, 0.0, 43867 / 798, 0.0, -174611 / 330]
    f3 = torch.zeros_like(x)
    for k in range(len(bern) - 1, -1, -1):
        f3 = f3 * x + bern[k] / math.factorial(k) / (k + 3)
    f3 = math.pi ** 4 / 15 - f3 * x ** 3
    f4 = 4 * f3 + torch.where(x > 0, x ** 4 / torch.expm1(x.clamp(min=1e-300)), torch.zeros_like(x))
    small = x < 0.9
    return torch.where(small, f3, g3), torch.where(small, f4, g4)


def _bins(op, T):
    """Bbar_b(T) and T dBbar_b/dT per bin, (cells, nlam); the first and last bin reach to 0 and infinity."""
    e = torch.tensor(op.lam_edges_um[1:-1], dtype=torch.float64, device=T.device) * 1e-4
    g3, g4 = _tails(HP * CL / (e[None, :] * KB * T[:, None]))
    z = torch.zeros(T.numel(), 1, dtype=torch.float64, device=T.device)
    g3 = torch.cat([z, g3, z + math.pi ** 4 / 15], 1)
    g4 = torch.cat([z, g4, z + 4 * math.pi ** 4 / 15], 1)
    pre = (2 * KB ** 4 / (HP ** 3 * CL ** 2)) * T[:, None] ** 4
    return pre * torch.diff(g3, dim=1), pre * torch.diff(g4, dim=1)


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _exact_T(d, tally, n_total):
    """Radiative-equilibrium temperatures of the tallies."""
    op = d.opacity
    m = d.rho * _volumes(d)
    with np.errstate(divide="ignore", invalid="ignore"):
        q = np.where((tally > 0) & (m > 0), tally.astype(np.float64) / EUNIT * d.star.L / n_total / m, 0.0)
    T = (q / (4 * SIGMA * op.kappa_abs[0])) ** 0.25
    if op.is_gray():
        return T
    at = np.nonzero(q.ravel())[0]
    qq = torch.from_numpy(q.ravel()[at]).to(_dev())
    ka = torch.from_numpy(op.kappa_abs).to(_dev())
    out = np.zeros(q.size)
    for lo in range(0, len(at), 16384):
        qt = qq[lo:lo + 16384]
        x = torch.log((qt / (4 * SIGMA * float(op.kappa_abs.mean()))) ** 0.25)
        for _ in range(60):
            B, dB = _bins(op, torch.exp(x))
            Q, dQ = 4 * math.pi * (ka * B).sum(1), 4 * math.pi * (ka * dB).sum(1)
            step = (torch.log(Q / qt) * Q / dQ).clamp(-1.0, 1.0)
            x = x - step
            if float(step.abs().max()) < 1e-15:
                break
        out[at[lo:lo + 16384]] = torch.exp(x).cpu().numpy()
    return out.reshape(q.shape)


def _block_solve(mask, Cr, Ct, rhs_list):
    """Direct solves of the finite-volume system on the cells with mask 2 (the others fixed at zero in the
    unknown): block Cholesky over the shells, couplings between shells diagonal; refined twice."""
    nr, nt = mask.shape
    cols = np.nonzero((mask == 2).any(0))[0]
    j0, j1 = cols[0], cols[-1] + 1
    w = j1 - j0
    if nr * float(w) ** 3 > 2e11:
        return None
    dev = _dev()
    diag = np.zeros(mask.shape)
    on = mask > 0
    diag[:-1] += np.where(on[1:], Cr[:-1], 0)
    diag[1:] += np.where(on[:-1], Cr[:-1], 0)
    diag[:, :-1] += np.where(on[:, 1:], Ct[:, :-1], 0)
    diag[:, 1:] += np.where(on[:, :-1], Ct[:, :-1], 0)
    un = mask == 2
    s = np.where(un, 1 / np.sqrt(np.where(un, diag, 1.0)), 0.0)
    ar = np.zeros(mask.shape)
    at = np.zeros(mask.shape)
    ar[:-1] = -Cr[:-1] * s[:-1] * s[1:]
    at[:, :-1] = -Ct[:, :-1] * s[:, :-1] * s[:, 1:]
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    AR, AT, S = t(ar[:, j0:j1]), t(at[:, j0:j1]), t(s[:, j0:j1])
    L = []
    eye = torch.eye(w, dtype=torch.float64, device=dev)
    prev = None
    for i in range(nr):
        A = eye + torch.diag(AT[i, :-1], 1) + torch.diag(AT[i, :-1], -1)
        if prev is not None:
            Y = torch.linalg.solve_triangular(prev, torch.diag(AR[i - 1]), upper=False)
            A = A - Y.T @ Y
        prev = torch.linalg.cholesky(A)
        L.append(prev)

    def solve(r):
        z, out = [], [None] * nr
        for i in range(nr):
            v = r[i] if i == 0 else r[i] - AR[i - 1] * torch.cholesky_solve(z[i - 1][:, None], L[i - 1])[:, 0]
            z.append(v)
        for i in range(nr - 1, -1, -1):
            v = z[i] if i == nr - 1 else z[i] - AR[i] * out[i + 1]
            out[i] = torch.cholesky_solve(v[:, None], L[i])[:, 0]
        return torch.stack(out)

    def apply(x):
        y = x.clone()
        y[1:] += AR[:-1] * x[:-1]
        y[:-1] += AR[:-1] * x[1:]
        y[:, 1:] += AT[:, :-1] * x[:, :-1]
        y[:, :-1] += AT[:, :-1] * x[:, 1:]
        return y

    res = []
    for rhs in rhs_list:
        b = t(rhs[:, j0:j1]) * S
        x = solve(b)
        for _ in range(2):
            x = x + solve(b - apply(x))
        full = np.zeros(mask.shape)
        full[:, j0:j1] = (x * S).cpu().numpy()
        res.append(full)
    return res


def _boundary_rhs(mask, Cr, Ct, u):
    b = np.zeros(mask.shape)
    v = np.where(mask == 1, u, 0.0)
    b[:-1] += Cr[:-1] * v[1:]
    b[1:] += Cr[:-1] * v[:-1]
    b[:, :-1] += Ct[:, :-1] * v[:, 1:]
    b[:, 1:] += Ct[:, :-1] * v[:, :-1]
    return b


def _pda_system(d, tally, visits, T, kappa=None):
    """Mask (2: diffusion cell, 1: fixed temperature), half-cell resistances, D and face conductances."""
    op = d.opacity
    rf, tf = d.r_faces_cm, d.theta_faces
    rc, tc = disks.cell_centres(rf, tf)
    chip = op.kappa_abs + (1 - op.g) * op.kappa_sca
    ext = np.minimum(np.diff(rf)[:, None], rc[:, None] * np.diff(tf)[None, :])
    dust = d.rho > 0
    with np.errstate(divide="ignore"):
        err = 0.25 / np.sqrt(tally.astype(np.float64) / EUNIT)
    pda = dust & (d.rho * chip.max() * ext >= 1.0) & ((visits < 30) | (err > 0.05))
    mask = np.where(pda, 2, np.where(dust & (tally > 0), 1, 0))
    if kappa is None:
        kappa = np.full(d.rho.shape, chip[0])
        if not op.is_gray():
            un = np.pad(mask == 2, 1)
            near = (mask == 1) & (un[:-2, 1:-1] | un[2:, 1:-1] | un[1:-1, :-2] | un[1:-1, 2:])
            Tk = np.maximum(np.where(tally > 0, T, T[near].mean() if near.any() else 1.0), 1.0)
            at = np.nonzero((mask == 2) | near)
            _, dB = _bins(op, torch.from_numpy(Tk[at]).to(_dev()))
            ch = torch.from_numpy(chip).to(_dev())
            kappa[at] = (dB.sum(1) / (dB / ch).sum(1)).cpu().numpy()
    D = np.where(mask > 0, 1.0 / (3.0 * np.where(mask > 0, d.rho, 1.0) * kappa), 0.0)
    om = 2 * math.pi * (np.cos(tf[:-1]) - np.cos(tf[1:]))[None, :]
    h_in, h_out = (1 / rf[:-1] - 1 / rc)[:, None] / om, (1 / rc - 1 / rf[1:])[:, None] / om
    with np.errstate(divide="ignore"):
        lt = np.log(np.tan(0.5 * tf))
    lt[0], lt[-1] = -np.inf, np.inf
    lc = np.log(np.tan(0.5 * tc))
    dr = (2 * math.pi * np.diff(rf))[:, None]
    h_lo, h_hi = (lc - lt[:-1])[None, :] / dr, (lt[1:] - lc)[None, :] / dr
    Cr, Ct = np.zeros(d.rho.shape), np.zeros(d.rho.shape)
    with np.errstate(divide="ignore", invalid="ignore"):
        fr = (mask[:-1] > 0) & (mask[1:] > 0) & ((mask[:-1] == 2) | (mask[1:] == 2))
        Cr[:-1] = np.where(fr, 1 / (h_out[:-1] / D[:-1] + h_in[1:] / D[1:]), 0.0)
        ft = (mask[:, :-1] > 0) & (mask[:, 1:] > 0) & ((mask[:, :-1] == 2) | (mask[:, 1:] == 2))
        Ct[:, :-1] = np.where(ft, 1 / (h_hi[:, :-1] / D[:, :-1] + h_lo[:, 1:] / D[:, 1:]), 0.0)
    return mask, kappa, D, Cr, Ct, (h_in, h_out, h_lo, h_hi)


def _exact_pda(c, seed):
    d = _model(c)
    tally, visits, n_total = _state(d, seed, c["half"])
    T = _exact_T(d, tally, n_total)
    kappa = None
    if c["kind"] == "grad":
        rng = np.random.default_rng(seed + 7)
        kappa = np.full(d.rho.shape, float(d.opacity.kappa_abs[0])) * (1 + 0.2 * rng.random(d.rho.shape))
        w = rng.random(d.rho.shape)
    mask, kappa, D, Cr, Ct, h = _pda_system(d, tally, visits, T, kappa)
    u0 = np.where(mask == 1, T ** 4, 0.0)
    sol = _block_solve(mask, Cr, Ct, [_boundary_rhs(mask, Cr, Ct, u0)])
    if sol is None:
        return None
    un = mask == 2
    u = np.where(un, sol[0], u0)
    Tp = np.where(un, np.maximum(u, 0.0) ** 0.25, T)
    if c["kind"] == "pda":
        return {"T_mc": T, "T": Tp}
    g = np.where(un, w * 0.25 * np.where(un, u, 1.0) ** -0.75, 0.0)
    lam = _block_solve(mask, Cr, Ct, [g])[0]
    dD = np.zeros(d.rho.shape)
    with np.errstate(divide="ignore", invalid="ignore"):
        jr = np.zeros(d.rho.shape)
        jr[:-1] = np.where(Cr[:-1] > 0, -np.diff(lam, axis=0) * np.diff(u, axis=0) * Cr[:-1] ** 2, 0.0)
        jt = np.zeros(d.rho.shape)
        jt[:, :-1] = np.where(Ct[:, :-1] > 0, -np.diff(lam, axis=1) * np.diff(u, axis=1) * Ct[:, :-1] ** 2, 0.0)
        D2 = np.where(mask > 0, D, 1.0) ** 2
        dD += np.where(jr != 0, jr * h[1], 0.0) / D2
        dD[1:] += np.where(jr[:-1] != 0, jr[:-1] * h[0][1:], 0.0) / D2[1:]
        dD += np.where(jt != 0, jt * np.where(np.isfinite(h[3]), h[3], 0.0), 0.0) / D2
        dD[:, 1:] += np.where(jt[:, :-1] != 0, jt[:, :-1] * np.where(np.isfinite(h[2][:, 1:]), h[2][:, 1:], 0.0), 0.0) / \
            D2[:, 1:]
    return {"T": Tp, "g_log_rho": -D * dD, "g_kappa": -D / kappa * dD}


def _exact_static(c, seed):
    mask, Cr, Ct, u = _static_system(c, seed)
    sol = _block_solve(mask, Cr, Ct, [_boundary_rhs(mask, Cr, Ct, u)])
    return None if sol is None else {"u": np.where(mask == 2, sol[0], u).ravel()}


def _exact_hydro(c, seed):
    d = _model(c)
    tally, _, n_total = _light_state(d, seed)
    T = np.maximum(_exact_T(d, tally, n_total), 10.0)
    rc, tc = disks.cell_centres(d.r_faces_cm, d.theta_faces)
    z, R = rc[:, None] * np.cos(tc), rc[:, None] * np.sin(tc)
    a = 6.67430e-8 * 2.5 * 1.98892e33 * z / R ** 3 * (2.3 * 1.66053906660e-24 / (KB * T))
    phi = np.zeros_like(T)
    phi[:, 1:] = np.cumsum(-0.5 * (a[:, 1:] + a[:, :-1]) * np.diff(z, axis=1), axis=1)
    lg = phi - np.log(T)
    dust = d.rho > 0
    top = np.max(np.where(dust, lg, -np.inf), axis=1, keepdims=True)
    p = np.where(dust, np.exp(np.where(dust, lg - np.where(np.isfinite(top), top, 0.0), 0.0)), 0.0)
    V = _volumes(d)
    M, tot = (d.rho * V).sum(1, keepdims=True), (p * V).sum(1, keepdims=True)
    return {"rho": np.where(tot > 0, p * M / np.where(tot > 0, tot, 1.0), 0.0)}


def _exact_rays(c, seed):
    """Every ray cut at its crossings with all spheres and cones, the cell of each piece from its middle."""
    d = _model(c)
    op, nr, nt = d.opacity, d.nr, d.ntheta
    rays = _rays(d, c)
    if float(rays.n) * (2 * nr + 2 * nt) * op.nlam > 1.2e10:
        return None
    dev = _dev()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float64)).to(dev)  # noqa: E731
    tally, _, n_total = _light_state(d, seed)
    T = _exact_T(d, tally, n_total).ravel()
    S = np.zeros((nr * nt, op.nlam))
    at = np.nonzero(T)[0]
    for lo in range(0, len(at), 16384):
        k = at[lo:lo + 16384]
        S[k] = _bins(op, t(T[k]))[0].cpu().numpy()
    chi = op.kappa_abs + op.kappa_sca
    S = t(S * (op.kappa_abs / chi))
    rho, chi_t = t(d.rho.ravel()), t(chi)
    inc, dist = math.radians(c["incl"]), 140 * PC_CM
    si, ci = math.sin(inc), math.cos(inc)
    rf, cf = t(d.r_faces_cm), t(np.cos(d.theta_faces))
    c2, s2 = t(np.cos(d.theta_faces[1:-1]) ** 2), t(np.sin(d.theta_faces[1:-1]) ** 2)
    mid = int(np.argmin(np.abs(d.theta_faces[1:-1] - math.pi / 2)))  # the midplane face: the plane z = 0
    rays_p, rays_q = t(rays.p), t(rays.q)
    per = max(64, int(6e8 / 8 / ((2 * nr + 2 * nt + 4) * op.nlam)))
    img = []
    for lo in range(0, rays.n, per):
        p, q = rays_p[lo:lo + per, None], rays_q[lo:lo + per, None]
        b2 = p * p + q * q
        smax = torch.sqrt((rf[-1] ** 2 - b2).clamp(min=0.0))
        sr = torch.sqrt((rf[None, :] ** 2 - b2).clamp(min=0.0))
        sr = torch.where(rf[None, :] ** 2 > b2, sr, torch.zeros_like(sr))
        A = c2 * si * si - s2 * ci * ci
        B = -q * si * ci * torch.ones_like(c2)
        C = c2 * (q * q * ci * ci + p * p) - s2 * (q * si) ** 2
        disc = B * B - A * C
        h = -(B + torch.where(B >= 0, 1.0, -1.0) * torch.sqrt(disc.clamp(min=0.0)))
        x1, x2 = h / A, C / h
        x1[:, mid:mid + 1] = -q * si / ci if ci != 0 else torch.zeros_like(q)
        x2[:, mid] = 0.0
        st = torch.cat([x1, x2], 1)
        bad = ~torch.isfinite(st) | (torch.cat([disc, disc], 1) < 0)
        bad[:, mid] = False
        st = torch.where(bad, torch.zeros_like(st), st)
        s = torch.cat([sr, -sr, st], 1)
        s = torch.minimum(torch.maximum(s, -smax), smax)
        s = torch.sort(s, 1).values
        L, m = torch.diff(s, dim=1), 0.5 * (s[:, 1:] + s[:, :-1])
        r = torch.sqrt(b2 + m * m)
        ir = (torch.searchsorted(rf, r, right=True) - 1).clamp(-1, nr - 1)
        mu = (q * si + m * ci) / r
        it = (torch.searchsorted(-cf, -mu, right=True) - 1).clamp(0, nt - 1)
        cell = (ir.clamp(min=0) * nt + it)
        a = torch.where((ir >= 0) & (b2 < rf[-1] ** 2), rho[cell] * L, torch.zeros_like(L))
        after = a.flip(1).cumsum(1).flip(1) - a  # column from the piece's end to the observer
        I = torch.zeros(p.shape[0], op.nlam, dtype=torch.float64, device=dev)
        for b0 in range(0, op.nlam, 8):
            ch = chi_t[b0:b0 + 8]
            I[:, b0:b0 + 8] = (S[cell][:, :, b0:b0 + 8] * -torch.expm1(-a[:, :, None] * ch) *
                               torch.exp(-after[:, :, None] * ch)).sum(1)
        img.append(I)
    I = torch.cat(img)
    w = t(rays.w)
    it = 0
    while it + 1 < nt and d.theta_faces[it + 1] <= inc:
        it += 1
    col = float((d.rho[:, it] * np.diff(d.r_faces_cm)).sum())
    Bs = _bins(op, t(np.array([d.star.T_K])))[0].cpu().numpy()[0]
    Fs = math.pi * d.star.R_cm ** 2 * Bs / dist ** 2 * np.exp(-col * chi)
    F = (w[:, None] * I).sum(0).cpu().numpy() / dist ** 2 + Fs
    vis = []
    for b in _vis_bins(d):
        f = 1e4 / (math.sqrt(op.lam_edges_um[b] * op.lam_edges_um[b + 1]) * 1e-4 * dist)
        ph = 2 * math.pi * torch.remainder(f * math.cos(0.4) * rays_p + f * math.sin(0.4) * rays_q, 1.0)
        wi = w * I[:, b] / dist ** 2
        re, im = float((wi * torch.cos(ph)).sum()) + Fs[b], float((wi * torch.sin(ph)).sum())
        tot = float(wi.sum()) + Fs[b]
        vis.append(math.hypot(re, im) / tot if tot > 0 else 0.0)
    out = {"F": F, "F_star": Fs, "vis": np.array(vis)}
    if c["image"]:
        out["I"] = I.cpu().numpy()
    return out


def exact(case, seed):
    """The results in 64 bits, by other means. Monte Carlo estimates have none."""
    kind = case["kind"]
    if kind in ("pda", "grad"):
        return _exact_pda(case, seed)
    if kind == "static":
        return _exact_static(case, seed)
    if kind == "hydro":
        return _exact_hydro(case, seed)
    if kind == "rays":
        return _exact_rays(case, seed)
    return None
