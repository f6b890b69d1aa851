"""Benchmark of the transport + MRW + PDA path on the very optically thick gray disk.

Workload (per rank, one step): the 200 x 120 rim-refined gray disk (albedo 0.5, isotropic, midplane
radial optical depth 1e6, star 4000 K / 2 R_sun) -- reset tallies, transport `--packets` photon
packets with the modified random walk (gamma = 2), radiative-equilibrium temperatures, partial
diffusion approximation. Metric: photon packets per second of the whole step (MRW + PDA), with the
plain Monte Carlo rate on the same disk, the PDA time and the end-to-end rate through the host C ABI
reported beside it.

    python bench.py [--gpus N --steps K --warmup W] [--impl reference]

N > 1 runs one rank per GPU (torchrun): each rank transports its own packet range and the integer
tallies are summed across ranks (the exchange of the Monte Carlo step) before the PDA.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import re
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "photon packets/s (MRW+PDA vs plain MC) at tau_mid=1e6, equal T accuracy; PDA ms"
UNIT = "packets/s"
WORKLOAD = "thick gray disk 200x120 rim-refined, tau_mid=1e6, albedo 0.5 isotropic, MRW gamma=2 + PDA"

# Work per transport step (an interaction, an MRW jump or a face crossing) of one FP32 transport call on
# this workload, from the ncu counts of its two kernels (the persistent transport kernel, and the tail
# kernel that finishes the packets in flight when the queue drains) on a 1e7-packet call: warp and thread
# instructions (smsp__inst_executed.sum, smsp__thread_inst_executed.sum) and DRAM bytes per step. The
# kernels are bound by instruction issue (divergent, latency-bound integer/FP32 work; tallies and tables
# stay in L2), so the roofline is issue slots: 152 SMs x 4 schedulers x 1 warp instruction per clock. The
# counts live in the profile summary written from that capture, so a kernel change without a new capture
# leaves the roofline figures null.
COUNTS_FILE = os.path.join(ROOT, "profiles", "transport_counts_thickgray_200x120.md")
# The same for the ray-tracing kernel: counts per ray segment through dust of the 200x120 disk at 45 degrees, 100 bins.
RAY_COUNTS_FILE = os.path.join(ROOT, "profiles", "raytrace_thickgray_200x120_ncu.md")
N_SMS, SCHEDULERS = 152, 4


def transport_counts(path=None):
    """Counts of a profile summary (the transport's): the indented `key: value` lines."""
    out = {}
    try:
        with open(path or COUNTS_FILE) as f:
            for ln in f:
                m = re.match(r"^    ([a-z0-9_]+): (\S+)\s*$", ln)
                if m:
                    try:
                        out[m.group(1)] = float(m.group(2))
                    except ValueError:
                        out[m.group(1)] = m.group(2)
    except OSError:
        pass
    return out


def code_only(src):
    """C/C++ source without its comments, whitespace runs collapsed (string and character literals kept)."""
    out, i, n = [], 0, len(src)
    while i < n:
        if src.startswith("//", i):
            j = src.find("\n", i)
            i = n if j < 0 else j
        elif src.startswith("/*", i):
            j = src.find("*/", i + 2)
            i = n if j < 0 else j + 2
            out.append(" ")
        elif src[i] in "\"'":
            j = i + 1
            while j < n and src[j] != src[i]:
                j += 2 if src[j] == "\\" else 1
            out.append(src[i:j + 1])
            i = j + 1
        else:
            out.append(src[i])
            i += 1
    return " ".join("".join(out).split())


def transport_source_hash(root=None, files=("common.cuh", "transport.cuh", "transport_f32.cu")):
    """Hash of the transport kernels' code (comments and layout left out): counts taken from another
    version of the code are not used."""
    import hashlib
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(root or ROOT, "paper_0902_3092_gb300", "csrc", f), encoding="utf-8") as fh:
            h.update(code_only(fh.read()).encode())
    return h.hexdigest()[:16]


def ray_source_hash(root=None):
    """The same of the ray-tracing kernel's code."""
    return transport_source_hash(root, ("common.cuh", "raymarch.cuh", "raytrace.cu"))


def ray_roofline(segments, t_call, sm_mhz):
    """Issue-slot roofline of one mcrt_raytrace call: the ray-tracing kernel's warp instructions per segment (ncu) x the
    call's segments / its CUDA-event time, against 152 SMs x 4 schedulers x the SM clock."""
    c = transport_counts(RAY_COUNTS_FILE)
    peak = N_SMS * SCHEDULERS * sm_mhz * 1e6
    roof = {"bound": "alu", "unit": "warp-inst/s", "peak": peak, "achieved": None, "frac": None, "traffic": None,
            "thread_inst_frac": None, "kernel": "k_raytrace<float, 4> (time: with k_sed_part and k_sed_final)",
            "counts_file": os.path.relpath(RAY_COUNTS_FILE, ROOT)}
    if c.get("source_sha16") != ray_source_hash():
        roof["note"] = "no ncu counts for the current ray-tracing kernel (its sources changed since the capture)"
        return roof
    wps, tps = c["warp_inst_per_segment"], c["thread_inst_per_segment"]
    ach = wps * segments / t_call
    roof.update({"achieved": ach, "frac": ach / peak, "traffic": c["dram_bytes_per_launch"],
                 "thread_inst_frac": tps * segments / t_call / (32 * peak),
                 "note": f"issue slots: {wps:.1f} warp instructions per segment through dust (ncu) x {segments} segments / "
                         f"CUDA-event call time; peak = 152 SMs x 4 schedulers x {sm_mhz:g} MHz; thread_inst_frac counts "
                         "active lanes"})
    return roof


def transport_roofline(steps_per_launch, t_launch, clocks, peaks):
    """Issue-slot roofline of one transport call (its two kernels): warp instructions per step from the
    ncu counts x steps per launch / the launch's CUDA-event time, against 152 SMs x 4 schedulers x the
    maximum SM clock; beside it the active-lane figure (thread instructions against 32 lanes per slot)."""
    c = transport_counts()
    mhz = clocks.get("sm_max_mhz") or peaks.get("sm_max_mhz") or 2070.0
    peak = N_SMS * SCHEDULERS * mhz * 1e6
    roof = {"bound": "alu", "unit": "warp-inst/s", "peak": peak, "achieved": None, "frac": None, "traffic": None,
            "thread_inst_frac": None,
            "kernel": "transport_kernel<float> + transport_tail_kernel<float> (one 1e8-packet transport call)",
            "counts_file": os.path.relpath(COUNTS_FILE, ROOT)}
    fresh = c.get("source_sha16") == transport_source_hash()
    if not c or not fresh:
        roof["note"] = "no ncu counts for the current transport kernels (their sources changed since the capture)"
        return roof
    wps, tps = c["warp_inst_per_step"], c["thread_inst_per_step"]
    ach = wps * steps_per_launch / t_launch
    roof.update({"achieved": ach, "frac": ach / peak,
                 "thread_inst_frac": tps * steps_per_launch / t_launch / (32 * peak),
                 "traffic": c.get("dram_bytes_per_launch"),
                 "note": f"issue slots: {wps:.2f} warp instructions per transport step (ncu, both kernels, "
                         f"{c.get('profiled_packets', 0):.0e}-packet call) x {steps_per_launch:.4g} steps per launch / "
                         f"{t_launch:.4g} s CUDA-event launch time; peak = 152 SMs x 4 schedulers x {mhz:g} MHz; "
                         f"thread_inst_frac = {tps:.1f} thread instructions per step against 32 lanes per slot "
                         "(the share of lanes doing work); traffic = DRAM bytes of one 1e8-packet call (ncu)"})
    return roof


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=3)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    p.add_argument("--packets", type=float, default=1e8, help="packets per step per rank")
    p.add_argument("--gamma", type=float, default=2.0)
    p.add_argument("--max-events", type=float, default=1e6, help="per-packet event cap (capped packets reported)")
    p.add_argument("--plain-packets", type=float, default=1e6)
    p.add_argument("--cpu-seconds", type=float, default=15.0)
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--no-cpu", action="store_true")
    p.add_argument("--pda-stress", type=int, default=0,
                   help="instead of the transport step: PDA solve on an N x N grid of the same disk (HBM roofline)")
    p.add_argument("--pda-iters", type=int, default=2000)
    p.add_argument("--batch-sweep", action="store_true",
                   help="instead of the transport step: the 64-model batched sweep (one graph replay per step)")
    p.add_argument("--pda-adjoint", action="store_true",
                   help="instead of the transport step: PDA solve and adjoint on the 400x200 non-gray disk")
    p.add_argument("--raytrace", action="store_true",
                   help="instead of the transport step: ray-traced SED and image of the 200x120 disk at 45 degrees")
    p.add_argument("--scattering", action="store_true",
                   help="with --raytrace: keep the mean-intensity tally in the transport run (timed with and "
                        "without it) and add the scattered light to the source function")
    p.add_argument("--viscous", action="store_true",
                   help="instead of the transport step: packets released by viscous heating in the 200x120 disk")
    p.add_argument("--polarized", action="store_true",
                   help="instead of the transport step: polarized transport (Rayleigh Mueller matrix) vs unpolarized")
    p.add_argument("--profile-transport", action="store_true",
                   help="instead of the step: one transport call of --packets packets on the workload, its "
                        "statistics as JSON (the program the ncu captures of the transport kernels run)")
    p.add_argument("--no-accuracy", action="store_true", help="skip the equal-accuracy study")
    p.add_argument("--cpu-threads", type=int, default=0, help="oracle threads (0: every host core)")
    p.add_argument("--pda-min-visits", type=int, default=0,
                   help="PDA visit threshold; 0 scales the paper's 30 entries at 1e5 packets with the packet count "
                        "(Sect. 3.1 uses 30000 for its 1e8-packet runs)")
    return p.parse_args()


def workload():
    from paper_0902_3092_gb300 import disks
    return disks.config_thick_gray(200, 120, 1e6)


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms during the timed region."""
    FIELDS = ["index", "clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.active",
              "clocks_event_reasons.hw_slowdown", "clocks_event_reasons.hw_thermal_slowdown",
              "clocks_event_reasons.sw_thermal_slowdown", "clocks_event_reasons.sw_power_cap"]

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={','.join(self.FIELDS)}",
                                          "--format=csv,noheader,nounits", "-lms", "200", "-i", str(self.index)],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() in ("active", "1", "yes"):
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"], "samples": 0}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def physical_gpu(local_rank):
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        ids = [x for x in vis.split(",") if x.strip()]
        if local_rank < len(ids) and ids[local_rank].strip().isdigit():
            return int(ids[local_rank])
    return local_rank


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def host_threads(args):
    return args.cpu_threads or os.cpu_count() or 1


def cpu_baseline(d, gamma, budget_s, max_events, threads):
    """The FP64 oracle as it stands, on `threads` host threads (its packet-parallel mode): MRW transport of
    a bounded packet sample of the same disk for about `budget_s` seconds, then its PDA solve on those
    tallies; value = sample packets / transport seconds."""
    from oracle import oracle as O
    O.build()
    run = O.Run(d)
    # a short call sets the rate, then one call of the rest of the budget: each call waits for its longest
    # packet, so one long call keeps every thread busy
    t0 = time.perf_counter()
    n = 500 * threads
    run.run(n, seed=1, first_id=0, n_total=10 ** 8, mrw=True, gamma=gamma, want_sed=False, max_events=max_events,
            threads=threads)
    rate = n / (time.perf_counter() - t0)
    m = int(max(0.0, budget_s - (time.perf_counter() - t0)) * rate)
    if m > 0:
        run.run(m, seed=1, first_id=n, n_total=10 ** 8, mrw=True, gamma=gamma, want_sed=False, max_events=max_events,
                threads=threads)
        n += m
    t_tr = time.perf_counter() - t0
    T, err = run.temperatures()
    t1 = time.perf_counter()
    try:
        O.solve_pda(d, T, run.tally, run.visits, err)
        pda_ms = (time.perf_counter() - t1) * 1e3
    except ValueError:
        pda_ms = None
    return {"value": n / t_tr, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": f"{n} packets of the workload disk (MRW gamma={gamma}) in {t_tr:.1f} s on {threads} host "
                      f"threads (oracle packet-parallel mode); oracle PDA (scipy sparse direct) on those tallies "
                      f"{pda_ms if pda_ms is None else round(pda_ms, 1)} ms",
            "pda_ms": pda_ms}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from oracle import oracle as O
    O.build()
    d = workload()
    threads = host_threads(args)
    per_step = 5000 * threads
    # warm-up then timed steps: each step is a bounded sample of the workload (transport + temperatures + PDA)
    times = []
    for s in range(args.warmup + args.steps):
        run = O.Run(d)
        t0 = time.perf_counter()
        run.run(per_step, seed=1, first_id=s * per_step, n_total=10 ** 8, mrw=True, gamma=args.gamma,
                want_sed=False, max_events=int(args.max_events), threads=threads)
        T, err = run.temperatures()
        try:
            O.solve_pda(d, T, run.tally, run.visits, err)
        except ValueError:
            pass
        if s >= args.warmup:
            times.append(time.perf_counter() - t0)
    t = float(np.sum(times))
    v = per_step * args.steps / t
    line = {"metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * t / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "packets_per_step": per_step},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": f"{per_step} packets + temperatures + PDA per step, FP64 oracle, "
                                       f"{threads} host threads (packet-parallel mode)"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def profile_transport(args):
    """One FP32 MRW transport call of the workload (the program the ncu captures of the transport kernels
    run); prints its statistics, whose steps (events + crossings) turn the captured counts into per-step
    figures."""
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    d = workload()
    g = mcrt.Disk.from_model(d, device=0)
    n = int(args.packets)
    st = g.run_photons(n, seed=1, first_id=0, n_total=n, mrw=True, gamma=args.gamma, want_sed=True,
                       max_events=int(args.max_events))
    st = {k: v for k, v in st.items() if not k.startswith("guard_")}
    st["steps"] = st["events"] + st["crossings"]
    print(json.dumps({"profile_transport": {"workload": WORKLOAD, "packets": n, **st}}), flush=True)


def midplane_errors(T, T_ref, rows, sel):
    """RMS and maximum relative error of the midplane temperatures (the two polar rows next to theta =
    pi/2) over the cells `sel` (Sect. 3.1-3.2 compare temperatures this way)."""
    t, r = T[:, rows], T_ref[:, rows]
    ok = sel & (r > 0)
    rel = np.abs(t[ok] / r[ok] - 1.0)
    return float(np.sqrt(np.mean(rel ** 2))), float(rel.max()), int(ok.sum())


def equal_accuracy(g, d, args):
    """The speed-up of MRW + PDA over plain Monte Carlo at equal midplane-temperature accuracy (Sect. 3.1,
    3.2), on this GPU. On this disk plain Monte Carlo cannot serve as the reference: a packet that reaches
    the midplane inside a few AU needs 1e7-1e10 events, so with any practical event cap the packets that
    carry energy into the midplane are dropped and its temperature there converges to a value that is
    too low (raising the cap from 1e6 to 1e7 events lifts the 1-2 AU midplane from ~50 K to ~120 K). The
    reference is therefore the MRW transport at 5e8 packets in two independent halves, used in the midplane
    cells where the halves agree within 2 %; on the disks of midplane optical depth 1e4 and 1e5, where
    plain Monte Carlo without a cap converges, the MRW agrees with it to 1.5 % RMS in the midplane
    (tests/test_gpu_mrw_validation.py). Both methods are swept over packet counts (other seeds) with the
    benchmark's event cap; each point's time is the transport kernels' device time plus the PDA call. The
    accuracy level is the lowest RMS error both methods reach over those cells (plain MC: cells it never
    reaches count with their full error); each method's time to come within 5 % of it (relative) is
    interpolated in log-log between sweep points, and the ratio is plain MC's time over MRW + PDA's. (On
    the whole midplane the level is plain MC's floor, where its error no longer falls with more packets:
    the 5 % makes the time to reach it a property of the curve rather than of the noise of its flat end.)"""
    from paper_0902_3092_gb300 import mcrt
    cap = int(args.max_events)
    j = d.ntheta // 2
    rows = [j - 1, j]
    ref_n = 25 * 10 ** 7
    halves, t_ref = [], 0.0
    for h in range(2):
        g.reset()
        # (without the tail kernel the FP32 gray run is bitwise repeatable, so the reference, and the set of
        # cells where its halves agree, is the same in every bench run)
        st = g.run_photons(ref_n, seed=1000 + h, mrw=True, gamma=args.gamma, max_events=cap, want_sed=False,
                           tail_warps=-1)
        t_ref += st["seconds"]
        halves.append((np.frombuffer(g.checkpoint(), np.uint64).copy(), g.temperatures()[0]))
    comb = halves[0][0].copy()
    comb[8:] = halves[0][0][8:] + halves[1][0][8:]
    comb[5] = 2 * ref_n
    comb[6] = np.frombuffer(np.array([float(2 * ref_n)]).tobytes(), np.uint64)[0]
    g.restore(comb.tobytes())
    T_ref = g.temperatures()[0]
    h0, h1 = halves[0][1][:, rows], halves[1][1][:, rows]
    with np.errstate(divide="ignore", invalid="ignore"):
        conv = (h0 > 0) & (h1 > 0) & (np.abs(h0 / h1 - 1) <= 0.02)
    # the outer midplane, r >= 7 AU: there plain Monte Carlo with the event cap converges too (its runs
    # with a 1e6- and a 1e7-event cap agree within 1 %), so both methods are compared on equal terms
    rc = 0.5 * (d.r_faces_cm[1:] + d.r_faces_cm[:-1])
    outer = conv & (rc >= 7.0 * 1.495978707e13)[:, None]
    sweeps = {"plain MC": (False, False, [10 ** 5, 3 * 10 ** 5, 10 ** 6, 3 * 10 ** 6, 10 ** 7, 3 * 10 ** 7, 10 ** 8]),
              "MRW+PDA": (True, True, [3 * 10 ** 3, 10 ** 4, 3 * 10 ** 4, 10 ** 5, 3 * 10 ** 5, 10 ** 6, 3 * 10 ** 6,
                                       10 ** 7, 3 * 10 ** 7, 10 ** 8])}
    pts = {}
    for name, (mrw, pda, ns) in sweeps.items():
        pts[name] = []
        for n in ns:
            g.reset()
            st = g.run_photons(n, seed=77, mrw=mrw, gamma=args.gamma, max_events=cap, want_sed=False)
            t = st["seconds"]
            if pda:
                t0 = time.perf_counter()
                g.solve_pda(min_visits=max(30, int(round(30 * n / 1e5))))
                t += time.perf_counter() - t0
                T = g.temperatures(mcrt.T_PDA)[0]
            else:
                T = g.temperatures()[0]
            rms, mx, _ = midplane_errors(T, T_ref, rows, conv)
            rms_o, mx_o, _ = midplane_errors(T, T_ref, rows, outer)
            reached = int(np.sum(conv & (T[:, rows] > 0)))
            pts[name].append({"packets": n, "seconds": t, "rms": rms, "max": mx, "rms_outer": rms_o, "max_outer": mx_o,
                              "cells_reached": reached})

    def compare(key, tol=0.05):
        """The lowest error `key` both methods reach, the time each needs to come within `tol` of it, and
        the ratio."""
        level = max(min(p[key] for p in pts[k]) for k in pts)
        target = level * (1 + tol)
        reach = {}
        for k in pts:
            seq = pts[k]
            i = next(i for i, p in enumerate(seq) if p[key] <= target)
            t, n = seq[i]["seconds"], float(seq[i]["packets"])
            if i > 0 and seq[i - 1][key] > target and seq[i][key] < target:
                # between two sweep points: log time and log packets linear in log error
                a, b = seq[i - 1], seq[i]
                f = math.log(a[key] / target) / math.log(a[key] / b[key])
                t = math.exp(math.log(a["seconds"]) + f * math.log(b["seconds"] / a["seconds"]))
                n = math.exp(math.log(a["packets"]) + f * math.log(b["packets"] / a["packets"]))
            # the first sweep point already below the target: the time there bounds the time to reach it
            reach[k] = {"seconds": t, "packets": n, "upper_bound": i == 0 and seq[0][key] < target}
        up_p, up_m = reach["plain MC"]["upper_bound"], reach["MRW+PDA"]["upper_bound"]
        return {"level_rms": level, "target_rms": target, "plain_mc": reach["plain MC"], "mrw_pda": reach["MRW+PDA"],
                "speedup": reach["plain MC"]["seconds"] / reach["MRW+PDA"]["seconds"],
                "speedup_is_lower_bound": bool(up_m and not up_p), "speedup_is_upper_bound": bool(up_p and not up_m),
                "speedup_is_bounded_only": bool(up_p and up_m)}

    whole, out = compare("rms"), compare("rms_outer")
    best = min(pts["MRW+PDA"], key=lambda p: p["rms"])
    return {**whole, "cells": int(conv.sum()), "midplane_cells": int(2 * d.nr),
            "plain_mc_floor_rms": min(p["rms"] for p in pts["plain MC"]),
            "mrw_pda_best": {"rms": best["rms"], "packets": best["packets"], "seconds": best["seconds"]},
            "outer_midplane": {**out, "cells": int(outer.sum()), "region": "r >= 7 AU"},
            "reference": {"method": "MRW gamma=2, two independent halves", "packets": 2 * ref_n, "kernel_s": t_ref,
                          "cells": "midplane cells whose halves agree within 2 %",
                          "validation": "MRW vs plain MC without an event cap on the tau_mid=1e4 and 1e5 disks: "
                                        "1.5 % and 1.3 % RMS in the midplane"},
            "sweeps": pts, "event_cap": cap,
            "note": "time to come within 5 % of the lowest midplane RMS error both methods reach (interpolated "
                    "in log-log between sweep points); transport device time + PDA call; on the whole midplane "
                    "that level is plain MC's floor, set by the packets its event cap drops (the ones that heat "
                    "the inner midplane), which it does not pass with any number of packets while MRW+PDA goes "
                    "on to mrw_pda_best; outer_midplane: the same where plain MC converges too"}


# algorithmic bytes per PDA cell and FP32 CG iteration: kernel A reads r, p_old and the two couplings and
# writes p, Ap; kernel B reads p, Ap, y, r and writes y, r (4-byte values; neighbour values are re-reads)
PDA_BYTES_PER_CELL_ITER = 4 * (4 + 2) + 4 * (4 + 2)


def pda_stress(args):
    """PDA solve on an N x N grid of the benchmark disk made 100 times more massive (midplane optical
    depth 1e8), so that most cells of the midplane band |theta - pi/2| < 0.3 are optically thick at
    this resolution: synthetic Monte Carlo state whose band has no packet entries, so that its thick
    cells form the PDA region; times FP32 CG iterations."""
    import torch
    from paper_0902_3092_gb300 import disks, dist as D, mcrt
    n = args.pda_stress
    d = disks.make_disk(disks.log_r_faces(0.1, 100.0, n), disks.midplane_refined_theta_faces(n), disks.paper_star(),
                        disks.gray_opacity(), 1e8, name=f"thickgray{n}x{n}")
    rc, tc = disks.cell_centres(d.r_faces_cm, d.theta_faces)
    band = (np.abs(tc - np.pi / 2) < 0.3)[None, :] & (d.rho > 0)
    rf, tf = d.r_faces_cm, d.theta_faces
    V = (2 * np.pi / 3) * (rf[1:] ** 3 - rf[:-1] ** 3)[:, None] * (np.cos(tf[:-1]) - np.cos(tf[1:]))[None, :]
    T = 300.0 * (rc[:, None] / disks.AU_CM) ** -0.5 * (1 + 0.3 * np.cos(tc)[None, :] ** 2)
    n_total = 10 ** 9
    q = 4 * d.opacity.kappa_abs[0] * 5.6704e-5 * T ** 4
    # every dusty cell carries a tally (unused in the band); the dusty cells outside the band are the
    # Dirichlet cells that the band touches on both sides
    tally = np.where(d.rho > 0, np.maximum(np.floor(q * d.rho * V * n_total * 65536 / d.star.L), 1e4 * 65536),
                     0).astype(np.uint64)
    visits = np.where(band, 0, 10 ** 6).astype(np.uint64)
    z = np.zeros(n * n, np.uint64)
    blob = D.make_blob(n, n, d.opacity.nlam, tally, visits, z, np.zeros(d.opacity.nlam * 10, np.uint64), n_total,
                       n_total)
    g = mcrt.Disk.from_model(d)
    g.restore(blob)
    m = args.pda_iters

    def solve(k):
        # one refinement step of k CG iterations; the iteration budget ends it before convergence
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        npda, it = g.solve_pda(max_outer=1, max_inner=k, inner_tol=1e-30, allow_notconv=True)
        if it != k:
            raise RuntimeError(f"PDA stress: {it} CG iterations instead of {k}")
        return npda, time.perf_counter() - t0

    solve(2 * m)  # allocation, temperatures and first-touch outside the timed calls
    npda, t_a = solve(m)
    _, t_b = solve(2 * m)
    t_it = (t_b - t_a) / m  # the setup, the mask checks and the final residual cancel
    byts = PDA_BYTES_PER_CELL_ITER * npda
    mp = measured_peaks()
    peak = mp.get("hbm_gbs", 6800.0) * 1e9
    peak_src = "measured (MEASURED_PEAKS.json hbm_gbs)" if "hbm_gbs" in mp else "fallback (6.8 TB/s copy, one earlier GB300 measurement)"
    line = {"metric": "PDA FP32 CG iteration bandwidth (stress grid)", "value": byts / t_it / 1e9, "unit": "GB/s",
            "n_gpus": 1, "higher_is_better": True, "dtype": "f32", "data": "synthetic",
            "config": {"workload": f"PDA on a {n}x{n} gray disk of midplane optical depth 1e8, thick cells of the "
                                   "midplane band |theta-pi/2|<0.3",
                       "cells": n * n, "pda_cells": npda, "cg_iterations_timed": args.pda_iters},
            "us_per_iteration": 1e6 * t_it, "setup_ms": 1e3 * (t_a - m * t_it),
            "roofline": {"bound": "hbm", "achieved": byts / t_it / 1e9, "peak": peak / 1e9, "unit": "GB/s",
                         "frac": byts / t_it / peak, "peak_source": peak_src, "traffic": None,
                         "note": f"{PDA_BYTES_PER_CELL_ITER} B per PDA cell per iteration (kernels A+B), "
                                 "host-timed difference of two solves"}}
    print(json.dumps(line), flush=True)


def batch_sweep_timing(args):
    """The batched sweep: 64 non-gray models of uneven grid, optical depth (1e2-1e6) and packet budget
    (1e5-1e7 each) from seed 1, MRW gamma = 2, in one persistent launch replayed from a CUDA graph whose
    launch shape the autotuner picked; packets/s over the whole batch (CUDA-event launch time)."""
    import torch
    from paper_0902_3092_gb300 import disks, mcrt
    ds, npk = disks.batch_sweep(64, seed=1)
    gs = [mcrt.Disk.from_model(d) for d in ds]
    B = mcrt.Batch(gs, npk, mrw=True, gamma=args.gamma, max_events=int(args.max_events), want_sed=False)
    cfg = B.config()
    for s in range(max(1, args.warmup)):
        B.run(seed=100 + s)
    secs, events, capped = [], 0, 0
    for s in range(args.steps):
        for g in gs:
            g.reset()
        torch.cuda.synchronize()
        st = B.run(seed=1 + s)
        secs.append(max(x["seconds"] for x in st))
        events += sum(x["events"] for x in st)
        capped += sum(x["capped"] for x in st)
    total = int(sum(npk))
    line = {"metric": "photon packets/s, 64-model batched sweep (one graph launch)", "unit": "packets/s",
            "value": total / float(np.mean(secs)), "higher_is_better": True, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * float(np.mean(secs)), "dtype": "f32", "data": "synthetic",
            "config": {"workload": "64 non-gray disks nr 50-300 x ntheta 30-180, tau_mid 1e2-1e6, MRW gamma=2",
                       "packets_per_step": total, "autotuned": cfg},
            "events_per_s": events / float(np.sum(secs)), "capped_fraction": capped / (total * args.steps)}
    print(json.dumps(line), flush=True)


def pda_adjoint_timing(args):
    """PDA forward solve and adjoint on the 400 x 200, tau_mid = 1e6 non-gray disk (the differentiable
    PDA case) after a 1e7-packet MRW run; J = mean midplane temperature. Host-timed calls, 5 repeats."""
    import torch
    from paper_0902_3092_gb300 import disks, mcrt
    d = disks.config_pda_adjoint(400, 200, 1e6)
    g = mcrt.Disk.from_model(d)
    g.run_photons(10_000_000, seed=1, mrw=True, gamma=2.0, max_events=10 ** 6, want_sed=False)
    w = np.zeros((d.nr, d.ntheta))
    j = d.ntheta // 2
    w[:, j - 1:j + 1] = 1.0 / (2 * d.nr)
    fw, bw, res = [], [], None
    for _ in range(6):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        res = g.solve_pda(min_visits=3000)
        t1 = time.perf_counter()
        g.pda_adjoint(w)
        t2 = time.perf_counter()
        fw.append(t1 - t0)
        bw.append(t2 - t1)
    fw, bw = fw[1:], bw[1:]  # the first call allocates
    line = {"metric": "PDA forward + adjoint time (400x200 non-gray disk, tau_mid=1e6)", "unit": "ms",
            "value": 1e3 * (np.median(fw) + np.median(bw)), "higher_is_better": False, "n_gpus": 1,
            "dtype": "f32 CG under f64 refinement", "data": "synthetic",
            "config": {"workload": "400x200 non-gray disk, 1e7 MRW packets, PDA threshold 3000 entries",
                       "pda_cells": res[0], "cg_iterations_forward": res[1]},
            "forward_ms": 1e3 * float(np.median(fw)), "adjoint_ms": 1e3 * float(np.median(bw))}
    print(json.dumps(line), flush=True)


def raytrace_timing(args):
    """Ray-traced SED and image (Sect. 2.3, 4.1) of the 200 x 120 rim-refined tau_mid = 1e6 gray disk at 45
    degrees and 140 pc, after a 1e7-packet MRW run (Monte Carlo temperatures): 104,448 rays (16 rings
    inside r_in, 4 per radial cell, 128 azimuths) x 100 wavelength bins, FP32. Timed: one mcrt_raytrace
    call (trace + star + SED) per step with CUDA events on the disk's stream, L2 flushed before each;
    the source table is built once (the temperatures do not change between views). --scattering: the
    transport run keeps the mean-intensity tally (its device time reported beside the same run without
    it) and the source function adds the scattered light sigma J / chi."""
    import torch
    from paper_0902_3092_gb300 import disks, mcrt
    d = disks.config_thick_gray(200, 120, 1e6)
    st = torch.cuda.Stream()
    g = mcrt.Disk.from_model(d, stream=st.cuda_stream)
    scat = bool(args.scattering)
    transport_s = {}
    for keep in ((False, True) if scat else (False,)):
        g.keep_mean_intensity(keep)  # resets the tallies
        s = g.run_photons(10_000_000, seed=1, mrw=True, gamma=2.0, max_events=10 ** 6, want_sed=scat)
        transport_s["with_j_tally" if keep else "plain"] = s["seconds"]
    rays = disks.polar_rays(d.r_faces_cm, n_sub=4, n_phi=128, n_inner=16)
    incl, dist = math.pi / 4, 140 * 3.0856775814913673e18
    g.set_rays(incl, dist, rays)
    out = g.raytrace(scattering=scat)  # source table and buffers
    flush = torch.empty(256 * 2 ** 20, dtype=torch.uint8, device="cuda")
    times = []
    with ClockSampler(physical_gpu(0)) as clk:
        for k in range(args.warmup + args.steps):
            with torch.cuda.stream(st):
                flush.zero_()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(st)
                out = g.raytrace(scattering=scat)
                e1.record(st)
            torch.cuda.synchronize()
            if k >= args.warmup:
                times.append(e0.elapsed_time(e1) * 1e-3)
    t = float(np.mean(times))
    n_bins = d.opacity.nlam
    seg = out["segments"]
    # end to end through the host C ABI: rays from host memory, trace, SED back to the host
    e2e = []
    for k in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        g.set_rays(incl, dist, rays)
        o2 = g.raytrace(scattering=scat)
        e2e.append(time.perf_counter() - t0)
    t_e2e = float(np.median(e2e))
    peaks = measured_peaks()
    clocks = clk.summary()
    roof = ray_roofline(seg, t, clocks["sm_mhz"] or 2070.0)
    # the oracle on the host cores: rays one by one for about ten seconds
    cpu = None
    if not args.no_cpu:
        from oracle import oracle as O
        from oracle import raytrace as ORT
        O.build()
        T, _, _ = g.temperatures()
        S = ORT.source(d, T)
        rng = np.random.default_rng(0)
        t0, k = time.perf_counter(), 0
        while time.perf_counter() - t0 < 10.0:
            j = int(rng.integers(rays.n))
            ORT.intensity(d, T, incl, rays.p[j], rays.q[j], S)
            k += 1
        cpu = {"value": k / (time.perf_counter() - t0), "unit": "rays/s", "cores": 1, "kind": "oracle",
               "sample": f"{k} random rays of the workload, all {n_bins} bins, FP64 numpy oracle, one core "
                         "(source table built outside the timing)"}
    line = {"metric": "ray-traced rays/s (SED + image, all wavelength bins)", "value": rays.n / t, "unit": "rays/s",
            "higher_is_better": True, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * t, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "200x120 rim-refined gray disk, tau_mid=1e6, 1e7 MRW packets; 45 deg, 140 pc",
                       "rays": rays.n, "wavelength_bins": n_bins, "segments": seg, "l2": "flushed (256 MB write)"},
            "e2e": {"value": rays.n / t_e2e, "unit": "rays/s", "h2d_bytes_per_step": 3 * 8 * rays.n,
                    "d2h_bytes_per_step": 16 * n_bins},
            "roofline": roof, "cpu_baseline": cpu, "clocks": clocks, "gpu_launches": 3 * args.steps,
            "flux_total_erg_s_cm2": float(out["F"].sum())}
    if scat:
        line["config"]["scattering"] = "mean-intensity tally, sigma J / chi in the source function"
        line["transport_seconds"] = transport_s
    print(json.dumps(line), flush=True)


def viscous_timing(args):
    """Viscous heating (Sect. 5): packets released inside the 200 x 120 rim-refined tau_mid = 1e6 gray
    disk by the steady accretion dissipation of disks.viscous_sources (scaled to 1e4 L* so that the
    star's packets are 1e-4 of all), transported with MRW (gamma = 1, the paper's setting) and, for
    comparison, without it under a 1e6-event cap. Timed: reset + transport of 2e5 packets per step with
    CUDA events on the disk's stream."""
    import torch
    from paper_0902_3092_gb300 import disks, mcrt
    d = disks.config_thick_gray(200, 120, 1e6)
    L = disks.viscous_sources(d)
    L *= 1e4 * d.star.L / L.sum()
    st = torch.cuda.Stream()
    g = mcrt.Disk.from_model(d, stream=st.cuda_stream)
    g.set_sources(L)
    n = 200_000
    cap = 10 ** 6
    g.run_photons(20_000, seed=99, mrw=True, gamma=1.0, max_events=cap, want_sed=False)
    times, stats = [], None
    with ClockSampler(physical_gpu(0)) as clk:
        for k in range(args.warmup + args.steps):
            with torch.cuda.stream(st):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(st)
                g.reset()
                stats = g.run_photons(n, seed=1 + k, mrw=True, gamma=1.0, max_events=cap, want_sed=False)
                e1.record(st)
            torch.cuda.synchronize()
            if k >= args.warmup:
                times.append(e0.elapsed_time(e1) * 1e-3)
    t = float(np.mean(times))
    # plain Monte Carlo (no MRW) on the same sources
    n_plain = 20_000
    g.reset()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    sp = g.run_photons(n_plain, seed=7, mrw=False, max_events=cap, want_sed=False)
    tp = time.perf_counter() - t0
    line = {"metric": "viscous-heating packets/s (released in the disk, MRW gamma=1)", "value": n / t,
            "unit": "packets/s", "higher_is_better": True, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * t, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "200x120 rim-refined gray disk, tau_mid=1e6, steady accretion dissipation "
                                   "(scaled to 1e4 L*), MRW gamma=1", "packets_per_step": n,
                       "max_events_per_packet": cap},
            "events_per_packet": stats["events"] / n, "mrw_jumps_per_packet": stats["mrw_jumps"] / n,
            "capped_fraction": stats["capped"] / n, "us_per_packet": 1e6 * t / n,
            "plain_mc": {"packets": n_plain, "packets_per_s": n_plain / tp, "us_per_packet": 1e6 * tp / n_plain,
                         "capped_fraction": sp["capped"] / n_plain, "events_per_packet": sp["events"] / n_plain},
            "clocks": clk.summary()}
    print(json.dumps(line), flush=True)


def polarized_timing(args):
    """Polarized transport (Sect. 2.3): the 200 x 120 rim-refined tau_mid = 1e6 gray disk with the exact
    Rayleigh Mueller matrix in every bin, MRW (gamma = 2), 1e7 packets per step, FP32; timed with CUDA
    events on the disk's stream (reset + transport), against the same run without polarization."""
    import torch
    from paper_0902_3092_gb300 import disks, mcrt
    d = disks.config_thick_gray(200, 120, 1e6)
    st = torch.cuda.Stream()
    g = mcrt.Disk.from_model(d, stream=st.cuda_stream)
    n = 10_000_000

    def timed(pol):
        g.set_mueller(disks.rayleigh_mueller(d.opacity.nlam, 181) if pol else None)
        g.run_photons(n // 10, seed=99, mrw=True, gamma=2.0, max_events=10 ** 6)
        ts, stats = [], None
        for k in range(args.warmup + args.steps):
            with torch.cuda.stream(st):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(st)
                g.reset()
                stats = g.run_photons(n, seed=1 + k, mrw=True, gamma=2.0, max_events=10 ** 6)
                e1.record(st)
            torch.cuda.synchronize()
            if k >= args.warmup:
                ts.append(e0.elapsed_time(e1) * 1e-3)
        return float(np.mean(ts)), stats

    with ClockSampler(physical_gpu(0)) as clk:
        t_pol, s_pol = timed(True)
        t_unp, _ = timed(False)
    g.set_mueller(disks.rayleigh_mueller(d.opacity.nlam, 181))
    g.run_photons(n, seed=1, mrw=True, gamma=2.0, max_events=10 ** 6)
    I, Q, U = (x.sum(axis=0) for x in g.sed_stokes())
    line = {"metric": "polarized packets/s (Rayleigh Mueller matrix, MRW gamma=2)", "value": n / t_pol,
            "unit": "packets/s", "higher_is_better": True, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * t_pol, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "200x120 rim-refined gray disk, tau_mid=1e6, albedo 0.5, Rayleigh Mueller matrix",
                       "packets_per_step": n},
            "unpolarized_packets_per_s": n / t_unp, "scatterings_per_packet": s_pol["scatterings"] / n,
            "Q_over_I_by_inclination": [float(x) for x in Q / I], "clocks": clk.summary()}
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    if args.profile_transport:
        profile_transport(args)
        return
    if args.pda_stress:
        pda_stress(args)
        return
    if args.pda_adjoint:
        pda_adjoint_timing(args)
        return
    if args.batch_sweep:
        batch_sweep_timing(args)
        return
    if args.raytrace:
        raytrace_timing(args)
        return
    if args.viscous:
        viscous_timing(args)
        return
    if args.polarized:
        polarized_timing(args)
        return
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    from paper_0902_3092_gb300 import build, mcrt
    build.build()
    d = workload()
    stream = torch.cuda.current_stream()
    g = mcrt.Disk.from_model(d, device=local, stream=stream.cuda_stream)
    Np = int(args.packets)
    ncell = d.nr * d.ntheta
    min_visits = args.pda_min_visits or max(30, int(round(30 * Np * world / 1e5)))

    from paper_0902_3092_gb300 import dist as D

    def combine():
        if world == 1:
            return
        # the exchange of the Monte Carlo step: integer tallies summed over ranks (exact in int64)
        g.restore(D.allreduce_blob(g.checkpoint()))

    guard_records = []

    def step(i):
        g.reset()
        first, _ = D.packet_range(rank, world, Np, i)
        try:
            # the rank's share is a run of its own (n_total = its packets); the exchange reads the summed
            # tallies with the total packet count
            st = g.run_photons(Np, seed=1, first_id=first, n_total=Np, mrw=True,
                               gamma=args.gamma, want_sed=True, max_events=int(args.max_events))
        except mcrt.McrtError as e:
            # a step guard dropped packets: the call still completed (the dropped packets count as capped);
            # keep its statistics and report the record of the first dropped packet
            if e.status != 5 or not getattr(e, "stats", None):
                raise
            st = e.stats
            guard_records.append({k: st[k] for k in ("guarded", "guard_packet", "guard_kind", "guard_in_tail",
                                                      "guard_cell", "guard_pos_cm", "guard_dir")})
        combine()
        n_pda, iters = g.solve_pda(min_visits=min_visits)
        return st, n_pda, iters

    flush = torch.empty(512 * 1024 * 1024, dtype=torch.uint8, device="cuda")
    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    stats = []
    l0 = g.launch_count()
    with ClockSampler(physical_gpu(local)) as clk:
        for i in range(args.steps):
            flush.fill_(i & 0xFF)  # L2 flush between timed steps, outside the timed region
            ev[i][0].record(stream)
            stats.append(step(args.warmup + i))
            ev[i][1].record(stream)
        torch.cuda.synchronize()
    launches = g.launch_count() - l0
    step_ms = [a.elapsed_time(b) for a, b in ev]
    t_local = float(np.sum(step_ms)) / 1e3
    if world > 1:
        tt = torch.tensor([t_local], dtype=torch.float64, device="cuda")
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        t_max = float(tt.item())
    else:
        t_max = t_local
    value = Np * world * args.steps / t_max
    tr_s = [s[0]["seconds"] for s in stats]
    ev_steps = [s[0]["events"] + s[0]["crossings"] for s in stats]
    pda_ms = [ms - 1e3 * ts for ms, ts in zip(step_ms, tr_s)]
    s0 = stats[-1][0]

    # plain Monte Carlo on the same disk (no MRW, no PDA), same per-packet event cap
    Npl = int(args.plain_packets)
    g.reset()
    stp = g.run_photons(Npl, seed=2, first_id=0, mrw=False, max_events=int(args.max_events), want_sed=True)
    plain = {"packets_per_s": Npl / stp["seconds"], "kernel_s": stp["seconds"], "packets": Npl,
             "events": stp["events"], "capped": stp["capped"], "event_cap": int(args.max_events),
             "max_packet_steps": stp["max_packet_steps"]}

    # end to end through the host C ABI: create from host arrays, transport, temperatures, PDA, read T
    e2e = None
    if not args.no_e2e:
        op = d.opacity
        h2d = 8 * (len(d.r_faces_cm) + len(d.theta_faces) + d.rho.size + len(op.lam_edges_um) + 3 * op.nlam)
        d2h = 3 * 8 * ncell
        torch.cuda.synchronize()
        te = []
        for i in range(args.steps):
            t0 = time.perf_counter()
            h = mcrt.Disk.from_model(d, device=local)
            h.run_photons(Np, seed=1, first_id=(rank + world * i) * Np, n_total=Np, mrw=True, gamma=args.gamma,
                          max_events=int(args.max_events))
            h.solve_pda(min_visits=min_visits)
            T, _, _ = h.temperatures(mcrt.T_PDA)
            h.close()
            te.append(time.perf_counter() - t0)
        t_e2e = float(np.sum(te))
        if world > 1:
            tt = torch.tensor([t_e2e], dtype=torch.float64, device="cuda")
            dist.all_reduce(tt, op=dist.ReduceOp.MAX)
            t_e2e = float(tt.item())
        e2e = {"value": Np * world * args.steps / t_e2e, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(d2h)}

    peaks = measured_peaks()
    clocks = clk.summary()
    roofline = transport_roofline(float(np.mean(ev_steps)), float(np.mean(tr_s)), clocks, peaks)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline(d, args.gamma, args.cpu_seconds, int(args.max_events), host_threads(args))

    acc = None
    if rank == 0 and world == 1 and not args.no_accuracy:
        acc = equal_accuracy(g, d, args)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": 1e3 * t_max / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": {"workload": WORKLOAD, "packets_per_step_per_rank": Np, "grid": [d.nr, d.ntheta],
                           "tau_mid": 1e6, "gamma": args.gamma, "mrw_min_interactions": 20,
                           "max_events_per_packet": int(args.max_events), "pda_min_visits": min_visits,
                           "pda_max_rel_err": 0.05,
                           "l2": "flushed between timed steps (512 MiB write outside the timed region)",
                           "parallelism": f"packet ranges per rank, int64 tally all-reduce" if world > 1 else "1 GPU"},
                "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": int(launches),
                "clocks": clocks, "equal_accuracy": acc,
                "transport": {"kernel_ms_per_step": 1e3 * float(np.mean(tr_s)), "events": s0["events"],
                              "crossings": s0["crossings"], "mrw_jumps": s0["mrw_jumps"], "capped": s0["capped"],
                              "capped_fraction": s0["capped"] / Np, "max_packet_steps": s0["max_packet_steps"],
                              "events_per_s": s0["events"] / s0["seconds"], "error_flags": s0["error_flags"],
                              "guarded_packets": int(sum(s[0]["guarded"] for s in stats)),
                              "guard_records": guard_records[:3]},
                "pda": {"ms_per_step": float(np.mean(pda_ms)), "cells": stats[-1][1], "cg_iterations": stats[-1][2]},
                "plain_mc": plain, "peaks_file": bool(peaks)}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
