#!/usr/bin/env python3
"""Throughput of the hybrid LB/FD step on GB300.

Workload (default, cube384): the 3D form of the method, D3Q19 on 384^3 sites,
FP32 state (populations stored as deviations from w_i n0), periodic in x and
y, cold walls at z = 0 and 383 (bounce-back, T_w = 0.5), Tc = 1, T0 = 1.1,
b = 1, kappa = -0.025, c = 0.02, Gamma = 0.05, xi = 1e-3, tau = 0.6, phi
i.i.d. uniform in [-0.05, 0.05] (synthetic, seeded).  One benchmark step is
one time step of the method (one lf_step(ctx, 1) call: the three passes of
the 3D step).  The state (2 x 9.5 GB) is far larger than the 129 MB L2.

prec1024 is the 2D precision form (D2Q9, 1024 x 1024, xi = 1e-3, tau = 1, one
fused kernel per step); its state (2 x 44 MiB) fits in L2, so a 256 MiB buffer
is written (and another read) before every timed step.  Each step is timed
alone with CUDA events on the library's stream.

Metric: MLUPS = 1e-6 x sites x steps / s (million lattice-site updates per
second), whole job over all ranks.  --impl reference times the FP64 CPU oracle
on the host cores instead (the only reference this method has).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

BYTES_PER_SITE = {("fp32", 2): 88, ("fp64", 2): 176, ("fp32", 3): 168, ("fp64", 3): 336}
METRIC = "coupled LB+FD MLUPS"


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as fh:
            j = json.load(fh)
        return float(j["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def ranks():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def max_over_ranks(x: float, device=None) -> float:
    """The largest value of x over all ranks (every rank gets it); x itself
    without an initialised process group of more than one rank."""
    import torch
    import torch.distributed as tdist
    if not (tdist.is_available() and tdist.is_initialized()) or tdist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], device=device, dtype=torch.float64)
    tdist.all_reduce(t, op=tdist.ReduceOp.MAX)
    return float(t.item())


def job_rate(units_per_rank: float, steps: int, world: int, seconds: float) -> float:
    """Whole-job throughput in millions of units per second: the units of all
    ranks (each rank runs its own replica) over the slowest rank's time."""
    return 1e-6 * units_per_rank * steps * world / seconds


class Clocks:
    """nvidia-smi samples during the timed region."""

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            import atexit
            atexit.register(self.__exit__)   # never leave the sampler running
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def window(self, t0, t1):
        """keep only the samples taken between t0 and t1 (host clock)."""
        self.lines = [(ts, ln) for ts, ln in self.lines if t0 <= ts <= t1]

    def summary_over(self, timed, run, min_samples=5):
        """Clock summary of the timed window (t0, t1) when it holds at least
        `min_samples` samples, else of the whole GPU run (warm-up, timed
        steps and the end-to-end leg), which short timed regions need."""
        keep = self.lines
        self.window(*timed)
        out = self.summary()
        out["window"] = "timed steps"
        if out["samples"] < min_samples:
            self.lines = [(ts, ln) for ts, ln in keep if run[0] <= ts <= run[1]]
            out = self.summary()
            out["window"] = "whole GPU run (warm-up, timed steps, end-to-end leg)"
        self.lines = keep
        return out

    def __exit__(self, *a):
        if self.proc and self.proc.poll() is None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for _, ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                smax = float(parts[1])
            except ValueError:
                continue
            for nm, v in zip(names, parts[4:8]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


def oracle_rate(nx, ny, xi, seconds=10.0, max_steps=10000, d=2, nz=1, tau=1.0, stencil=0, restore=0):
    """The FP64 CPU oracle as it stands on a bounded sample: steps of an
    nx x ny (x nz) lattice with the workload's physics, for about `seconds`.
    With `restore` > 0 the initial quench is taken up again every `restore`
    steps (outside the timed intervals), as the GPU workload does, so that
    every timed step advances a finite state."""
    from oracle import oracle as O

    cfg = O.make_cfg(d=d, nx=nx, ny=ny, nz=nz, xi=xi, tau=tau, stencil=stencil)
    st0 = O.init(cfg)
    st = O.run(st0, 1)   # warm: compile/load, first touch
    steps, el, since = 0, 0.0, 1
    chunk = 1
    while el < seconds and steps < max_steps:
        if restore > 0 and since + chunk > restore:
            st, since = st0.copy(), 0
            chunk = min(chunk, restore)
        t0 = time.perf_counter()
        st = O.run(st, chunk)
        el += time.perf_counter() - t0
        steps += chunk
        since += chunk
        if el < seconds / 4:
            chunk *= 2
    return 1e-6 * nx * ny * nz * steps / el, steps, el, O.threads()


def run_reference(args):
    """The oracle as it stands, on the host cores, on a bounded sample of the
    workload: 256x256 of the 2D quench, 64^3 of the 3D one (same physics and
    stencils)."""
    rank, world, _ = ranks()
    if rank != 0:
        return 0
    if args.workload in ("ens96", "sur256"):
        print(json.dumps({"impl": "reference", "unavailable": "the oracle times single lattices; the ensemble and "
                          "surrogate workloads have no CPU reference arm (their baselines are the single-run GPU "
                          "path, reported in their own lines)"}), flush=True)
        return 0
    from oracle import oracle as O

    iso = int(args.stencil == "isotropic")
    if args.workload == "cube384":
        d, nx, ny, nz, tau = 3, 64, 64, 64, 0.6
        full = f"cube384: 3D D3Q19 lamellar quench between cold walls (z), sampled as {nx}x{ny}x{nz} per step"
    else:
        d, nx, ny, nz, tau = 2, 256, 256, 1, 1.0
        full = f"prec1024: 2D D2Q9 lamellar quench between cold walls, sampled as {nx}x{ny} per step"
    if iso:
        full += ", isotropic stencils"
    cfg = O.make_cfg(d=d, nx=nx, ny=ny, nz=nz, xi=args.xi, tau=tau, stencil=iso)
    st = O.init(cfg)
    for _ in range(args.warmup):
        st = O.run(st, 1)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        st = O.run(st, 1)
    el = time.perf_counter() - t0
    sites = nx * ny * nz
    value = 1e-6 * sites * args.steps / el
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": full, "sites_per_step": sites, "grid": [nx, ny, nz][:d], "xi": args.xi, "tau": tau},
        "cpu_baseline": {"value": value, "unit": "MLUPS", "cores": O.threads(), "kind": "oracle",
                         "sample": f"{args.steps} FP64 oracle steps of a {'x'.join(map(str, [nx, ny, nz][:d]))} "
                                   f"lattice (same physics as the full workload), OpenMP over rows"},
        "e2e": {"value": value, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def traffic_for(kernel: str, param: int):
    """(DRAM bytes per launch, the shape they were captured at) from the committed
    ncu summary, if it still describes the current kernel source: those of the
    shape of `param` (key suffix _p<param>), else of the default shape (no suffix),
    which moves the same fields; (None, None) without either."""
    for shape, key in ((f"param {param}" if param else "default", f"{kernel}_p{param}" if param else kernel),
                       ("default", kernel)):
        b = _captured_bytes(key)
        if b is not None:
            return b, shape
    return None, None


def _captured_bytes(kernel_key: str):
    import hashlib
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as fh:
        j = json.load(fh)
    ent = j.get(kernel_key)
    if not ent:
        return None
    srcs = ent["source"] if isinstance(ent["source"], list) else [ent["source"]]
    data = b"".join(open(os.path.join(ROOT, s_), "rb").read() for s_ in srcs)
    h = hashlib.sha256(data).hexdigest()[:16]
    return ent["dram_bytes_per_launch"] if h == ent.get("source_sha256_16") else None


def run_ensemble(args):
    """96 independent runs (mixed sizes, xi, tau): batched (one graph-replayed
    persistent launch per step, shapes from the ensemble autotuner) against
    the same runs stepped one after another by lf_step at their own tuned
    shapes; results equal to FP32 rounding, compared at the end.  Runs whose state goes non-finite (fast
    quenches at tau = 0.6 diverge for the method itself) are retired every
    --ens-prune-every steps, in both arms, and only the runs still finite at
    the end of a block of steps count towards the rate."""
    import numpy as np
    import torch

    from paper_1102_3094_gb300 import lf, synth

    rank, world, local = ranks()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:                       # one replica of the whole ensemble per GPU
        import torch.distributed as tdist
        tdist.init_process_group("nccl")
    stream = torch.cuda.Stream(dev)
    members = synth.ensemble_members()
    if args.stencil == "isotropic":
        members = [dict(m, stencil="isotropic") for m in members]
    sites_r = [m["nx"] * m["ny"] for m in members]
    sites = sum(sites_r)
    with torch.cuda.stream(stream):
        ens = lf.Ensemble(members, stream=stream)
        t0 = time.time()
        ens.tune(reps=5)
        tune_s = time.time() - t0
        shapes = {}
        for r, m in enumerate(members):
            pr = ens.param(r)
            shapes[f"{m['nx']}x{m['ny']}" + ("-iso" if m.get("stencil") == "isotropic" else "")] = \
                {"cta_threads": 64 if pr >> 16 else 128, "rows": pr & 0xFFFF}
        # the plain single-run path at its own best shapes (lf_tune, cached per lattice size)
        singles = [lf.Lattice(precision="fp32", stream=stream, **m) for m in members]
        single_shapes = {}
        for r, s_ in enumerate(singles):
            v_, p_, _ = s_.tune(reps=3)
            single_shapes[f"{members[r]['nx']}x{members[r]['ny']}" + ("-iso" if members[r].get("stencil") else "")] = \
                {"variant": v_, "param": p_}
        ens.step(args.warmup)
        for s_ in singles:
            s_.step(args.warmup)
        torch.cuda.synchronize(dev)
        live = [True] * len(members)
        live_s = [True] * len(members)
        ens.prune()
        for r in range(len(members)):
            live[r] = ens.active(r)
            live_s[r] = not singles[r].diag()["nonfinite"]
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        clk = Clocks(local)
        t_batch = t_seq = 0.0
        site_steps = 0
        left = args.steps
        block = args.ens_prune_every if args.ens_prune_every > 0 else args.steps
        with clk:
            time.sleep(0.5)
            tb = time.time()
            while left > 0:
                k = min(block, left)
                ev[0].record(stream)
                ens.step(k)
                ev[1].record(stream)
                ev[2].record(stream)
                for r, s_ in enumerate(singles):
                    if live_s[r]:
                        s_.step(k)
                ev[3].record(stream)
                torch.cuda.synchronize(dev)
                t_batch += ev[0].elapsed_time(ev[1]) / 1e3
                t_seq += ev[2].elapsed_time(ev[3]) / 1e3
                ens.prune()
                for r in range(len(members)):
                    live[r] = ens.active(r)
                    if live_s[r]:
                        live_s[r] = not singles[r].diag()["nonfinite"]
                site_steps += k * sum(sr for sr, a in zip(sites_r, live) if a)
                left -= k
            te = time.time()
        clk.window(tb, te + 0.15)
        t_batch = max_over_ranks(t_batch, dev)
        t_seq = max_over_ranks(t_seq, dev)
        # the two arms split the rows differently (each at its own best shape), so
        # they agree to FP32 rounding, not bit for bit: compare what the runs are
        # for, the structure factor peak and the order parameter field
        sk_err, l2_err = 0.0, 0.0
        for r in range(len(members)):
            if not (live[r] and live_s[r]):
                continue
            da, db = ens.run(r).diag(), singles[r].diag()
            sk_err = max(sk_err, abs(da["k_peak"] / db["k_peak"] - 1), abs(da["s_peak"] / db["s_peak"] - 1))
            a = ens.run(r).get("phi", "fp32")
            b = singles[r].get("phi", "fp32")
            l2_err = max(l2_err, float(np.linalg.norm(a - b) / np.linalg.norm(b)))
        n_live = sum(live)
        same_retirement = live == live_s
    value = 1e-6 * site_steps * world / t_batch
    peak, peak_kind = peaks()
    achieved = 88 * site_steps / t_batch / 1e9
    line = {
        "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * t_batch / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "ens96: 96 independent 2D runs, 24 each of 128^2, 256^2, 384^2, 512^2, xi "
                               "log-uniform in [1e-4, 1], tau in {0.6, 1, 3}, one persistent launch per step "
                               "replayed from a CUDA graph, CTA width and segment height from the autotuner"
                               + (", isotropic 9-point stencils (two-lane isotropic march items)" if args.stencil == "isotropic" else ""),
                   "sites_per_step_all_runs": sites, "tuned_shapes": shapes,
                   "sequential_shapes": single_shapes,
                   "l2": "inputs (1 GB of state) larger than L2",
                   "rate_counts": "site updates of the runs still finite at the end of each block of "
                                  f"{block} steps (non-finite runs retired between blocks, outside the timing)"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": None, "peak_kind": peak_kind, "algorithmic_bytes_per_site": 88,
                     "kernel": ("k_ens_march2d_iso" if args.stencil == "isotropic" else "k_ens_march2d")
                               + " (+ k_ens_tsub2d for runs with xi/nsub sub-steps)"},
        "batched_vs_sequential": {"t_batched_s": t_batch, "t_sequential_s": t_seq, "speedup": t_seq / t_batch,
                                  "max_sk_peak_err": sk_err, "max_phi_rel_l2": l2_err, "tune_s": tune_s,
                                  "what": "time to solution of the same runs and steps: batched against one "
                                          "after another by lf_step at each run's own tuned shape; S(k) peak "
                                          "position/height and phi compared at the end over the finite runs",
                                  "runs_finite_at_end": n_live, "runs_retired": len(members) - n_live,
                                  "same_runs_retired_in_both_arms": same_retirement,
                                  "note": "runs with tau = 0.6 and fast quenches diverge for the method itself at "
                                          "these parameters (the CPU oracle diverges the same way); both arms "
                                          "retire them at the same block boundaries"},
        "clocks": clk.summary(),
    }
    if world > 1:
        line["config"]["parallelism"] = f"replicas x{world} (the whole ensemble on every GPU)"
    if rank == 0:
        print(json.dumps(line), flush=True)
    ens.close()
    for s_ in singles:
        s_.close()
    if world > 1:
        import torch.distributed as tdist
        tdist.destroy_process_group()
    return 0


def run_surrogate(args):
    """Learned surrogate at 256 x 256.  Trajectories of the plain solver (one
    ensemble, xi log-uniform in [1e-4, 1]) are kept on the device as states
    every K steps; consecutive states form the (state, state K steps later)
    training pairs.  Whole trajectories are held out for the accuracy test,
    optionally with a learning curve over the amount of training data.  Then a
    fresh run is advanced plain-only and interleaved 1:1 with the surrogate,
    every surrogate window checked by a plain shadow window at the 2 %
    threshold; the time to solution is reported counting a surrogate window as
    a gain only when its check passed."""
    import numpy as np
    import torch

    from paper_1102_3094_gb300 import lf

    rank, world, local = ranks()
    if rank != 0:
        return 0        # a single-GPU workload: the other ranks of a multi-GPU launch have no work
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    NY = NX = 256
    K = 50
    rng = np.random.default_rng(2011)
    nruns, nwin, warm = args.sur_runs, args.sur_windows, 400
    members = [dict(nx=NX, ny=NY, xi=float(10 ** rng.uniform(-4, 0)), tau=1.0, seed=500 + i) for i in range(nruns)]
    B = args.sur_batch
    with torch.cuda.stream(stream):
        t0 = time.time()
        # states[r, w] = (phi, T, ux, uy) of run r after warm + w K steps
        S = torch.empty((nruns, nwin + 1, 4, NY, NX), dtype=torch.float32, device=dev)
        chunk = 128                          # runs per ensemble
        for c0 in range(0, nruns, chunk):
            ms = members[c0:c0 + chunk]
            ens = lf.Ensemble(ms, stream=stream)
            ens.step(warm)
            for w in range(nwin + 1):
                if w:
                    ens.step(K)
                for r in range(len(ms)):
                    ctx = lf.lf_ens_run(ens.ens, r)
                    for ci, name in enumerate(("phi", "T", "ux", "uy")):
                        dst = S[c0 + r, w, ci]
                        lf.lf_fields(ctx, lf.FIELDS[name], dst.data_ptr(), dst.numel() * 4, True)
            ens.close()
        # a pair is usable while the run stays finite and at low Mach (|u| < 0.2):
        # runs with fast quenches diverge for the method itself at these parameters
        umax = S[:, :, 2:].abs().amax(dim=(2, 3, 4))
        ok_state = torch.isfinite(S).flatten(2).all(dim=2) & (umax < 0.2)
        ok_pair = ok_state[:, :-1] & ok_state[:, 1:]
        held = torch.zeros(nruns, dtype=torch.bool, device=dev)
        held[7::8] = True                    # whole trajectories held out
        tr_idx = torch.nonzero(ok_pair & ~held[:, None])
        ho_idx = torch.nonzero(ok_pair & held[:, None])
        n_dropped = int((~ok_pair).sum())
        torch.cuda.synchronize(dev)
        t_data = time.time() - t0
        X0 = S[tr_idx[:, 0], tr_idx[:, 1]]
        offset = X0.permute(1, 0, 2, 3).reshape(4, -1).mean(dim=1).cpu().numpy()
        dY = S[tr_idx[:, 0], tr_idx[:, 1] + 1] - X0
        scale = dY.permute(1, 0, 2, 3).reshape(4, -1).std(dim=1).clamp_min(1e-6).cpu().numpy()
        del X0, dY
        probe = lf.Lattice(nx=NX, ny=NY, precision="fp32", xi=1e-2, tau=1.0, seed=1, stream=stream, device=dev)

        def sk(phi):
            probe.set("phi", phi)
            d_ = probe.diag()
            return d_["k_peak"], d_["s_peak"]

        def sk_err(a, b):
            (ka, sa), (kb, sb) = sk(a), sk(b)
            return max(abs(ka / kb - 1), abs(sa / sb - 1))

        def train(pairs, iters, seed):
            """A network trained on the given (run, window) pairs; returns it,
            the training time and the loss trace."""
            sur = lf.Surrogate(NY, NX, B, scale=scale, offset=offset, seed=seed, stream=stream)
            sur.set_clip(1.0)
            gen = torch.Generator().manual_seed(seed)
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            losses = []
            ev[0].record(stream)
            for it in range(iters):
                lr = args.sur_lr * 0.5 * (1 + math.cos(math.pi * it / iters))
                sel = pairs[torch.randint(0, pairs.shape[0], (B,), generator=gen).to(dev)]
                x = S[sel[:, 0], sel[:, 1]].contiguous()
                y = S[sel[:, 0], sel[:, 1] + 1].contiguous()
                l = sur.train_step(x, y, lr)
                if it % 500 == 0 or it == iters - 1:
                    losses.append((it, l))
            ev[1].record(stream)
            torch.cuda.synchronize(dev)
            return sur, ev[0].elapsed_time(ev[1]) / 1e3, losses

        def heldout(sur, limit=None):
            """One-window accuracy on the held-out trajectories against keeping
            the state unchanged: phi relative L2 error and S(k) peak error."""
            idx = ho_idx if limit is None else ho_idx[:limit]
            acc = {"pairs": int(idx.shape[0]), "phi_l2": [], "sk": [], "persist_phi_l2": [], "persist_sk": []}
            for r_, w_ in idx.tolist():
                x = S[r_, w_:w_ + 1].contiguous()
                yt = S[r_, w_ + 1]
                yp = sur.predict(x)[0]
                acc["phi_l2"].append(float((yp[0] - yt[0]).norm() / yt[0].norm()))
                acc["persist_phi_l2"].append(float((x[0, 0] - yt[0]).norm() / yt[0].norm()))
                acc["sk"].append(sk_err(yp[0].contiguous(), yt[0].contiguous()))
                acc["persist_sk"].append(sk_err(x[0, 0].contiguous(), yt[0].contiguous()))
            out = {k: (float(np.mean(v)) if isinstance(v, list) else v) for k, v in acc.items()}
            out.update({k + "_median": float(np.median(v)) for k, v in acc.items() if isinstance(v, list)})
            out["within_2pct"] = float(np.mean([max(a, b) <= 0.02 for a, b in zip(acc["phi_l2"], acc["sk"])]))
            return out

        # learning curve: networks on random subsets of the training pairs, each
        # trained for as many steps as the main network (the last point)
        curve = []
        perm = torch.randperm(tr_idx.shape[0], generator=torch.Generator().manual_seed(3)).to(dev)
        for frac in [float(v) for v in args.sur_curve.split(",") if v and float(v) < 1.0]:
            n = max(B, int(frac * tr_idx.shape[0]))
            net, t_tr, _ = train(tr_idx[perm[:n]], args.sur_iters, 7)
            h = heldout(net, limit=args.sur_curve_pairs)
            curve.append({"train_pairs": n, "iters": args.sur_iters, "phi_l2": h["phi_l2"],
                          "phi_l2_median": h["phi_l2_median"], "sk": h["sk"], "within_2pct": h["within_2pct"]})
            net.close()
        sur, t_train, losses = train(tr_idx, args.sur_iters, 7)
        ho = heldout(sur)
        if curve:
            h = heldout(sur, limit=args.sur_curve_pairs)
            curve.append({"train_pairs": int(tr_idx.shape[0]), "iters": args.sur_iters, "phi_l2": h["phi_l2"],
                          "phi_l2_median": h["phi_l2_median"], "sk": h["sk"], "within_2pct": h["within_2pct"]})
        # evaluation run: fresh state, same physics, xi in the middle of the range
        ev_kw = dict(nx=NX, ny=NY, precision="fp32", xi=1e-2, tau=1.0, seed=9001, stream=stream, device=dev)
        plain = lf.Lattice(**ev_kw)
        hyb = lf.Lattice(**ev_kw)
        plain.step(warm)
        hyb.step(warm)
        torch.cuda.synchronize(dev)
        nsteps = args.sur_eval_windows * K
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record(stream)
        plain.step(nsteps)
        e[1].record(stream)
        torch.cuda.synchronize(dev)
        t_plain = e[0].elapsed_time(e[1]) / 1e3
        t1 = time.time()
        try:
            rep = sur.run(hyb, K, args.sur_eval_windows, args.sur_shadow_every, 0.02)
            run_error = None
        except lf.LFError as ex:      # e.g. the solver diverging after an accepted prediction
            rep, run_error = {}, str(ex)
        t_hyb = time.time() - t1
        dp, dh = plain.diag(), hyb.diag()
        pp, ph = plain.get("phi", "fp32"), hyb.get("phi", "fp32")
        l2 = float(np.linalg.norm(ph - pp) / np.linalg.norm(pp))
        probe.close()
    final_sk_err = max(abs(dh["k_peak"] / dp["k_peak"] - 1), abs(dh["s_peak"] / dp["s_peak"] - 1))
    # time to solution counting only windows known to be within the threshold:
    # plain windows, the predictions whose check passed, and for every other
    # surrogate window its prediction and a plain window
    tts = None
    if rep and rep.get("shadow_checks"):
        n_sur = (args.sur_eval_windows + 1) // 2
        n_plain = args.sur_eval_windows // 2
        t_pred = rep["t_surrogate_s"] / n_sur
        t_pw = rep["t_plain_s"] / max(1, n_plain + rep["rejected"])
        passed = rep["shadow_checks"] - rep["fallbacks"]
        unknown = n_sur - passed
        t_known = n_plain * t_pw + passed * t_pred + unknown * (t_pred + t_pw)
        tts = {"t_s": t_known, "speedup_vs_plain": t_plain / t_known, "windows_passed": passed,
               "windows_checked": rep["shadow_checks"], "t_prediction_s": t_pred, "t_plain_window_s": t_pw,
               "what": "plain windows + predictions whose shadow check passed + (prediction + plain window) for "
                       "every other surrogate window; shadow windows are the verification, not counted"}
    conv = conv_kernel_times(lf, torch, dev, stream)
    sites = NX * NY
    value = 1e-6 * sites * nsteps / tts["t_s"] if tts else 0.0
    line = {
        "metric": METRIC + " (surrogate-interleaved time to solution, counting only windows checked within 2 %)",
        "value": value, "unit": "MLUPS", "n_gpus": 1, "steps": nsteps, "warmup": warm,
        "ms_per_step": 1e3 * tts["t_s"] / nsteps if tts else None,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16/f32", "data": "synthetic",
        "config": {"workload": "sur256: 256x256 lamellar quench, 6-layer 64-channel residual CNN advancing "
                               f"(phi, T, ux, uy) by K={K} steps, trained on {int(tr_idx.shape[0])} pairs from "
                               f"{nruns - nruns // 8} solver trajectories of {warm + nwin * K} steps (xi log-uniform "
                               f"in [1e-4, 1]; the stated data volume is 2000 trajectories of 20k steps); "
                               f"{nruns // 8} whole trajectories held out; evaluation at xi = 1e-2",
                   "train_iters": args.sur_iters, "batch": B, "lr": args.sur_lr, "lr_schedule": "cosine",
                   "grad_clip": 1.0, "pairs_dropped": n_dropped,
                   "shadow_every": args.sur_shadow_every, "threshold": 0.02},
        "surrogate": {"t_data_s": t_data, "t_train_s": t_train, "losses": losses, "heldout": ho,
                      "learning_curve": curve, "report": rep, "run_error": run_error,
                      "t_plain_only_s": t_plain, "t_interleaved_wall_s": t_hyb,
                      "time_to_solution_known_good": tts, "conv_kernels": conv,
                      "final_phi_rel_l2_vs_plain": l2, "final_sk_peak_err_vs_plain": final_sk_err},
    }
    print(json.dumps(line), flush=True)
    for o in (plain, hyb, sur):
        o.close()
    return 0


def conv_kernel_times(lf, torch, dev, stream, B=8, NY=256, NX=256, reps=30):
    """Device time of single tensor-core convolutions and weight gradients (the surrogate's layer shapes at
    batch B): each launch after a 256 MB L2 flush and a sleep kernel, so that the stream
    is busy when the start event is recorded; CUDA events on the launching stream."""
    bf = torch.bfloat16
    g = torch.Generator(device=dev).manual_seed(7)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    err = torch.zeros(1, dtype=torch.int32, device=dev)
    out = {}
    cases = [("64->64 no residual", 64, 64, False, False), ("64->64 residual = input", 64, 64, True, False),
             ("64->64 residual = input, pre-activation out", 64, 64, True, True),
             ("16->64", 16, 64, False, False), ("64->16", 64, 16, False, False)]
    with torch.cuda.stream(stream):
        for name, cin, cout, res, zo in cases:
            inp = torch.randn((B, NY + 2, NX + 2, cin), device=dev, generator=g).to(bf)
            w = (0.1 * torch.randn((9, cout, cin), device=dev, generator=g)).to(bf).contiguous()
            bias = torch.randn(cout, device=dev, generator=g)
            o = torch.zeros((B, NY + 2, NX + 2, cout), dtype=bf, device=dev)
            z = torch.zeros_like(o) if zo else None
            x4 = torch.zeros((B, NY, NX, 4), device=dev) if cout == 16 else None
            y4 = torch.zeros_like(x4) if cout == 16 else None

            def call():
                lf.lf_sur_conv3x3(B, NY, NX, cin, cout, inp, w, bias, 1, inp if res else None, None, o, None, z,
                                  x4, y4, err, stream=stream)
            for _ in range(3):
                call()
            tot = 0.0
            for _ in range(reps):
                flush.zero_()
                torch.cuda._sleep(2_000_000)
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                call()
                e1.record(stream)
                e1.synchronize()
                tot += e0.elapsed_time(e1)
            us = 1e3 * tot / reps
            flop = 2 * 9 * cin * cout * B * NY * NX
            out[name] = {"us": us, "tflops": flop / us / 1e6}
        for cin, cout in ((64, 64), (16, 64), (64, 16)):   # weight gradients
            h = torch.randn((B, NY + 2, NX + 2, cin), device=dev, generator=g).to(bf)
            gr = torch.randn((B, NY + 2, NX + 2, cout), device=dev, generator=g).to(bf)
            dW = torch.zeros((9, cout, cin), device=dev)
            for _ in range(3):
                lf.lf_sur_conv3x3_wgrad(B, NY, NX, cin, cout, h, gr, dW, err, stream=stream)
            tot = 0.0
            for _ in range(reps):
                flush.zero_()
                torch.cuda._sleep(2_000_000)
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                lf.lf_sur_conv3x3_wgrad(B, NY, NX, cin, cout, h, gr, dW, err, stream=stream)
                e1.record(stream)
                e1.synchronize()
                tot += e0.elapsed_time(e1)
            us = 1e3 * tot / reps
            out[f"weight gradient {cin}->{cout}"] = {"us": us, "tflops": 2 * 9 * cin * cout * B * NY * NX / us / 1e6}
        torch.cuda.synchronize()
        if int(err.item()) != 0:
            raise RuntimeError("convolution kernel reported an error")
    out["shape"] = f"batch {B}, {NY}x{NX}, BF16 in, FP32 accumulate"
    return out


def run_ours(args):
    import numpy as np
    import torch

    from paper_1102_3094_gb300 import lf

    rank, world, local = ranks()
    dist = world > 1
    if dist:
        import torch.distributed as tdist
        tdist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    prec = args.precision
    if args.workload == "cube384":
        d, nx, ny, nz = 3, args.size3, args.size3, args.size3
        tau = 0.6
    else:
        d, nx, ny, nz = 2, args.size, args.size, 1
        tau = 1.0
    sim = lf.Lattice(d=d, nx=nx, ny=ny, nz=nz, precision=prec, xi=args.xi, tau=tau, seed=1 + rank, stream=stream,
                     device=dev)
    iso = args.stencil == "isotropic"
    if iso:
        sim.set_stencil("isotropic")        # 2D: the isotropic row march; 3D: the variant set (three passes by default)
    names = {lf.LF_VARIANT_MARCH: "march", lf.LF_VARIANT_TILE: "tile", lf.LF_VARIANT_MARCH2: "march2",
             lf.LF_VARIANT_SPLIT3: "split3"}
    variant = args.variant
    tuned = None
    if variant == "auto":
        # the library's autotuner picks the kernel variant and shape for this lattice
        v_, p_, ms_ = sim.tune(reps=5)
        variant, param = names[v_], p_
        tuned = {"variant": variant, "param": p_, "ms_per_step_in_tuning": ms_}
    else:
        param = args.tune
        sim.set_variant(variant, param)
    N = nx * ny * nz
    # The compact 3D step at these parameters goes non-finite after about 150
    # steps (the FP64 oracle too), so the 3D workload restores its initial quench
    # every `restore` steps, between the timed events: every timed step then
    # advances a finite state a few dozen steps after the quench.
    restore = args.restore_every if args.restore_every is not None else (100 if d == 3 else 0)
    state0 = None
    if restore > 0:
        state0 = {k: sim.get(k, device=True) for k in ("pop", "phi", "T")}
        torch.cuda.synchronize(dev)
    n_restores = 0

    def restore_state():
        for k_, v_ in state0.items():
            sim.set(k_, v_)                 # one unpack kernel per field, on the library stream
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    flush_rd = torch.ones(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev) if args.flush == "write+read" else None
    flush_sum = torch.zeros((), dtype=torch.float32, device=dev)

    def l2_flush(v):
        # evict the state from L2 by writing 256 MiB; with write+read, then
        # read another 256 MiB so the flush's dirty lines are written back
        # before the timed step instead of during it
        flush.fill_(v)
        if flush_rd is not None:
            torch.sum(flush_rd, dim=0, out=flush_sum)

    def barrier():
        torch.cuda.synchronize(dev)
        if dist:
            tdist.barrier()
        torch.cuda.synchronize(dev)

    # nvidia-smi samples the clocks from before the warm-up to the end of the
    # end-to-end leg; the line reports the timed window, or the whole run when
    # the timed window is too short to hold enough samples
    clk = Clocks(local)
    clk.__enter__()
    time.sleep(0.5)                          # let the sampler start
    t_run0 = time.time()
    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            l2_flush(1.0)
            sim.step(1)
    barrier()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    t_begin = time.time()
    with torch.cuda.stream(stream):
        for k in range(args.steps):
            if restore > 0 and k % restore == 0:
                restore_state()
                n_restores += 1
            l2_flush(float(k))
            starts[k].record(stream)
            sim.step(1)
            ends[k].record(stream)
    barrier()
    t_end = time.time()
    times_ms = [s.elapsed_time(e) for s, e in zip(starts, ends)]
    total_s = max_over_ranks(sum(times_ms) / 1e3, dev)
    dg = sim.diag()
    value = job_rate(N, args.steps, world, total_s)
    ms = 1e3 * total_s / args.steps
    bps = BYTES_PER_SITE[(prec, d)]
    peak, peak_kind = peaks()
    passes = 3 if (d == 3 and variant == "split3") else 1
    extra = lf.lf_nsub(args.xi, d) - 1 if args.xi not in (0.0, math.inf) else 0
    if d == 2 and prec == "fp32":
        extra = (extra + 3) // 4            # up to four temperature sub-steps per launch
    launches_per_step = passes + extra
    # the three-pass 3D step is measured as a whole: algorithmic bytes of the
    # step over the step time
    per_kernel = 1 if passes > 1 else launches_per_step
    kernel_ms = statistics.mean(times_ms) / per_kernel
    achieved = bps * N / (kernel_ms * 1e-3) / 1e9
    if d == 3:
        kname = ("k_force3d+k_lb3d+k_phi3d" if variant == "split3" else "k_march3d") + ("_iso" if iso else "")
    elif iso:
        kname = {"march": "k_march2d_iso", "march2": "k_march2d_iso_x2", "tile": "k_step2d_iso"}[variant]
    else:
        kname = {"march": "k_march2d", "march2": "k_march2d_x2", "tile": "k_step2d"}[variant]
    if kname.startswith("k_march2d") and kname.endswith("x2") and prec == "fp64":
        kname = kname[:-3]                  # the packed kernels are FP32 only
    traffic, traffic_shape = traffic_for(f"{kname}_{prec}_{nx}", param)
    roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "traffic": traffic, "traffic_shape": traffic_shape, "peak_kind": peak_kind,
            "algorithmic_bytes_per_site": bps,
            "kernel": kname + (f" ({passes} passes; bytes and time of the whole step)" if passes > 1
                               else " (fused phi-chain + LB + FD)"),
            "kernel_ms_mean": kernel_ms, "kernel_ms_median": statistics.median(times_ms) / per_kernel}

    # ---- the three passes of the 3D step, timed one by one ------------------
    # (CUDA events at the pass boundaries, recorded by the library on its
    # stream; a short sequence after the timed steps, L2 flushed before each
    # step as above)
    def pass_breakdown(sim_, iso_, param_, restore_fn):
        sel = (param_ >> 16) & 15
        if iso_:
            packed = prec == "fp32" and (sel == 4 or (param_ & 0xFFFFF) == 0)
            force = "k_force3d_iso_x2" if packed else "k_force3d_iso"
            phi_k = "k_phi3d_iso_q" if prec == "fp32" else "k_phi3d_isoz"
        else:
            force = "k_force3d_x2" if (sel == 0 and prec == "fp32") else "k_force3d"
            phi_k = "k_phi3d_q" if prec == "fp32" else "k_phi3d"
        esz = 4 if prec == "fp32" else 8
        per_site = [6 * esz, 44 * esz, 8 * esz]      # A: phi, T in, mu, F out; B: f in/out, F, u; C: phi, u, mu, T in, phi, T out
        acc, cnt = [0.0, 0.0, 0.0], 0
        sim_.set_pass_timing(True)
        with torch.cuda.stream(stream):
            if restore_fn:
                restore_fn()
            for k in range(min(args.steps, 30)):
                l2_flush(float(k))
                sim_.step(1)
                ms_ = sim_.pass_times()
                if len(ms_) == 3:
                    acc = [a + b for a, b in zip(acc, ms_)]
                    cnt += 1
        sim_.set_pass_timing(False)
        if cnt == 0:
            return None
        out = []
        for name, b, t in zip((force, "k_lb3d", phi_k), per_site, acc):
            ms_ = t / cnt
            gbs = b * N / (ms_ * 1e-3) / 1e9
            out.append({"kernel": name, "ms": ms_, "algorithmic_bytes_per_site": b, "achieved_gbs": gbs,
                        "frac": gbs / peak})
        dom = max(out, key=lambda x: x["ms"])
        return {"steps": cnt, "passes": out,
                "dominant": {"kernel": dom["kernel"], "achieved_gbs": dom["achieved_gbs"], "frac": dom["frac"],
                             "share_of_step": dom["ms"] / sum(x["ms"] for x in out)}}

    if d == 3 and variant == "split3":
        roof["per_pass"] = pass_breakdown(sim, iso, param, restore_state if restore > 0 else None)

    # ---- end to end through the C ABI with host buffers ---------------------
    e2e = None
    if args.e2e_steps > 0:
        tdt = torch.float32 if prec == "fp32" else torch.float64
        shp = sim.shape
        pop_h = torch.empty((sim.Q,) + shp, dtype=tdt, pin_memory=True)
        phi_h = torch.empty(shp, dtype=tdt, pin_memory=True)
        T_h = torch.empty(shp, dtype=tdt, pin_memory=True)
        out_h = torch.empty(shp, dtype=tdt, pin_memory=True)
        es = pop_h.element_size()
        lf.lf_fields(sim.ctx, lf.FIELDS["pop"], pop_h.data_ptr(), pop_h.numel() * es, False)
        lf.lf_fields(sim.ctx, lf.FIELDS["phi"], phi_h.data_ptr(), phi_h.numel() * es, False)
        lf.lf_fields(sim.ctx, lf.FIELDS["T"], T_h.data_ptr(), T_h.numel() * es, False)
        barrier()
        t0 = time.perf_counter()
        for _ in range(args.e2e_steps):
            lf.lf_fields_set(sim.ctx, lf.FIELDS["pop"], pop_h.data_ptr(), pop_h.numel() * es, False)
            lf.lf_fields_set(sim.ctx, lf.FIELDS["phi"], phi_h.data_ptr(), phi_h.numel() * es, False)
            lf.lf_fields_set(sim.ctx, lf.FIELDS["T"], T_h.data_ptr(), T_h.numel() * es, False)
            lf.lf_step(sim.ctx, 1)
            lf.lf_fields(sim.ctx, lf.FIELDS["phi"], out_h.data_ptr(), out_h.numel() * es, False)
        el = max_over_ranks(time.perf_counter() - t0, dev)
        torch.cuda.synchronize(dev)
        e2e = {"value": job_rate(N, args.e2e_steps, world, el), "unit": "MLUPS",
               "h2d_bytes_per_step": (sim.Q + 2) * N * es, "d2h_bytes_per_step": N * es,
               "steps": args.e2e_steps,
               "what": "per step: lf_fields_set of f, phi, T from pinned host, lf_step(1), lf_fields of phi to "
                       "pinned host"}

    t_run1 = time.time()
    clk.__exit__(None, None, None)
    clocks = clk.summary_over((t_begin, t_end + 0.1), (t_run0, t_run1 + 0.1))
    cpu = None
    if rank == 0 and args.cpu_seconds > 0:
        if d == 3:
            rate, steps, el, cores = oracle_rate(64, 64, args.xi, seconds=args.cpu_seconds, d=3, nz=64, tau=tau,
                                                 stencil=int(iso), restore=restore)
            smp = "64x64x64" + (f", initial quench restored every {restore} steps" if restore > 0 else "")
        else:
            rate, steps, el, cores = oracle_rate(256, 256, args.xi, seconds=args.cpu_seconds, stencil=int(iso))
            smp = "256x256"
        cpu = {"value": rate, "unit": "MLUPS", "cores": cores, "kind": "oracle",
               "sample": f"{steps} FP64 oracle steps of a {smp} lattice with the workload's physics "
                         f"({el:.1f} s)"}
    # The compact 3D step at tau = 0.6 goes non-finite after about 150 steps (the
    # oracle too), hence the restores above.  The configuration that runs to its
    # stated 20k steps at this size is tau = 3 with the isotropic stencils: time
    # it too, without restores, beside the main line.
    stable = None
    if d == 3 and args.stable_run and not iso:
        sim.close()
        sim = lf.Lattice(d=3, nx=nx, ny=ny, nz=nz, precision=prec, xi=args.xi, tau=3.0, seed=1 + rank,
                         stream=stream, device=dev, stencil="isotropic")
        v_, p_, _ = sim.tune(reps=3)
        with torch.cuda.stream(stream):
            for _ in range(args.warmup):
                sim.step(1)
        barrier()
        ts = []
        with torch.cuda.stream(stream):
            for k in range(args.steps):
                starts[k].record(stream)
                sim.step(1)
                ends[k].record(stream)
        barrier()
        ts = [a.elapsed_time(b) for a, b in zip(starts, ends)]
        tot = max_over_ranks(sum(ts) / 1e3, dev)
        ach = bps * N * args.steps / tot / 1e9
        traffic, traffic_shape = traffic_for(f"k_force3d+k_lb3d+k_phi3d_iso_{prec}_{nx}", p_) if v_ == 3 else (None, None)
        stable = {"what": "tau = 3, isotropic 19-point stencils (runs the 20k steps finite); no restores",
                  "value": job_rate(N, args.steps, world, tot), "unit": "MLUPS",
                  "ms_per_step": 1e3 * tot / args.steps, "frac": ach / peak, "achieved_gbs": ach,
                  "traffic": traffic, "traffic_shape": traffic_shape,
                  "per_pass": pass_breakdown(sim, True, p_, None) if v_ == 3 else None,
                  "kernel_shape": {"variant": names[v_], "param": p_}, "diag_after": {"rc": sim.diag()["rc"]}}
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32" if prec == "fp32" else "f64", "data": "synthetic",
            "config": {"workload": (f"prec1024: 2D D2Q9 lamellar quench between cold walls, {nx}x{ny}, "
                                    if d == 2 else
                                    f"cube384: 3D D3Q19 lamellar quench between cold walls (z), {nx}x{ny}x{nz}, ")
                                   + f"{prec.upper()} state (deviation populations), xi={args.xi}, tau={tau}"
                                   + ((", isotropic 9-point stencils" if d == 2 else ", isotropic 19-point stencils")
                                      if iso else ""),
                       "sites": N, "l2": ("flushed before every timed step (256 MiB write"
                                          + (", then a 256 MiB read so no dirty flush lines are written back "
                                             "inside the timed step" if args.flush == "write+read" else "")
                                          + "); each step timed alone with CUDA events on the library stream"),
                       "parallelism": f"replicas x{world} (one independent lattice per GPU)",
                       "kernel_shape": tuned if tuned else {"variant": variant, "param": param, "from": "--variant"}},
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": args.steps * launches_per_step + 3 * n_restores,
            "restores": ({"every": restore, "count": n_restores, "launches": 3 * n_restores,
                          "what": "lf_fields_set of f, phi, T from a device copy of the initial state, "
                                  "between the timed events"} if restore > 0 else None),
            "clocks": clocks,
            "diag_after": {"mass": dg["mass"], "mach": dg["mach"], "rc": dg["rc"]},
            "stable_configuration": stable,
        }
        print(json.dumps(line), flush=True)
    sim.close()
    if dist:
        tdist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=["prec1024", "cube384", "ens96", "sur256"], default="cube384")
    ap.add_argument("--ens-prune-every", type=int, default=500,
                    help="ens96: retire non-finite runs every this many steps (0 = never)")
    ap.add_argument("--sur-runs", type=int, default=512, help="solver trajectories (every 8th held out)")
    ap.add_argument("--sur-windows", type=int, default=40, help="K-step windows per trajectory after the warm-up")
    ap.add_argument("--sur-iters", type=int, default=40000)
    ap.add_argument("--sur-batch", type=int, default=16)
    ap.add_argument("--sur-lr", type=float, default=1e-3)
    ap.add_argument("--sur-curve", default="", help="comma-separated fractions below 1 of the training pairs "
                    "for a learning curve (one network each, as many steps as the main network)")
    ap.add_argument("--sur-curve-pairs", type=int, default=512, help="held-out pairs per learning-curve point")
    ap.add_argument("--sur-eval-windows", type=int, default=40)
    ap.add_argument("--sur-shadow-every", type=int, default=1)
    ap.add_argument("--size", type=int, default=1024, help="2D lattice side (prec1024)")
    ap.add_argument("--size3", type=int, default=384, help="3D lattice side (cube384)")
    ap.add_argument("--precision", choices=["fp32", "fp64"], default="fp32")
    ap.add_argument("--xi", type=float, default=1e-3)
    ap.add_argument("--e2e-steps", type=int, default=20)
    ap.add_argument("--restore-every", type=int, default=None,
                    help="restore the initial state every R timed steps, outside the timed events "
                         "(default: 100 in 3D, never in 2D; 0 = never)")
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--stable-run", type=int, default=1,
                    help="3D compact workload: also time tau = 3 with the isotropic stencils (1) or not (0)")
    ap.add_argument("--variant", choices=["auto", "march", "tile", "march2", "split3"], default="auto",
                    help="step kernel variant (all compute the same step); auto = the choice of the library's "
                         "autotuner (lf_tune) for this lattice")
    ap.add_argument("--flush", choices=["write", "write+read"], default="write+read",
                    help="L2 eviction between timed steps (2D and 3D single-lattice workloads)")
    ap.add_argument("--tune", type=int, default=0, help="param of an explicit --variant (see lf_set_kernel_variant)")
    ap.add_argument("--stencil", choices=["compact", "isotropic"], default="compact",
                    help="finite-difference stencils (isotropic: the 2D tile kernel; in 3D the chosen variant)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "ens96":
        return run_ensemble(args)
    if args.workload == "sur256":
        return run_surrogate(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
