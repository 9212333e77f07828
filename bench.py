"""Benchmark of the LBM-GNN hot path on GB300.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

One JSON line on stdout, on rank 0: the headline, short enough to be read whole
from the end of a log; the full record of the run (the GNN workloads, training,
tables, sweeps) goes to stderr and to the --log file.  A "step" is one lattice update of the
Taylor-Green workload 4096 x 4096 (periodic, FP32 SoA populations, u0 = 0.05,
k = 2 pi / 4096), timed with CUDA events on the stream the kernels run on;
`value` is million lattice-node updates per second (MLUPS) over all ranks.
Each rank advances its own lattice (weak scaling, no collective on the data
path).  The GNN-LBM step on the 1024 x 1024 TGV (Re = 1000) is measured in
the same run and reported beside it under "gnn" (a summary in the headline).

`--impl reference` times the FP64 CPU oracle (the slow, obviously-correct
restatement of the method) on the host cores, one bounded sub-lattice per
step, and prints the same line with "impl": "reference".
"""
import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "MLUPS, plain BGK vs GNN-LBM on 1 GB300, at stated TGV velocity L2 error"
from paper_2504_14494_gb300 import workloads as W  # noqa: E402  (sizes, taus, seeds)

N_SIDE = W.TGV_4096.n
U0 = W.TGV_4096.u0
TAU = W.TGV_4096.tau
TAU_SWEEP = W.TGV_4096.tau_sweep
BYTES_PER_NODE = 72  # 9 FP32 loads + 9 FP32 stores
RUNS = 5  # the timed steps are split into this many consecutive runs; median run reported

# DRAM bytes per launch from one ncu capture of the kernel, keyed by the
# SHA-256 of its source file at capture time; ignored once the source changed.
NCU_TRAFFIC = {
    # ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum
    #     --clock-control none -k regex:bgk_step_x4 -s 3 -c 1
    #     python bench.py --only bgk --steps 10 --warmup 3      (4096 x 4096, one launch)
    "bgk_step_x4": {"bytes_per_launch": 604035328 + 547279360,
                    "src_sha": "c361951bbca67452362ae7d5185e3edf6334a82adc138553e6b85d5e3f24f94f"},
    # ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum
    #     --clock-control none -k regex:"gnn_(step_first|round)_kernel" -s 3 -c 3
    #     python bench.py --only gnn --steps 20 --warmup 3   (one GNN-LBM step, 1024 x 1024:
    #     the fused encoder, 2 rounds; key files gnn_fwd.cu and gnn_mlp.cu)
    "lbm_step_gnn": {"bytes_per_launch": (38159104 + 208859904) + (269575680 + 213989632)
                     + (306580992 + 25687808), "nodes": 1024 * 1024,
                     "file": ["gnn_fwd.cu", "gnn_mlp.cu"],
                     "src_sha": ["86e1c5868386e4054fb61fdaa400a213954ffb464747652614837dbfe7c89f15",
                                 "41f9d20607b65813e446e6c6f6830da66e64035e4d5e69bcb07ada862437133c"]},
    # ncu --metrics dram__bytes_read.sum,dram__bytes_write.sum,gpu__time_duration.sum
    #     --clock-control none -k regex:gnn_mlp_step -s 3 -c 1
    #     python bench.py --only mlp --side 4096 --steps 10 --warmup 3   (one fused step)
    "gnn_mlp_step_kernel": {"bytes_per_launch": 604060416 + 554683904, "nodes": 4096 * 4096,
                            "file": "gnn_mlp.cu",
                            "src_sha": "41f9d20607b65813e446e6c6f6830da66e64035e4d5e69bcb07ada862437133c"},
}


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            p = json.load(fh)
        return float(p["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


def _finite(obj):
    """Non-finite floats (a diverged rollout's error) become null so that the
    line stays strict JSON."""
    if isinstance(obj, float):
        return obj if np.isfinite(obj) else None
    if isinstance(obj, dict):
        return {k: _finite(v) for k, v in obj.items()}
    if isinstance(obj, (list, tuple)):
        return [_finite(v) for v in obj]
    return obj


def _src_sha(name):
    """SHA-256 of a csrc file, or the list of them for a list of names."""
    if isinstance(name, (list, tuple)):
        return [_src_sha(n) for n in name]
    with open(os.path.join(ROOT, "paper_2504_14494_gb300", "csrc", name), "rb") as fh:
        return hashlib.sha256(fh.read()).hexdigest()


def _re(tau, n=N_SIDE, u0=U0):
    return u0 * n / ((tau - 0.5) / 3.0)


def headline(out):
    """The stdout line of a full record: every field but the long ones, with the
    GNN workloads' rates in the place of their records."""
    h = {k: v for k, v in out.items() if k not in ("tau_sweep", "tgv64")}
    if "timing" in h:
        h["timing"] = {k: v for k, v in h["timing"].items() if not isinstance(v, (list, tuple))}
    if "cpu_baseline" in h:
        h["cpu_baseline"] = {k: v for k, v in h["cpu_baseline"].items() if not isinstance(v, dict)}
    if "gnn" in h:
        g = out["gnn"]
        pick = {"xavier": ("workload", "mlups_gnn", "ms_per_step_gnn"),
                "training": ("workload", "ms_per_fused_train_step"),
                "mlp_fused": ("workload", "mlups_gnn_mlp", "ms_per_step_gnn_mlp"),
                "batch": ("workload", "mlups_total", "ms_per_step")}
        h["gnn"] = {name: {k: g[name].get(k) for k in keys} for name, keys in pick.items() if name in g}
    return h


class ClockSampler:
    """Samples SM clock and throttle reasons with nvidia-smi during a region."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            time.sleep(0.3)
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            time.sleep(0.15)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.t.join(timeout=2)

    def summary(self):
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                smax = float(parts[1])
            except ValueError:
                continue
            for nm, v in zip(names, parts[3:7]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------------
def run_ours(args, rank, world, local_rank):
    import torch
    from paper_2504_14494_gb300 import build, lib as L, parallel
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    build.build()
    L.load()
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    if args.only == "gnn":
        res = gnn_bench(args, L, dev, torch.cuda.current_stream(), side=args.side, only=True)
        print(json.dumps(_finite({"case": f"gnn {args.side}x{args.side}", **res})))
        return None
    if args.only == "mlp":
        res = mlp_bench(args, L, dev, torch.cuda.current_stream(), side=args.side)
        print(json.dumps(_finite({"case": f"gnn_mlp {args.side}x{args.side}", **res})))
        return None
    if args.only == "batch":  # the 512-lattice serving batch, untrained conserving network
        from paper_2504_14494_gb300 import inputs
        theta = inputs.xavier_params(W.TGV_GNN_1024.weight_seed, variant=2)
        res = batch_bench(args, L, dev, torch.cuda.current_stream(), theta)
        print(json.dumps(_finite({"case": res["workload"], **res})))
        return None
    if args.only == "channel":  # Poiseuille study, untrained conserving fixed-tau network
        from paper_2504_14494_gb300 import inputs
        res = channel_bench(L, dev, {"xavier_v6": inputs.xavier_params(0, variant=6, s_df=1e-4)})
        print(json.dumps(_finite({"case": res["workload"], **res})))
        return None
    if args.only == "train":
        from paper_2504_14494_gb300 import inputs
        from paper_2504_14494_gb300.train import Trainer
        tr = Trainer(dev, theta=inputs.xavier_params(0), lr=1e-4, wd=0.0, seed=1, n=args.side,
                     batch=64, episode=64)
        f_in, f_tg, taus = tr.data.next()
        for i in range(args.warmup):
            L.gnn_train_step(f_in, f_tg, tr.data.coarse, 1.0, taus, tr.params, tr.packed, tr.m,
                             tr.v, 1 + i, 1e-4, 0.0, tr.loss, None, tr.ws)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for i in range(args.steps):
            L.gnn_train_step(f_in, f_tg, tr.data.coarse, 1.0, taus, tr.params, tr.packed, tr.m,
                             tr.v, 100 + i, 1e-4, 0.0, tr.loss, None, tr.ws)
        e1.record()
        torch.cuda.synchronize()
        print(json.dumps({"case": f"train 64x{args.side}^2",
                          "ms_per_step": e0.elapsed_time(e1) / args.steps,
                          "status": L.lbm_get_status()}))
        return None
    n = args.side
    nodes = n * n
    s = L.shape(n, n)
    k = 2 * np.pi / n
    stream = torch.cuda.current_stream()
    fa = torch.empty(9 * nodes, dtype=torch.float32, device=dev)
    fb = torch.empty_like(fa)
    L.lbm_init_tgv(fa, s, 1.0, U0, k, k, False)

    def steps(count, tau, bufs):
        for _ in range(count):
            L.lbm_step_bgk(bufs[0], bufs[1], None, s, tau, nsteps=1)
            bufs.reverse()

    bufs = [fa, fb]
    steps(args.warmup, TAU, bufs)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    # The K timed steps run back to back as R consecutive runs of about K/R
    # steps, an event on the launching stream between runs; the headline
    # takes the median run (per-step time), the whole region is reported too.
    runs = chunk_sizes(args.steps, RUNS)
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(len(runs) + 1)]
    with ClockSampler(local_rank) as clk:
        evs[0].record(stream)
        for i, c in enumerate(runs):
            steps(c, TAU, bufs)
            evs[i + 1].record(stream)
        torch.cuda.synchronize()
    ms_region = evs[0].elapsed_time(evs[-1])
    per_step = [evs[i].elapsed_time(evs[i + 1]) / c for i, c in enumerate(runs)]
    ms = statistics.median(per_step) * args.steps
    if dist:
        dist.barrier()
    # node updates summed over ranks / the slowest rank's (median-run) time
    _, t_max, rate = parallel.aggregate_throughput(nodes * args.steps, ms, device=dev)
    done_steps = args.warmup + args.steps
    assert L.lbm_get_status() == 0
    if args.only == "bgk":
        if rank == 0:
            print(json.dumps({"case": f"bgk {n}x{n}", "ms_per_step": ms / args.steps,
                              "mlups": nodes * args.steps / (ms / 1e3) / 1e6}))
        return None

    # TGV velocity L2 error of the state after done_steps steps (closed form).
    l2 = tgv_l2(L, bufs[0], s, n, U0, TAU, done_steps, dev)

    # tau sweep (same lattice, fresh TGV state each)
    sweep = []
    for tau in TAU_SWEEP:
        L.lbm_init_tgv(fa, s, 1.0, U0, k, k, False)
        b2 = [fa, fb]
        steps(max(3, args.warmup), tau, b2)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        kk = max(10, min(args.steps, 2000))
        e0.record(stream)
        steps(kk, tau, b2)
        e1.record(stream)
        torch.cuda.synchronize()
        sweep.append({"tau": tau, "re": round(_re(tau), 1),
                      "mlups": round(nodes * kk / (e0.elapsed_time(e1) / 1e3) / 1e6, 1)})

    # end to end through the C ABI with host buffers (lbm_step_bgk_host): per
    # step the state is copied from pinned host memory (in row blocks that
    # overlap the step), stepped, and the stepped state and its FP64 totals
    # are copied back to pinned host memory.  The output of one step is the
    # input of the next (host ping-pong), as a host-resident simulation runs.
    host = [torch.empty(9 * nodes, dtype=torch.float32, pin_memory=True) for _ in range(2)]
    L.lbm_init_tgv(fa, s, 1.0, U0, k, k, False)
    host[0].copy_(fa)
    host_tot = torch.empty(5, dtype=torch.float64, pin_memory=True)
    hws = torch.empty(L.lbm_host_workspace_bytes(s), dtype=torch.uint8, device=dev)
    ke = max(3, min(args.steps, 30))
    for _ in range(3):
        L.lbm_step_bgk_host(host[0], host[1], s, TAU, None, 1, host_tot, hws)
        host.reverse()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(ke):
        L.lbm_step_bgk_host(host[0], host[1], s, TAU, None, 1, host_tot, hws)
        host.reverse()
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = e0.elapsed_time(e1) / ke
    assert L.lbm_get_status() == 0
    e2e_l2 = tgv_l2(L, host[0].to(dev), s, n, U0, TAU, 3 + ke, dev)

    thetas, train_info = train_bench(args, L, dev, stream)
    ch_thetas, ch_info = channel_train(L, dev)
    names = {0: "message passing (Eq. 3 as printed)", 2: "message passing, conserving correction",
             3: "Fig. 2 MLP-only, conserving correction",
             4: "message passing, tau_adj fixed at 1 (64 x 256^2 recipe)"}
    trained = {}
    for v, th in thetas.items():
        if not isinstance(v, int):  # the weighted and the high-Re networks: below
            continue
        r = gnn_bench(args, L, dev, stream, theta=th, label=f"trained in this run: {names[v]}")
        r["rollout_1000_steps"] = rollout_error(L, dev, th)
        trained[str(v)] = r
    gnn = {"trained": trained,
           "xavier": gnn_bench(args, L, dev, stream, label="xavier-uniform seed 0, untrained"),
           "training": train_info,
           "held_out_rollout": held_out_rollout(L, dev, thetas[4], names[4]),
           "rollout_relative_seed2": rollout_error(L, dev, thetas["relative"][2]),
           "held_out_rollout_weighted": {
               f"seed{sd}": held_out_rollout(L, dev, th, "Eq. 3 as printed, trained with "
                                             "per-instance relative weights, seed %d" % sd)
               for sd, th in thetas["relative"].items()},
           "batch": batch_bench(args, L, dev, stream, thetas[2]),
           "tgv_tables": tgv_tables(L, dev, {"conserving_v2": thetas[2], "mlp_v3": thetas[3],
                                             "tau_fixed_v4": thetas[4],
                                             "eq3_relative_seed2": thetas["relative"][2]}),
           "stability": {**{str(v): stability_bench(L, dev, thetas[v]) for v in (0, 2, 4)},
                         "2_high_re": stability_bench(L, dev, thetas["2_high_re"])},
           "channel_training": ch_info,
           "poiseuille": channel_bench(L, dev, {
               "tau_fixed_v4": thetas[4], "conserving_v2": thetas[2],
               "eq3_relative_seed2": thetas["relative"][2], **ch_thetas}),
           "mlp_fused": mlp_bench(args, L, dev, stream, theta=thetas[3])}

    if rank != 0:
        return None
    peak, peak_kind = _peaks()
    ms_step = t_max / args.steps
    achieved = BYTES_PER_NODE * nodes / (ms / args.steps / 1e3) / 1e9
    sha = _src_sha("bgk.cu")
    tr = NCU_TRAFFIC.get("bgk_step_x4")
    traffic = tr["bytes_per_launch"] if tr and tr.get("src_sha") == sha else None
    out = {
        "metric": METRIC,
        "value": round(rate / 1e6, 1),
        "unit": "MLUPS",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(ms_step, 5),
        "timing": {"runs": len(runs), "steps_per_run": runs,
                   "median_run_ms_per_step": round(statistics.median(per_step), 5),
                   "run_ms_per_step": [round(v, 5) for v in per_step],
                   "whole_region_ms_per_step": round(ms_region / args.steps, 5),
                   "headline": "median run"},
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": "tgv_bgk_4096x4096", "nx": n, "ny": n, "tau": TAU,
                   "re": round(_re(TAU), 1), "u0": U0, "k": "2*pi/4096",
                   "l2_flush": "inputs larger than L2 (604 MB per population buffer)",
                   "parallelism": f"replicas x{world}"},
        "tgv_l2_error": l2, "tgv_steps_run": done_steps,
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak,
                     "unit": "GB/s", "frac": round(achieved / peak, 4), "traffic": traffic,
                     "peak_kind": peak_kind, "kernel": "bgk_step_x4",
                     "algorithmic_bytes_per_launch": BYTES_PER_NODE * nodes},
        "tau_sweep": sweep,
        "tgv64": small_tgv_bench(L, dev),
        "e2e": {"value": round(nodes / (e2e_ms / 1e3) / 1e6, 1), "unit": "MLUPS",
                "h2d_bytes_per_step": 9 * nodes * 4, "d2h_bytes_per_step": 9 * nodes * 4 + 5 * 8,
                "call": "lbm_step_bgk_host: pinned host state in, stepped state and FP64 "
                        "totals out, every step",
                "velocity_l2_error": e2e_l2},
        "clocks": clk.summary(),
        "gpu_launches": args.steps,
        "gnn": gnn,
    }
    if not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline()
        out["cpu_baseline"]["all_cores"] = cpu_baseline_all_cores()
        out["cpu_baseline"]["gnn"] = cpu_baseline_gnn()
    return out


def chunk_sizes(k, r):
    """k steps as min(r, k) consecutive runs of near-equal length."""
    r = max(1, min(r, k))
    return [k // r + (1 if i < k % r else 0) for i in range(r)]


def _gnn_oracle_worker(args):
    """One host core: the oracle GNN-LBM step (brute-force 130-wide edge MLP,
    numpy FP64) on an n x n TGV at Re = 1000, `count` steps."""
    n, count = args
    from oracle import gnn, lbm
    from paper_2504_14494_gb300 import inputs
    theta = inputs.xavier_params(W.TGV_GNN_1024.weight_seed)
    k = 2 * np.pi / n
    tau = 0.5 + 3.0 * U0 * n / W.TGV_GNN_1024.re
    f = lbm.tgv_init(n, n, 1.0, U0, k, k)
    t0 = time.perf_counter()
    for _ in range(count):
        f = gnn.gnn_step(f, theta, tau)
    return time.perf_counter() - t0


def cpu_baseline_gnn(n=256, count=3):
    """The FP64 oracle's GNN-LBM step, as it stands, on one host core (BLAS
    limited to one thread in a spawned process): n x n TGV, `count` steps."""
    import multiprocessing as mp
    saved = {v: os.environ.get(v) for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS",
                                             "MKL_NUM_THREADS")}
    for v in saved:
        os.environ[v] = "1"
    try:
        with mp.get_context("spawn").Pool(1) as pool:
            dt = pool.map(_gnn_oracle_worker, [(n, count)])[0]
    finally:
        for v, old in saved.items():
            if old is None:
                os.environ.pop(v, None)
            else:
                os.environ[v] = old
    return {"value": round(n * n * count / dt / 1e6, 4), "unit": "MLUPS", "cores": 1,
            "kind": "oracle",
            "sample": f"oracle.gnn.gnn_step (numpy FP64, brute-force 130-wide edge MLP) on a "
                      f"{n}x{n} TGV at Re = 1000, {count} steps, {dt:.1f} s"}


def small_tgv_bench(L, dev, n=W.TGV_64.n, tau=W.TGV_64.tau, u0=W.TGV_64.u0,
                    steps=W.TGV_64.steps):
    """The 64^2 Taylor-Green workload: 1000 BGK steps (one call), the
    velocity L2 error against the closed form, the kinetic-energy error
    against E0 exp(-4 nu k^2 t), and the mass / momentum drift of the FP64
    totals; its MLUPS are latency-bound (147 KB per buffer) and not a
    bandwidth figure."""
    import torch
    s = L.shape(n, n)
    k = 2 * np.pi / n
    f0 = torch.empty(9 * n * n, device=dev)
    L.lbm_init_tgv(f0, s, 1.0, u0, k, k, False)
    t0 = torch.zeros(5, dtype=torch.float64, device=dev)
    L.lbm_moments(f0, s, None, None, None, t0)
    f1, tmp = torch.empty_like(f0), torch.empty_like(f0)
    tot = torch.zeros(5, dtype=torch.float64, device=dev)
    L.lbm_step_bgk(f0, f1, tmp, s, tau, nsteps=10)  # warm-up
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    L.lbm_step_bgk(f0, f1, tmp, s, tau, nsteps=steps, totals=tot)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    a, b = t0.cpu().numpy(), tot.cpu().numpy()
    nu = (tau - 0.5) / 3.0
    e_ref = a[3] * np.exp(-4.0 * nu * k * k * steps)
    return {"workload": f"tgv_bgk_{n}x{n}", "tau": tau, "u0": u0, "steps": steps,
            "mlups": round(n * n * steps / (ms / 1e3) / 1e6, 1),
            "velocity_l2_error": tgv_l2(L, f1, s, n, u0, tau, steps, dev),
            "energy_rel_error": float(abs(b[3] - e_ref) / e_ref),
            "mass_rel_drift": float(abs(b[0] - a[0]) / a[0]),
            "momentum_drift": [float(b[1] - a[1]), float(b[2] - a[2])],
            "status": L.lbm_get_status()}


def tgv_l2(L, f, s, n, u0, tau, t, dev):
    """Relative L2 velocity error of state f (n x n) against the closed-form
    TGV decay u0 exp(-2 nu k^2 t), k = 2 pi / n (evaluated with torch)."""
    import torch
    k = 2 * np.pi / n
    rho = torch.empty(n * n, device=dev)
    ux = torch.empty(n * n, device=dev)
    uy = torch.empty(n * n, device=dev)
    L.lbm_moments(f, s, rho, ux, uy)
    xs = torch.arange(n, device=dev, dtype=torch.float64)
    decay = float(np.exp(-((tau - 0.5) / 3.0) * 2 * k * k * t))
    uxa = (u0 * decay * torch.cos(k * xs)[None, :] * torch.sin(k * xs)[:, None]).reshape(-1)
    uya = (-u0 * decay * torch.sin(k * xs)[None, :] * torch.cos(k * xs)[:, None]).reshape(-1)
    return float(torch.sqrt(((ux.double() - uxa) ** 2 + (uy.double() - uya) ** 2).sum()
                            / (uxa ** 2 + uya ** 2).sum()).item())


GNN_SIDE = W.TGV_GNN_1024.n
GNN_RE = W.TGV_GNN_1024.re
# Elementwise roofline of the message passing: each pair of edge-feature
# GELUs is 7 packed-FP16 operations (z = A + c + B: 2, u: 3, accumulate
# z + z tanh u: 2) and one tanh.approx.f16x2.  Measured on GB300
# (paper_2504_14494_gb300/microbench/fp16_rate.cu): HFMA2 issues at 2.07 warp
# instructions per clock per SM, tanh.approx.f16x2 at 0.25 (the MUFU unit
# binds: 16 edge-feature GELUs per clock per SM), and the whole message
# sequence at 15.3 edge-feature GELUs per clock per SM.  Peak = 15.3 x SMs x
# the maximum SM clock.
GELU_PER_CLK_SM = 15.3
EDGE_GELUS_PER_NODE = 2 * 8 * 64


def _sm_count(dev):
    import torch
    return torch.cuda.get_device_properties(dev).multi_processor_count


def _max_sm_hz(dev):
    """Maximum SM clock of the device (nvidia-smi), else GB300's 2,070 MHz."""
    try:
        out = subprocess.run(["nvidia-smi", "-i", str(dev.index or 0),
                              "--query-gpu=clocks.max.sm", "--format=csv,noheader,nounits"],
                             capture_output=True, text=True, timeout=20).stdout.strip()
        return float(out.splitlines()[0]) * 1e6
    except (OSError, ValueError, IndexError, subprocess.SubprocessError):
        return 2.07e9


def gnn_bench(args, L, dev, stream, side=GNN_SIDE, only=False, theta=None, label="xavier"):
    """GNN-LBM MLUPS on the 1024^2 TGV (Re = 1000, u0 = 0.05) beside BGK MLUPS
    on the same lattice, and both TGV velocity L2 errors after the same number
    of steps from the same initial state.  `theta`: parameter vector (default
    Xavier-uniform, seed 0)."""
    import torch
    from paper_2504_14494_gb300 import inputs
    n = side
    s = L.shape(n, n)
    k = 2 * np.pi / n
    tau = 0.5 + 3.0 * U0 * n / GNN_RE
    theta = torch.from_numpy(inputs.xavier_params(0) if theta is None else theta).to(dev)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
    L.gnn_pack(theta, packed)
    ws = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=dev)
    fa = torch.empty(9 * n * n, device=dev)
    fb = torch.empty_like(fa)

    def run(kind, count, bufs):
        for _ in range(count):
            if kind == "gnn":
                L.lbm_step_gnn(bufs[0], bufs[1], s, tau, None, packed, None, ws)
            else:
                L.lbm_step_bgk(bufs[0], bufs[1], None, s, tau)
            bufs.reverse()

    kk = max(10, min(args.steps, 200))
    res = {}
    for kind in ("gnn", "bgk"):
        L.lbm_init_tgv(fa, s, 1.0, U0, k, k, False)
        bufs = [fa, fb]
        run(kind, args.warmup, bufs)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        run(kind, kk, bufs)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / kk
        st = L.lbm_get_status()
        res[kind] = {"ms_per_step": round(ms, 4), "mlups": round(n * n / (ms / 1e3) / 1e6, 1),
                     "l2_error": tgv_l2(L, bufs[0], s, n, U0, tau, args.warmup + kk, dev),
                     "status": st}
    if only:
        return res
    peak = GELU_PER_CLK_SM * _sm_count(dev) * _max_sm_hz(dev) / 1e9
    ach = EDGE_GELUS_PER_NODE * n * n / (res["gnn"]["ms_per_step"] / 1e3) / 1e9
    mlp_only = int(round(float(theta[-1].item()))) & 1
    tr = NCU_TRAFFIC.get("lbm_step_gnn")
    traffic = (tr["bytes_per_launch"] if tr and tr["nodes"] == n * n and not mlp_only
               and tr["src_sha"] == _src_sha(tr["file"]) else None)
    return {"workload": f"tgv_gnn_{n}x{n}", "re": GNN_RE, "tau": round(tau, 5), "u0": U0,
            "roofline": None if mlp_only else {
                "bound": "alu",
                "kernel": "lbm_step_gnn (fused encoder gnn_step_first_kernel + 2 x gnn_round_kernel)",
                "peak_basis": f"{GELU_PER_CLK_SM:.2f} edge GELUs/clock/SM x {_sm_count(dev)} SMs "
                              f"x {_max_sm_hz(dev) / 1e6:.0f} MHz (measured issue rate of the "
                              f"message sequence, MUFU tanh bound; microbench/fp16_rate.cu)",
                "achieved": round(ach, 1), "peak": round(peak, 1), "unit": "G edge-feature GELU/s",
                "frac": round(ach / peak, 4), "traffic": traffic,
                "traffic_note": "DRAM bytes of one step (fused encoder, 2 rounds), ncu"},
            "weights": label,
            "steps_timed": kk, "steps_run": args.warmup + kk,
            "mlups_gnn": res["gnn"]["mlups"], "mlups_bgk_same_lattice": res["bgk"]["mlups"],
            "ms_per_step_gnn": res["gnn"]["ms_per_step"],
            "l2_error_gnn": res["gnn"]["l2_error"], "l2_error_bgk": res["bgk"]["l2_error"],
            "gnn_rollout_diverged": not np.isfinite(res["gnn"]["l2_error"]),
            "gnn_over_bgk_time": round(res["gnn"]["ms_per_step"] / res["bgk"]["ms_per_step"], 2),
            "status": res["gnn"]["status"]}


MLP_SIDE = 4096


def mlp_bench(args, L, dev, stream, theta=None, side=MLP_SIDE):
    """The paper's Fig. 2 network (MLP-only; here with the conserving
    correction, variant 3) stepped by the fused kernel lbm_step_gnn_mlp on
    the side x side TGV (u0 = 0.05, Re = 1000 by tau): MLUPS beside the BGK
    step on the same lattice, and the HBM roofline of the fused kernel (72
    algorithmic bytes per node, as BGK; the two 604 MB buffers exceed L2)."""
    import torch
    from paper_2504_14494_gb300 import inputs
    n = side
    s = L.shape(n, n)
    k = 2 * np.pi / n
    tau = 0.5 + 3.0 * U0 * n / GNN_RE
    if theta is None:
        theta = inputs.xavier_params(0, s_df=1e-4, variant=3)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
    L.gnn_pack(torch.from_numpy(np.asarray(theta, np.float32)).to(dev), packed)
    fa = torch.empty(9 * n * n, device=dev)
    fb = torch.empty_like(fa)
    kk = max(10, min(args.steps, 200))
    res = {}
    for kind in ("mlp", "bgk"):
        L.lbm_init_tgv(fa, s, 1.0, U0, k, k, False)
        bufs = [fa, fb]

        def run(count):
            for _ in range(count):
                if kind == "mlp":
                    L.lbm_step_gnn_mlp(bufs[0], bufs[1], s, tau, None, packed, None)
                else:
                    L.lbm_step_bgk(bufs[0], bufs[1], None, s, tau)
                bufs.reverse()
        run(max(3, args.warmup))
        torch.cuda.synchronize()
        runs = chunk_sizes(kk, RUNS)
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(len(runs) + 1)]
        evs[0].record(stream)
        for i, c in enumerate(runs):
            run(c)
            evs[i + 1].record(stream)
        torch.cuda.synchronize()
        ms = statistics.median(evs[i].elapsed_time(evs[i + 1]) / c for i, c in enumerate(runs))
        res[kind] = {"ms_per_step": round(ms, 5), "mlups": round(n * n / (ms / 1e3) / 1e6, 1),
                     "status": L.lbm_get_status()}
    peak, peak_kind = _peaks()
    ach = BYTES_PER_NODE * n * n / (res["mlp"]["ms_per_step"] / 1e3) / 1e9
    tr = NCU_TRAFFIC.get("gnn_mlp_step_kernel")
    traffic = (tr["bytes_per_launch"] if tr and tr["nodes"] == n * n
               and tr["src_sha"] == _src_sha(tr["file"]) else None)
    return {"workload": f"tgv_gnn_mlp_{n}x{n}", "network": "Fig. 2 MLP-only, conserving (variant 3)",
            "call": "lbm_step_gnn_mlp (one fused kernel: gnn_mlp_step_kernel)", "tau": round(tau, 5),
            "steps_timed": kk, "timing": "median of 5 runs",
            "mlups_gnn_mlp": res["mlp"]["mlups"], "mlups_bgk_same_lattice": res["bgk"]["mlups"],
            "ms_per_step_gnn_mlp": res["mlp"]["ms_per_step"],
            "ms_per_step_bgk": res["bgk"]["ms_per_step"],
            "gnn_over_bgk_time": round(res["mlp"]["ms_per_step"] / res["bgk"]["ms_per_step"], 3),
            "roofline": {"bound": "hbm", "kernel": "gnn_mlp_step_kernel", "achieved": round(ach, 1),
                         "peak": peak, "unit": "GB/s", "frac": round(ach / peak, 4),
                         "peak_kind": peak_kind, "algorithmic_bytes_per_node": BYTES_PER_NODE,
                         "traffic": traffic},
            "status": res["mlp"]["status"]}


def rollout_error(L, dev, theta, n=GNN_SIDE, re=GNN_RE, u0=U0, steps=1000):
    """Velocity L2 error against the closed-form TGV decay after `steps`
    steps of the n^2 TGV at Re: BGK and the GNN-LBM step with parameters
    theta, from the uniform initial density of the timed GNN-LBM workload
    (its start-up acoustic waves dominate the error) and, under
    `pressure_consistent`, from the pressure-consistent density (the
    discretisation error alone)."""
    import torch
    tau = 0.5 + 3.0 * u0 * n / re
    k = 2 * np.pi / n
    s = L.shape(n, n)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
    L.gnn_pack(torch.from_numpy(np.asarray(theta, np.float32)).to(dev), packed)
    ws = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=dev)
    out = {"workload": f"tgv_{n}x{n}_re{re:g}", "steps": steps}
    for pc in (False, True):
        res = out if not pc else out.setdefault("pressure_consistent", {})
        for kind in ("bgk", "gnn"):
            f = [torch.empty(9 * n * n, device=dev) for _ in range(2)]
            L.lbm_init_tgv(f[0], s, 1.0, u0, k, k, pc)
            for _ in range(steps):
                if kind == "bgk":
                    L.lbm_step_bgk(f[0], f[1], None, s, tau)
                else:
                    L.lbm_step_gnn(f[0], f[1], s, tau, None, packed, None, ws)
                f.reverse()
            res[f"l2_error_{kind}"] = tgv_l2(L, f[0], s, n, u0, tau, steps, dev)
        res["gnn_over_bgk"] = res["l2_error_gnn"] / res["l2_error_bgk"]
    L.lbm_get_status()
    return out


def tgv_tables(L, dev, thetas, u0=U0):
    """Analogs of the paper's TGV tables (Sec. 3.2-3.3; the paper states
    neither its u0 nor its error norm): velocity error (relative L2 against
    the closed form) and kinetic-energy error (relative, against
    E(0) exp(-4 nu k^2 t)) for BGK and each network in `thetas`.
      table2: 64^2, Re = 100, after 1000, 3000 and 5000 steps;
      table3: 32^2, 64^2, 128^2 at Re = 100, after the same convective time
              (1000 steps at 64^2, scaled with N);
      energy_re800: 64^2, Re = 800, energy error after 1000 and 5000 steps.
    Re = u0 N / nu; uniform initial density."""
    import torch
    packs = {}
    for name, th in thetas.items():
        pk = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
        L.gnn_pack(torch.from_numpy(np.asarray(th, np.float32)).to(dev), pk)
        packs[name] = pk

    def run(n, re, marks, kind):
        s = L.shape(n, n)
        k = 2 * np.pi / n
        tau = 0.5 + 3.0 * u0 * n / re
        nu = (tau - 0.5) / 3.0
        fa = torch.empty(9 * n * n, device=dev)
        fb = torch.empty_like(fa)
        tot = torch.zeros(5, dtype=torch.float64, device=dev)
        ws = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=dev)
        L.lbm_init_tgv(fa, s, 1.0, u0, k, k, False)
        L.lbm_moments(fa, s, None, None, None, tot)
        e0 = tot[3].item()
        bufs, done, out = [fa, fb], 0, {}
        for mark in marks:
            while done < mark:
                if kind == "bgk":
                    L.lbm_step_bgk(bufs[0], bufs[1], None, s, tau)
                else:
                    L.lbm_step_gnn(bufs[0], bufs[1], s, tau, None, packs[kind], None, ws)
                bufs.reverse()
                done += 1
            L.lbm_moments(bufs[0], s, None, None, None, tot)
            t = tot.cpu().numpy()
            ea = e0 * np.exp(-4 * nu * k * k * mark)
            ok = t[4] == 0 and np.isfinite(t[3])
            out[str(mark)] = {"velocity_l2": tgv_l2(L, bufs[0], s, n, u0, tau, mark, dev) if ok else None,
                              "energy_rel_error": float(abs(t[3] - ea) / ea) if ok else None}
        L.lbm_get_status()
        return {"n": n, "re": re, "tau": round(tau, 6), "errors": out}

    kinds = ["bgk"] + list(packs)
    table2 = {kd: run(64, 100.0, (1000, 3000, 5000), kd) for kd in kinds}
    table3 = {kd: [run(n, 100.0, (1000 * n // 64,), kd) for n in (32, 64, 128)] for kd in kinds}
    energy = {kd: run(64, 800.0, (1000, 5000), kd) for kd in kinds}
    return {"u0": u0, "networks": list(packs), "table2_64_re100": table2,
            "table3_resolution_re100": table3, "energy_64_re800": energy}


def held_out_rollout(L, dev, theta, label, marks=(10, 25, 50, 100, 200, 400)):
    """The held-out rollout check (k = 4 (2 pi / 256), u0 = 0.08, Re = 5000 on
    256^2 coarse nodes): velocity error of BGK and of the GNN-LBM step against
    the restricted 4x refined run, both from the restricted initial state."""
    import torch
    from paper_2504_14494_gb300.train import HeldOutRollout
    run = HeldOutRollout(dev, theta)
    rows = []
    for t in range(1, max(marks) + 1):
        run.step()
        if t in marks:
            (rx, ry), (bx, by), (gx, gy) = [tuple(v.double() for v in u) for u in run.velocities()]
            den = float(torch.sqrt((rx ** 2 + ry ** 2).sum()))
            e_b = float(torch.sqrt(((bx - rx) ** 2 + (by - ry) ** 2).sum())) / den
            e_g = float(torch.sqrt(((gx - rx) ** 2 + (gy - ry) ** 2).sum())) / den
            rows.append({"step": t, "l2_error_bgk": e_b, "l2_error_gnn": e_g,
                         "ratio": e_g / e_b if e_b > 0 else None})
    return {"case": "held-out TGV k = 4 (2 pi / 256), u0 = 0.08, Re = 5000, 256^2 coarse, "
                    "against the restricted 4x refined run", "network": label,
            "rows": rows, "status": L.lbm_get_status()}


def train_bench(args, L, dev, stream, variants=(0, 2, 3)):
    """Training throughput on the 64 x 256^2 batch workload (4x refined data
    generated on the GPU, fused train step), then a short training run on
    64^2 pairs (16 per batch, 3000 steps, lr 1e-4, head starting at zero so
    the network starts as BGK) for each network variant (0: the default
    message-passing network, 2: with the conserving correction, 3: the
    paper's Fig. 2 MLP-only network with the conserving correction) and the
    held-out Eq. 4 loss ratio against BGK.  Returns ({variant: theta}, info)."""
    import torch
    from paper_2504_14494_gb300 import inputs
    from paper_2504_14494_gb300.train import Evaluator, PairStream, Trainer
    theta = inputs.xavier_params(0, s_df=1e-4)
    theta[38272:38922] = 0.0
    T = W.TRAIN_64x256
    tr = Trainer(dev, theta=theta.copy(), lr=T.lr, wd=T.weight_decay, seed=T.seed, n=T.n,
                 batch=T.batch, m=T.refine, episode=T.episode)
    for _ in range(3):
        tr.step()
    torch.cuda.synchronize()
    kk = 20
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(kk):
        tr.step()
    e1.record(stream)
    torch.cuda.synchronize()
    ms_full = e0.elapsed_time(e1) / kk
    f_in, f_tg, taus = tr.data.next()
    e0.record(stream)
    for i in range(kk):
        L.gnn_train_step(f_in, f_tg, tr.data.coarse, 1.0, taus, tr.params, tr.packed, tr.m, tr.v,
                         100 + i, 1e-4, 0.0, tr.loss, None, tr.ws)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_step = e0.elapsed_time(e1) / kk
    del tr
    thetas, runs = {}, {}
    # (variant, lr, weight decay): lr 1e-4 without decay for the networks
    # used below, and the default network at AdamW lr 1e-3, decay 1e-2
    plan = [(v, 1e-4, 0.0) for v in variants] + [(0, 1e-3, 1e-2)]
    for var, lr, wd in plan:
        th = inputs.xavier_params(0, s_df=1e-4, variant=var)
        th[38272:38922] = 0.0
        small = Trainer(dev, theta=th, lr=lr, wd=wd, seed=1, n=64, batch=16, episode=64)
        curve = []
        t0 = time.perf_counter()
        for i in range(3000):
            small.step()
            if i % 250 == 0 or i == 2999:
                curve.append([i + 1, small.loss.item()])  # Eq. 4 loss before step i+1's update
        torch.cuda.synchronize()
        t_train = time.perf_counter() - t0
        held = PairStream(dev, n=64, batch=16, m=4, episode=24, seed=12345)
        ev = Evaluator(dev, held.coarse)
        zero = torch.from_numpy(inputs.zero_params(s_df=1e-4, variant=var)).to(dev)
        lg = lb = 0.0
        for _ in range(48):
            a, b, t = held.next()
            lg += ev.loss_of(small.params, a, b, t)
            lb += ev.loss_of(zero, a, b, t)
        key = str(var) if lr == 1e-4 else f"{var}_lr{lr:g}_wd{wd:g}"
        if lr == 1e-4:
            thetas[var] = small.theta()
        runs[key] = {"steps": 3000, "lr": lr, "weight_decay": wd, "wall_s": round(t_train, 2),
                     "held_out_eq4_loss_gnn": lg / 48, "held_out_eq4_loss_bgk": lb / 48,
                     "ratio": round(lg / lb, 4), "loss_curve": curve}
    # the fixed-tau network of the held-out rollout check: message passing,
    # Delta f unconstrained, tau_adj = 1; 16 x 256^2 pairs per batch (4x
    # refined), AdamW lr 1e-3, weight decay 1e-2, 3000 steps
    th = inputs.xavier_params(0, s_df=1e-4, variant=inputs.FIXED_TAU)
    th[38272:38922] = 0.0
    fixed = Trainer(dev, theta=th, lr=1e-3, wd=1e-2, seed=1, n=256, batch=16, m=4, episode=32)
    t0 = time.perf_counter()
    curve = []
    for i in range(3000):
        fixed.step()
        if i % 500 == 0 or i == 2999:
            curve.append([i + 1, fixed.loss.item()])
    torch.cuda.synchronize()
    thetas[4] = fixed.theta()
    t_fixed = time.perf_counter() - t0
    # the network of Eq. 3 as printed trained with each instance weighted by
    # its error relative to BGK (lbm_pair_weights + gnn_train_step_weighted),
    # same recipe, three training seeds
    thetas["relative"] = {}
    for sd in (1, 2, 3):
        th = inputs.xavier_params(0, s_df=1e-4)
        th[38272:38922] = 0.0
        wtr = Trainer(dev, theta=th, lr=1e-3, wd=1e-2, seed=sd, n=256, batch=16, m=4, episode=32,
                      weighting="relative")
        t0 = time.perf_counter()
        for _ in range(3000):
            wtr.step()
        torch.cuda.synchronize()
        thetas["relative"][sd] = wtr.theta()
        runs[f"0_relative_256_seed{sd}"] = {"steps": 3000, "lr": 1e-3, "weight_decay": 1e-2,
                                            "batch": 16, "coarse": 256, "weighting": "relative",
                                            "wall_s": round(time.perf_counter() - t0, 2),
                                            "last_weighted_loss": wtr.loss.item()}
        del wtr
    runs["4_fixed_tau_256"] = {"steps": 3000, "lr": 1e-3, "weight_decay": 1e-2, "batch": 16,
                               "coarse": 256, "wall_s": round(t_fixed, 2), "loss_curve": curve}
    del fixed
    # the conserving network trained on high-Re pairs for the stability
    # sweep: u0 ~ U[0.1, 0.3], Re log-uniform in [400, 51200], 64^2 coarse
    # (4x refined), 16 per batch, AdamW lr 1e-3, decay 1e-2, 3000 steps
    th = inputs.xavier_params(0, s_df=1e-4, variant=inputs.CONSERVATIVE)
    th[38272:38922] = 0.0
    hre = Trainer(dev, theta=th, lr=1e-3, wd=1e-2, seed=7, n=64, batch=16, m=4, episode=64,
                  instances={"u0_range": (0.1, 0.3), "re_range": (400.0, 51200.0),
                             "log_re": True})
    t0 = time.perf_counter()
    curve = []
    for i in range(3000):
        hre.step()
        if i % 500 == 0 or i == 2999:
            curve.append([i + 1, hre.loss.item()])
    torch.cuda.synchronize()
    thetas["2_high_re"] = hre.theta()
    runs["2_high_re_64"] = {"steps": 3000, "lr": 1e-3, "weight_decay": 1e-2, "batch": 16,
                            "coarse": 64, "u0": [0.1, 0.3], "re_log_uniform": [400, 51200],
                            "wall_s": round(time.perf_counter() - t0, 2), "loss_curve": curve}
    del hre
    info = {"workload": "train_64x256x256_refined4",
            "ms_per_train_step_incl_datagen": round(ms_full, 3),
            "ms_per_fused_train_step": round(ms_step, 3),
            "samples_per_s": round(64 / (ms_full / 1e3), 1),
            "node_updates_per_s_M": round(64 * 256 * 256 / (ms_step / 1e3) / 1e6, 1),
            "short_runs_by_variant": runs,
            "short_run_data": "64^2 coarse pairs from 256^2 refined runs, 16 per batch; "
                              "loss_curve: [step, Eq. 4 loss of that step's batch]"}
    return thetas, info


def batch_bench(args, L, dev, stream, theta, n_lat=W.BATCH_512.lattices, seed=W.BATCH_512.seed):
    """The serving-style batch: 512 TGV lattices, sides log-uniform in
    [32, 1024], Re ~ U[100, 5000], u0 ~ U[0.01, 0.08], first half plain BGK,
    second half GNN-corrected (trained weights); 1,000 steps of all lattices
    are one replay of a recorded CUDA graph (lbm_batch_run; the timed call
    records it).  Each half is also timed alone (100 steps, on a second call
    that replays the recorded graph) for its own MLUPS."""
    import torch
    from paper_2504_14494_gb300 import inputs
    B = W.BATCH_512
    draws = inputs.batch_lattices(n_lat, seed, B.side_lo, B.side_hi, B.re_lo, B.re_hi)
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
    L.gnn_pack(torch.from_numpy(theta).to(dev), packed)

    def run(sel, steps, replay=False):
        ds = [d for d in draws if sel(d)]
        lat = [(d["side"], d["side"], 1 if d["gnn"] else 0, 0.5 + 3.0 * d["nu"]) for d in ds]
        plan = L.lbm_batch_plan_create(lat)
        try:
            n = L.lbm_batch_nodes(plan)
            prm = np.array([(1.0, d["u0"], 2 * np.pi / d["side"], 2 * np.pi / d["side"])
                            for d in ds])
            f0 = torch.empty(9 * n, device=dev)
            f1, f2 = torch.empty_like(f0), torch.empty_like(f0)
            L.lbm_batch_init_tgv(plan, f0, prm, True)
            ws = torch.empty(max(L.lbm_batch_workspace_bytes(plan), 16), dtype=torch.uint8,
                             device=dev)
            L.lbm_batch_run(plan, f0, f1, f2, 1, packed, ws)   # autotune
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for _ in range(2 if replay else 1):  # a second identical call replays the graph
                e0.record(stream)
                L.lbm_batch_run(plan, f0, f1, f2, steps, packed, ws)  # (records +) runs the graph
                e1.record(stream)
                torch.cuda.synchronize()
            ms = e0.elapsed_time(e1)
            return n, ms, L.lbm_get_status()
        finally:
            L.lbm_batch_plan_destroy(plan)

    kk = B.steps if args.steps >= B.steps else max(2, args.steps)
    n, ms, st = run(lambda d: True, kk)
    import tempfile
    with tempfile.TemporaryDirectory() as tdir:
        path = os.path.join(tdir, "tune.json")
        L.lbm_autotune_save(path)
        with open(path) as fh:
            tuned = json.load(fh)
    halves = {}
    for name, sel in (("bgk_half", lambda d: not d["gnn"]), ("gnn_half", lambda d: d["gnn"])):
        nh, msh, sth = run(sel, min(kk, 100), replay=True)
        halves[name] = {"lattices": sum(1 for d in draws if sel(d)), "nodes": int(nh),
                        "steps": min(kk, 100), "ms_per_step": round(msh / min(kk, 100), 3),
                        "mlups": round(nh * min(kk, 100) / (msh / 1e3) / 1e6, 1), "status": sth,
                        "timing": "second identical call: the recorded graph replayed"}
    return {"workload": f"batch_{n_lat}_lattices_sides_32_1024", "seed": seed,
            "nodes": int(n), "nodes_gnn": halves["gnn_half"]["nodes"], "steps": kk,
            "graph_launches": 1, "ms_per_step": round(ms / kk, 3),
            "mlups_total": round(n * kk / (ms / 1e3) / 1e6, 1), "status": st,
            "timing": "one lbm_batch_run call of all steps (graph recording included)",
            "autotuner_choices": tuned,
            **halves}


def stability_bench(L, dev, theta, n=64, u0s=(0.1, 0.2, 0.3),
                    res=(400.0, 1600.0, 3200.0, 12800.0, 51200.0), steps=5000, chunk=250):
    """Reynolds-number study on the 64^2 TGV (paper Sec. 3.4), widened in
    Mach number (u0) and Re until the plain BGK step fails: BGK and GNN-LBM
    (the network trained in this run) for `steps` steps at each u0 and
    Re = u0 n / nu; the first chunk of `chunk` steps whose state holds a
    non-finite value (FP64 totals of the library), and the kinetic-energy
    error against the closed-form decay E(0) exp(-4 nu k^2 t) at the last
    finite chunk."""
    import torch
    s = L.shape(n, n)
    k = 2 * np.pi / n
    packed = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
    L.gnn_pack(torch.from_numpy(theta).to(dev), packed)
    ws = torch.empty(L.gnn_step_workspace_bytes(s), dtype=torch.uint8, device=dev)
    fa = torch.empty(9 * n * n, device=dev)
    fb, fc = torch.empty_like(fa), torch.empty_like(fa)
    tot = torch.zeros(5, dtype=torch.float64, device=dev)
    out = []
    for u0, re in [(a, b) for a in u0s for b in res]:
        nu = u0 * n / re
        tau = 0.5 + 3.0 * nu
        row = {"u0": u0, "re": re, "tau": round(tau, 6)}
        for kind in ("bgk", "gnn"):
            L.lbm_init_tgv(fa, s, 1.0, u0, k, k, False)
            L.lbm_moments(fa, s, None, None, None, tot)
            e0 = tot[3].item()
            done, bad, err = 0, None, None
            cur, nxt = fa, fb
            while done < steps:
                if kind == "bgk":
                    L.lbm_step_bgk(cur, nxt, fc, s, tau, nsteps=chunk, totals=tot)
                else:
                    for _ in range(chunk):
                        L.lbm_step_gnn(cur, nxt, s, tau, None, packed, None, ws)
                        cur, nxt = nxt, cur
                    cur, nxt = nxt, cur
                    L.lbm_moments(nxt, s, None, None, None, tot)
                done += chunk
                cur, nxt = nxt, cur
                t = tot.cpu().numpy()
                if t[4] > 0 or not np.isfinite(t[3]):
                    bad = done
                    break
                err = abs(t[3] - e0 * np.exp(-4 * nu * k * k * done)) / (e0 * np.exp(-4 * nu * k * k * done))
            L.lbm_get_status()  # clear the non-finite flag of an unstable run
            row[kind] = {"first_nonfinite_by_step": bad, "steps_finite": done if bad is None else bad - chunk,
                         "energy_rel_error": err}
        out.append(row)
    return {"workload": f"tgv_{n}x{n}", "steps": steps, "chunk": chunk, "rows": out}


def _channel_profile_error(L, f, s, h, nx, g, nu, umax, dev):
    """Maximum |u - u_Eq.5| over the channel's rows, relative to u_max, with
    the forced velocity (sum f e + F/2)/rho of column 0."""
    import torch
    n = nx * h
    rho = torch.empty(n, device=dev)
    ux = torch.empty(n, device=dev)
    L.lbm_moments(f, s, rho, ux, None)
    u = (ux.double() + 0.5 * g / rho.double()).view(h, nx)[:, 0].cpu().numpy()
    y = np.arange(h) + 0.5
    ua = g / (2 * nu) * y * (h - y)
    return float(np.abs(u - ua).max() / umax) if np.all(np.isfinite(u)) else None


def _channel_gnn_run(L, dev, s, fa, fb, tau, g, steps, packed, ws, chunk=100):
    """`steps` GNN-LBM steps of the channel from fa, ping-pong between fa
    and fb; `chunk` steps (even) replayed as one CUDA graph.  Returns the
    buffer holding the final state."""
    import torch

    def step(a, b):
        L.lbm_step_gnn_channel(a, b, s, tau, None, g, packed, None, ws)

    cur, nxt = fa, fb
    done = 0
    while done < min(steps, 2):  # warm-up outside the capture
        step(cur, nxt)
        cur, nxt = nxt, cur
        done += 1
    torch.cuda.synchronize()
    if steps - done >= chunk:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, capture_error_mode="thread_local"):
            for _ in range(chunk // 2):
                step(cur, nxt)
                step(nxt, cur)
        while steps - done >= chunk:
            graph.replay()
            done += chunk
    while done < steps:
        step(cur, nxt)
        cur, nxt = nxt, cur
        done += 1
    torch.cuda.synchronize()
    return cur


def channel_train(L, dev, steps=20000):
    """Channel networks trained on refined-channel data (Sec. 2.4 data for
    the flow of Sec. 3.1): a ChannelPairBank of 16 groups x 8 lattices x 14
    snapshot times (H = 32, nx = 8, refined 3x, u_ref ~ U[0.03, 0.07], Re_ref
    log-uniform in [8, 250]), 64 lattices per batch, AdamW lr 1e-3, decay
    1e-2, s_Delta_f = 1e-3, head starting at zero (the network starts as
    BGK), for the network of Eq. 3 as printed (variant 0) and the conserving
    one (variant 2).  The Eq. 4 loss is reported on the whole training bank
    and on a held-out bank (4 groups, another seed) against the zero network
    (BGK with Guo forcing).  Returns ({name: theta}, info)."""
    import torch
    from paper_2504_14494_gb300 import inputs
    from paper_2504_14494_gb300.train import ChannelPairBank, ChannelTrainer
    t0 = time.perf_counter()
    bank = ChannelPairBank(dev, seed=0)
    held = ChannelPairBank(dev, seed=1, groups=4)
    torch.cuda.synchronize()
    t_bank = time.perf_counter() - t0
    thetas, runs = {}, {}
    for name, var in (("channel_eq3_v0", 0), ("channel_conserving_v2", inputs.CONSERVATIVE)):
        th = inputs.xavier_params(0, s_df=1e-3, variant=var)
        th[38272:38922] = 0.0
        tr = ChannelTrainer(dev, bank, theta=th, lr=1e-3, wd=1e-2, batch=64, seed=1)
        zero = torch.from_numpy(inputs.zero_params(s_df=1e-3, variant=var)).to(dev)
        curve = [[0, tr.bank_loss(bank)]]
        t1 = time.perf_counter()
        for i in range(steps):
            tr.step()
            if (i + 1) % 5000 == 0:
                curve.append([i + 1, tr.bank_loss(bank)])
        torch.cuda.synchronize()
        lg, lb = tr.bank_loss(held), tr.bank_loss(held, zero)
        thetas[name] = tr.theta()
        runs[name] = {"variant": var, "steps": steps, "lr": 1e-3, "weight_decay": 1e-2,
                      "s_df": 1e-3, "batch": 64, "wall_s": round(time.perf_counter() - t1, 2),
                      "bank_loss_curve": curve, "held_out_eq4_loss_gnn": lg,
                      "held_out_eq4_loss_bgk": lb, "ratio": round(lg / lb, 4)}
    info = {"bank": {"lattices": bank.nb, "h": bank.h, "nx": bank.nx, "refine": bank.m,
                     "snapshots_efold": list(ChannelPairBank.SNAPSHOTS),
                     "held_out_lattices": held.nb, "build_s": round(t_bank, 2)},
            "runs": runs}
    return thetas, info


def channel_bench(L, dev, thetas=None, h=32, nx=4, umax=0.05, res=(10.0, 50.0, 100.0, 200.0),
                  sides=(4, 8, 16, 32), re_sides=10.0, tau_sides=1.0):
    """Poiseuille channel (paper Sec. 3.1, Table 1 analog): halfway
    bounce-back walls and Guo forcing, H = 32, centre-line velocity 0.05.
    BGK runs from rest to steady state (35 e-folding times h^2/(pi^2 nu) of
    the slowest mode); each network in `thetas` (GNN-LBM step of the channel,
    lbm_step_gnn_channel) then runs from the BGK steady state for 7 more
    e-folding times (its own steady state differs from BGK's by a small
    offset, which decays at the same rate), with the error after 6 reported
    as a convergence check.  Error: maximum |u - u_Eq.5| over the rows,
    relative to the centre-line velocity.  Grid refinement: heights `sides`
    at fixed tau_sides and Re = re_sides (u_max = Re nu / H: the diffusive
    scaling, under which the wall slip of halfway bounce-back,
    (G/nu)(16 tau^2 - 8 tau - 3)/24, falls as 1/H^2 relative to u_max).  The
    FP32 populations put a floor under the error: the iteration settles
    within ~ulp(f) H^2/(pi^2 nu) of its fixed point, which relative to
    u_max = Re nu / H grows as H^3 and passes the slip beyond H ~ 32 at
    tau = 1, Re = 10 (and at smaller H for smaller tau)."""
    import torch
    thetas = thetas or {}
    packs = {}
    for name, th in thetas.items():
        pk = torch.empty(L.gnn_packed_bytes(), dtype=torch.uint8, device=dev)
        L.gnn_pack(torch.from_numpy(np.asarray(th, np.float32)).to(dev), pk)
        packs[name] = pk

    def case(hh, re, tau=None):
        s = L.shape(nx, hh)
        n = nx * hh
        if tau is None:
            um = umax
            nu = um * hh / re
            tau = 0.5 + 3.0 * nu
        else:
            nu = (tau - 0.5) / 3.0
            um = re * nu / hh
        g = 8.0 * nu * um / (hh * hh)
        efold = hh * hh / (np.pi ** 2 * nu)
        steps = int(35 * efold)
        fa = torch.empty(9 * n, device=dev)
        fb, fc = torch.empty_like(fa), torch.empty_like(fa)
        L.lbm_init_tgv(fa, s, 1.0, 0.0, 0.0, 0.0, False)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        L.lbm_step_channel(fa, fb, fc, s, tau, None, g, steps)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        row = {"re": re, "h": hh, "tau": round(tau, 5), "u_max": round(um, 6), "steps": steps,
               "max_velocity_error": _channel_profile_error(L, fb, s, hh, nx, g, nu, um, dev),
               "mlups": round(n * steps / dt / 1e6, 1)}
        if packs:
            ws = torch.empty(L.gnn_channel_workspace_bytes(s), dtype=torch.uint8, device=dev)
            gnn = {}
            k6, k1 = int(6 * efold), int(efold)
            for name, pk in packs.items():
                fa.copy_(fb)
                fin = _channel_gnn_run(L, dev, s, fa, fc, tau, g, k6, pk, ws)
                e6 = _channel_profile_error(L, fin, s, hh, nx, g, nu, um, dev)
                other = fc if fin is fa else fa
                fin = _channel_gnn_run(L, dev, s, fin, other, tau, g, k1, pk, ws)
                err = _channel_profile_error(L, fin, s, hh, nx, g, nu, um, dev)
                L.lbm_get_status()  # clear a non-finite flag
                base = row["max_velocity_error"]
                gnn[name] = {"max_velocity_error": err, "after_6_efolds": e6,
                             "improvement_pct": (None if err is None or not base
                                                 else round(100 * (1 - err / base), 2))}
            row["gnn_from_bgk_steady_state"] = {"steps": k6 + k1, "networks": gnn}
        return row

    t0 = time.perf_counter()
    out = [case(h, re) for re in res]
    grid = [case(hh, re_sides, tau_sides) for hh in sides]
    for a, b in zip(grid, grid[1:]):
        if a["max_velocity_error"] and b["max_velocity_error"]:
            b["order_vs_previous"] = round(float(np.log2(a["max_velocity_error"]
                                                         / b["max_velocity_error"])), 3)
    return {"workload": f"poiseuille_{nx}x{h}", "u_max": umax,
            "call": "lbm_step_channel (BGK); lbm_step_gnn_channel (GNN, CUDA-graph chunks)",
            "networks": list(packs), "rows": out,
            "grid_refinement": {"re": re_sides, "tau": tau_sides, "rows": grid},
            "wall_s": round(time.perf_counter() - t0, 1)}


def cpu_baseline(budget_s=12.0):
    """The FP64 oracle BGK step, as it stands, on a bounded sample: a periodic
    TGV sub-lattice of 1024 x 1024 nodes stepped until ~budget_s of CPU time
    (numpy, one thread)."""
    from oracle import lbm
    n = 1024
    k = 2 * np.pi / n
    f = lbm.tgv_init(n, n, 1.0, U0, k, k)
    steps = 0
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < budget_s:
        f = lbm.bgk_step(f, TAU)
        steps += 1
    dt = time.perf_counter() - t0
    return {"value": round(n * n * steps / dt / 1e6, 3), "unit": "MLUPS", "cores": 1,
            "kind": "oracle",
            "sample": f"oracle.lbm.bgk_step (numpy FP64) on a 1024x1024 TGV sub-lattice, "
                      f"{steps} steps, {dt:.1f} s"}


def _oracle_worker(budget_s):
    """One host core: the oracle BGK step on its own 512 x 512 TGV lattice
    until ~budget_s have passed; returns node updates."""
    from oracle import lbm
    n = 512
    k = 2 * np.pi / n
    f = lbm.tgv_init(n, n, 1.0, U0, k, k)
    steps = 0
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < budget_s:
        f = lbm.bgk_step(f, TAU)
        steps += 1
    return n * n * steps


def cpu_baseline_all_cores(budget_s=8.0):
    """The same oracle on every host core at once (one process per core, each
    with an independent lattice: weak scaling, no exchange)."""
    import multiprocessing as mp
    cores = os.cpu_count() or 1
    for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ.setdefault(var, "1")
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_worker, [0.0] * cores)  # interpreters and numpy loaded
        t0 = time.perf_counter()
        updates = sum(pool.map(_oracle_worker, [budget_s] * cores))
        dt = time.perf_counter() - t0
    return {"value": round(updates / dt / 1e6, 3), "unit": "MLUPS", "cores": cores,
            "kind": "oracle",
            "sample": f"oracle.lbm.bgk_step (numpy FP64) on {cores} independent 512x512 TGV "
                      f"lattices, one process per core, {dt:.1f} s"}


def run_reference(args, rank):
    """The CPU oracle arm: each step is one oracle BGK step on a sub-lattice
    sized so that the whole run takes about two minutes."""
    if rank != 0:
        return None
    from oracle import lbm
    total = args.warmup + args.steps
    # measured oracle throughput on this host, to size the per-step sample
    probe = lbm.tgv_init(256, 256, 1.0, U0, 2 * np.pi / 256, 2 * np.pi / 256)
    t0 = time.perf_counter()
    lbm.bgk_step(probe, TAU)
    rate = 256 * 256 / max(time.perf_counter() - t0, 1e-6)
    per_step = 120.0 / total
    side = int(np.sqrt(rate * per_step) // 64 * 64)
    side = max(64, min(N_SIDE, side))
    k = 2 * np.pi / side
    f = lbm.tgv_init(side, side, 1.0, U0, k, k)
    for _ in range(args.warmup):
        f = lbm.bgk_step(f, TAU)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        f = lbm.bgk_step(f, TAU)
    dt = time.perf_counter() - t0
    val = round(side * side * args.steps / dt / 1e6, 3)
    sample = (f"oracle.lbm.bgk_step (numpy FP64, 1 thread) on a {side}x{side} TGV sub-lattice "
              f"of the 4096x4096 workload per step")
    return {"impl": "reference", "metric": METRIC, "value": val, "unit": "MLUPS",
            "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(dt / args.steps * 1e3, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "tgv_bgk_4096x4096", "nx": N_SIDE, "ny": N_SIDE,
                       "tau": TAU, "u0": U0, "sample_side": side},
            "cpu_baseline": {"value": val, "unit": "MLUPS", "cores": 1, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": val, "unit": "MLUPS", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--only", choices=["bgk", "gnn", "train", "batch", "mlp", "channel"],
                    default=None,
                    help="time one kernel family only (profiling runs)")
    ap.add_argument("--side", type=int, default=N_SIDE, help="lattice side for --only runs")
    ap.add_argument("--log", default=None,
                    help="also append the full record to this JSON-lines file (rank 0)")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.only is None and args.side != N_SIDE:
        ap.error("--side applies to --only runs")
    if args.only == "gnn" and args.side == N_SIDE:
        args.side = GNN_SIDE
    if args.only == "train" and args.side == N_SIDE:
        args.side = 256
    if args.only == "mlp" and args.side == N_SIDE:
        args.side = MLP_SIDE
    if args.impl == "reference":
        out = run_reference(args, rank)
    else:
        out = run_ours(args, rank, world, local_rank)
    if out is not None and rank == 0:
        line = json.dumps(_finite(out), allow_nan=False)
        print("full record: " + line, file=sys.stderr, flush=True)
        print(json.dumps(_finite(headline(out)), allow_nan=False), flush=True)
        if args.log:
            d = os.path.dirname(os.path.abspath(args.log))
            os.makedirs(d, exist_ok=True)
            with open(args.log, "a") as fh:
                fh.write(line + "\n")


if __name__ == "__main__":
    main()
