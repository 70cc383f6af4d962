#!/usr/bin/env python3
"""Benchmark of the ECASQ hot path on one GB300 (or N replicas).

One step = one budgeted solve of the workload vector (sort, weighted
histogram, prefix sums, approximate-DP multiplier search, traceback,
refinement to 1e-9 relative) followed by the stochastic-rounding encode of the
vector with the chosen codebook.  Default workload: d = 2^17 Student-t(3) x 1e-3,
s = 16, budget 2.5 bits/entry (the configuration the headline metric names).

Prints one JSON line (rank 0).  `value` is min-plus candidate evaluations per
second over the whole job (inputs resident in HBM); `e2e` is the same metric
through the C ABI with host buffers; `roofline` relates the min-plus kernel to
the FP32-pipe issue peak; `cpu_baseline` is the CPU oracle on a bounded sample.

Other rows of the path, each timed the same way on the chosen --config:
  --mode grid       the codebook drawn from a uniform min-max grid of --grid values
                    (Sec. 5 / App. E general P); metric: solves/s
  --mode timeshare  the budgeted solve with two-way time-sharing (Sec. 7) and the
                    time-shared encode; metric: solves/s
  --mode opt        one pass of the optimal DP (Sec. 4) at 8 multipliers over a uniform
                    grid of --grid values; metric: candidate evaluations/s
  --mode hbm        the HBM-bound rows on vectors far larger than L2: the encode (A10,
                    2^28 entries) and the sort + histogram + prefix sums (A1-A3, 2^26
                    entries); metric: GB/s of algorithmic traffic
  --mode rows       the batched solve of many independent short rows (the KV-cache-like
                    workload, 8192 rows of 128 entries); metric: rows/s
  --mode pass       one DP pass (sort, histogram, interval costs, the min-plus layers, the
                    exact stage, traceback) of the --config vector at the multipliers of
                    --lambdas; metric: candidate evaluations/s
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "ECASQ approx-DP solve ms & candidate evals/s at d=2^17,s=16; % of ALU peak"
UNIT = "candidate evals/s"
FP32_LANES = 128          # FP32-pipe lanes per SM (adds and min/max share them)
SM_MAX_MHZ = 2070.0
# Ops counted per candidate: one add (packed f32x2) and one min (3-input integer min on
# the float bits).  W = C + lambda' Phi is the same for every layer of a (pair, multiplier);
# the near phase forms it once, the far phase again in each task (an FMA that is not counted).
OPS_PER_CANDIDATE = 2
BK = BJ = 64              # the kernel's tile: 64 k by 64 columns
# Bytes that the min-plus kernel copies per interval-cost tile: the tile's 34 816 B of C and Phi, each
# fetched tile once in a pass, from HBM or L2 -- an upper bound of the DRAM reads.  (Of one solve's copies at
# d = 16384, 3.66 GB, 1.95 GB came from HBM; at d = 131072 a pass copies 26 GB.)
TRAFFIC_PER_FETCHED_TILE = 34816
ORACLE_SAMPLE = 16384     # entries of the CPU baseline's bounded sample


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--config", default="studentt_d131072_s16")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--mode", default="solve",
                    choices=["solve", "grid", "timeshare", "opt", "hbm", "rows", "pass", "linear"])
    ap.add_argument("--lambdas", default="0.02", help="comma-separated multipliers (vNMSE scale) for --mode pass")
    ap.add_argument("--grid", type=int, default=256, help="grid size for --mode grid")
    ap.add_argument("--prefix", type=int, default=0,
                    help="--mode pass: use only the first N entries of the configuration's vector")
    return ap.parse_args()


def max_over_ranks(x, dist, device):
    """The largest x over all ranks (the job's time is its slowest replica's)."""
    if dist is None:
        return float(x)
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(world, units_per_rank, ms):
    """Units per second of the whole job: every replica processes units_per_rank in ms
    (the max over ranks), so the aggregate is world * units / time (weak scaling)."""
    return world * units_per_rank / (ms / 1000.0)


def candidates_per_multiplier(p, s):
    """Candidates of eq. apx_rec for one multiplier: layers 3..s, j in [i-1, p-1], k in [i-2, j-1]."""
    c = 0
    for i in range(3, s + 1):
        n = p - (i - 1)
        if n <= 0:
            break
        c += n * (n + 1) // 2
    return c


def executed_candidates(st, p, s, multipliers):
    """Candidates the min-plus kernel evaluated in one solve, from its own counters:
    every off-diagonal (multiplier, tile) unit it ran is 64 x 64 pairs times the s - 2
    layers; every diagonal block is evaluated for each multiplier of its pass, with its
    pairs k < j (a 64-column triangle) over the s - 2 layers."""
    L = max(s - 2, 0)
    n_blocks = -(-p // BJ)
    off = st["tiles_run"] * BK * BJ * L
    diag = multipliers * n_blocks * (BJ * (BJ - 1) // 2) * L
    return off + diag


def cost_mode_flags(E, d, s, free_bytes, share=0.6):
    """Interval-cost mode of the fast DP: the whole table resident when it fits in `share` of
    the free device memory, else band by band through a bounded buffer when that fits, else
    the kernel that rebuilds the costs panel by panel in every pass."""
    for flag in (E.RESIDENT_COSTS, E.STREAMED_COSTS):
        need = E.ecasq_workspace_size_flags(d, s, 1, flag)
        if 0 < need <= share * free_bytes:
            return flag
    return 0


def cost_mode_name(E, flags):
    return "resident" if flags & E.RESIDENT_COSTS else ("streamed" if flags & E.STREAMED_COSTS else "fused")


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""
    REASONS = {0x1: "gpu_idle", 0x2: "applications_clocks_setting", 0x4: "sw_power_cap", 0x8: "hw_slowdown",
               0x10: "sync_boost", 0x20: "sw_thermal_slowdown", 0x40: "hw_thermal_slowdown",
               0x80: "hw_power_brake_slowdown", 0x100: "display_clock_setting"}

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=clocks.sm,clocks.max.sm,power.draw,"
                 "clocks_event_reasons.active", "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            threading.Thread(target=self._read, daemon=True).start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        for ln in self.lines:
            parts = [t.strip() for t in ln.split(",")]
            if len(parts) < 4:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
                mask = int(parts[3], 16) if parts[3].startswith("0x") else int(parts[3])
            except ValueError:
                continue
            for bit, name in self.REASONS.items():
                if mask & bit and name != "gpu_idle":
                    reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def cpu_baseline(x, cfg):
    """The oracle (as it stands) on a bounded sample: the full multiplier search
    on the first ORACLE_SAMPLE entries, timed on this host's cores."""
    import oracle
    xs = x[:ORACLE_SAMPLE]
    t0 = time.perf_counter()
    H = oracle.Hist(xs)
    H.cache()
    r = H.search(cfg["s"], cfg["budgets"][0])
    dt = time.perf_counter() - t0
    cand = r["n_evaluated"] * candidates_per_multiplier(H.p, cfg["s"])
    return {"value": cand / dt, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": "full lambda search (%d multipliers) on the first %d of the %d entries, %.2f s" %
                      (r["n_evaluated"], xs.size, x.size, dt)}


def run_reference(args, cfg, x):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    for _ in range(args.warmup):
        cpu_baseline(x, cfg)
    vals, t0 = [], time.perf_counter()
    for _ in range(args.steps):
        vals.append(cpu_baseline(x, cfg))
    dt = time.perf_counter() - t0
    v = statistics.mean(b["value"] for b in vals)
    cb = dict(vals[0])
    cb["value"] = v
    out = {"metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": 1000.0 * dt / args.steps, "higher_is_better": True,
           "impl": "reference", "dtype": "f64", "data": "synthetic",
           "config": {"workload": args.config, "s": cfg["s"], "budget_bits": cfg["budgets"][0],
                      "sample_entries": ORACLE_SAMPLE},
           "cpu_baseline": cb, "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "vs_baseline": None}
    print(json.dumps(out), flush=True)


def run_other_mode(args, cfg, x_np):
    """--mode grid / timeshare: solves per second of that entry point on one GPU,
    timed with CUDA events around `steps` solves (+ encodes), inputs in HBM."""
    import torch
    import paper_2608_18147_gb300 as E
    s, budget = cfg["s"], cfg["budgets"][0]
    d = x_np.size
    x = torch.as_tensor(x_np).cuda()
    idx = torch.empty(d, dtype=torch.uint8, device="cuda")
    counts = torch.empty(2 * s, dtype=torch.int32, device="cuda")
    qws = torch.empty(256, dtype=torch.uint8, device="cuda")
    flags = E.TIME_KERNELS
    if args.mode == "opt":
        run_opt_mode(args, cfg, x_np)
        return
    if args.mode == "hbm":
        run_hbm_mode(args)
        return
    if args.mode == "rows":
        run_rows_mode(args)
        return
    if args.mode == "pass":
        run_pass_mode(args, cfg, x_np)
        return
    if args.mode == "linear":
        run_linear_mode(args, cfg, x_np)
        return
    if args.mode == "grid":
        g = torch.as_tensor(E.uniform_grid(x_np, args.grid)).cuda()
        ws = torch.empty(int(E.lib().ecasq_workspace_size_grid(d, g.numel(), s, flags)), dtype=torch.uint8,
                         device="cuda")

        def step():
            Q, res = E.ecasq_solve_grid(x, g, s, budget_bits=budget, ws=ws, flags=flags)
            _, _, he = E.ecasq_quantize(x, Q, seed=12345, ws=qws, idx=idx, counts=counts[:Q.numel()])
            return res, {}
    else:
        flags |= cost_mode_flags(E, d, s, torch.cuda.mem_get_info()[0])
        ws = E.workspace(d, s, flags=flags)

        def step():
            Qm, Qp, res, ts = E.ecasq_solve_timeshare(x, s, budget, ws=ws, flags=flags)
            _, _, _, rate = E.ecasq_quantize_timeshare(x, Qm, Qp, ts["beta"], 12345, 678, ws=qws)
            ts["rate_emp"] = rate
            return res, ts
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    launches0 = E.ecasq_kernel_launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    out_res = []
    with ClockSampler(int(os.environ.get("LOCAL_RANK", "0"))) as clk:
        ev0.record(stream)
        for _ in range(args.steps):
            out_res.append(step())
        ev1.record(stream)
        torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    res, ts = out_res[-1]
    dp_ms = sum(r["dp_kernel_ms"] for r, _ in out_res)
    dp_launches = sum(r["dp_kernel_launches"] for r, _ in out_res)
    out = {"metric": "ECASQ %s solve: solves/s" % args.mode, "value": args.steps / (ms / 1000.0),
           "unit": "solves/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": ms / args.steps, "higher_is_better": True, "vs_baseline": None,
           "dtype": "f64" if args.mode == "grid" else "f32 (fp64 exact stage)", "data": "synthetic",
           "config": {"workload": args.config, "mode": args.mode, "d": d, "s": s, "budget_bits": budget,
                      "grid": args.grid if args.mode == "grid" else None,
                      "cost_mode": cost_mode_name(E, flags)},
           "solve": {"m": res["m"], "p": res["p"], "lambda": res["lambda"], "vnmse": res["vnmse"],
                     "h_surrogate": res["h_surrogate"], "h_exact": res["h_exact"], "passes": res["passes"],
                     "candidates_per_solve": res["candidates"], "dp_ms_per_solve": dp_ms / args.steps,
                     "dp_launches_per_solve": dp_launches / args.steps},
           "timeshare": ts or None, "gpu_launches": E.ecasq_kernel_launches() - launches0,
           "clocks": clk.summary()}
    print(json.dumps(out), flush=True)


def run_hbm_mode(args):
    """Encode (4 B read + 1 B written per entry) and preparation (four 8-bit LSD radix
    passes, 8 B per entry each, then the histogram and prefix sums) on seeded normal
    vectors generated on the device.  Each call synchronises its stream, so the CUDA-event
    time of a call includes the host's part of it: the GB/s are lower bounds."""
    import torch
    import paper_2608_18147_gb300 as E
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {"hbm_gbs": 6800.0}
    gen = torch.Generator(device="cuda").manual_seed(0)
    out = {"metric": "ECASQ HBM-bound rows: GB/s of algorithmic traffic", "unit": "GB/s", "n_gpus": 1,
           "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "vs_baseline": None,
           "data": "synthetic (seeded normal, generated on the device)", "dtype": "f32 in, u8 out"}
    stream = torch.cuda.current_stream()

    def timed(fn):
        for _ in range(args.warmup):
            fn()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ts = []
        for _ in range(args.steps):
            torch.cuda.synchronize()
            ev0.record(stream)
            fn()
            ev1.record(stream)
            torch.cuda.synchronize()
            ts.append(ev0.elapsed_time(ev1))
        return statistics.median(ts)

    d = 1 << 28
    x = torch.randn(d, generator=gen, device="cuda", dtype=torch.float32)
    Q = torch.quantile(x[: 1 << 20], torch.linspace(0, 1, 16, device="cuda")).contiguous()
    Q[0], Q[-1] = x.min(), x.max()
    Q = torch.unique(Q)
    idx = torch.empty(d, dtype=torch.uint8, device="cuda")
    counts = torch.empty(Q.numel(), dtype=torch.int32, device="cuda")
    qws = torch.empty(256, dtype=torch.uint8, device="cuda")
    ms_q = timed(lambda: E.ecasq_quantize(x, Q, seed=1, ws=qws, idx=idx, counts=counts))
    gbs_q = 5.0 * d / (ms_q / 1000.0) / 1e9
    ms_t = timed(lambda: E.ecasq_quantize_timeshare(x, Q, Q, 0.5, 1, 2, ws=qws))
    gbs_t = 6.0 * d / (ms_t / 1000.0) / 1e9
    del x, idx
    torch.cuda.empty_cache()
    d2 = 1 << 26
    x2 = torch.randn(d2, generator=gen, device="cuda", dtype=torch.float32)
    ws2 = torch.empty(int(E.lib().ecasq_workspace_size_prep(d2)), dtype=torch.uint8, device="cuda")
    ms_p = timed(lambda: E.ecasq_prepare(x2, ws=ws2))
    gbs_p = 32.0 * d2 / (ms_p / 1000.0) / 1e9
    peak = peaks["hbm_gbs"]
    out.update(value=gbs_q, ms_per_step=ms_q,
               config={"workload": "normal, 2^28 entries (encode), 2^26 (prepare)", "mode": "hbm",
                       "codebook": int(Q.numel()), "l2": "vectors of 1 GiB and 256 MiB, far above the 129 MB L2"},
               roofline={"bound": "hbm", "achieved": gbs_q, "peak": peak, "unit": "GB/s", "frac": gbs_q / peak,
                         "traffic": None, "kernel": "k_quantize_short", "peak_basis": "MEASURED_PEAKS.json hbm_gbs"},
               rows={"encode": {"ms": ms_q, "bytes_per_entry": 5, "GBs": gbs_q, "frac": gbs_q / peak},
                     "encode_timeshare": {"ms": ms_t, "bytes_per_entry": 6, "GBs": gbs_t, "frac": gbs_t / peak},
                     "prepare": {"ms": ms_p, "bytes_per_entry": 32, "GBs": gbs_p, "frac": gbs_p / peak,
                                 "basis": "4 LSD radix passes x (4 B read + 4 B written); the histogram, "
                                          "prefix sums and count passes are extra"}})
    print(json.dumps(out), flush=True)


def _timed_steps(args, step):
    """CUDA-event time (ms) of args.steps calls of step() after args.warmup untimed ones,
    with the clocks sampled meanwhile."""
    import torch
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    outs = []
    with ClockSampler(int(os.environ.get("LOCAL_RANK", "0"))) as clk:
        ev0.record(stream)
        for _ in range(args.steps):
            outs.append(step())
        ev1.record(stream)
        torch.cuda.synchronize()
    return ev0.elapsed_time(ev1), outs, clk.summary()


def run_rows_mode(args):
    """Batched budgeted solves of the KV-cache-like rows (8192 x 128, s = 8, b = 3):
    rows per second, inputs in HBM."""
    import torch
    import paper_2608_18147_gb300 as E
    from paper_2608_18147_gb300 import workloads
    name = "kvrows_8192x128_s8"
    cfg = workloads.CONFIGS[name]
    X = torch.as_tensor(workloads.make(name)).cuda()
    rows, d = X.shape
    s, budget = cfg["s"], cfg["budgets"][0]
    ws = E.workspace(d, s, rows)
    launches0 = E.ecasq_kernel_launches()
    ms, outs, clocks = _timed_steps(args, lambda: E.ecasq_solve_batched(X, s, budget_bits=budget, ws=ws))
    Q, m, res = outs[-1]
    ok = int((res.field("status") == 0).sum())
    # candidates of eq. apx_rec over all rows and their evaluated multipliers, against the
    # same FP32 issue peak as the single-vector kernel (2 ops per candidate), over the whole
    # step (host search logic and copies included, so a lower bound for the kernel)
    cand = sum(int(l) * candidates_per_multiplier(int(pr), s)
               for pr, l in zip(res.field("p"), res.field("lambdas_evaluated")))
    sm_count = torch.cuda.get_device_properties(0).multi_processor_count
    peak = sm_count * 128 * 2.07e9 / 1e12
    achieved = 2.0 * cand / (ms / args.steps / 1000.0) / 1e12
    out = {"metric": "ECASQ batched solve: rows/s", "value": args.steps * rows / (ms / 1000.0), "unit": "rows/s",
           "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
           "higher_is_better": True, "vs_baseline": None, "dtype": "f32 (fp64 where a decision is ambiguous)",
           "data": "synthetic", "config": {"workload": name, "mode": "rows", "rows": rows, "d": d, "s": s, "budget_bits": budget},
           "rows_ok": ok, "mean_m": float(m.float().mean().item()),
           "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TOP/s", "frac": achieved / peak,
                        "traffic": None, "kernel": "k_rows_pass",
                        "candidates_per_step": cand,
                        "note": "2 ops per candidate of eq. apx_rec over the whole step; the first search round "
                                "builds each row's fp32 pair costs, every round runs three 8-warp blocks an SM (shared "
                                "memory per row); about half of the step is the host's search"},
           "gpu_launches": E.ecasq_kernel_launches() - launches0, "clocks": clocks}
    print(json.dumps(out), flush=True)


def run_pass_mode(args, cfg, x_np):
    """One DP pass of the configuration's vector at the --lambdas multipliers (resident
    interval costs when they fit in 60 % of the free memory, else costs rebuilt in every pass)."""
    import torch
    import paper_2608_18147_gb300 as E
    s = cfg["s"]
    lams = [float(t) for t in args.lambdas.split(",")]
    if args.prefix > 0:
        x_np = x_np[:args.prefix]
    x = torch.as_tensor(x_np).cuda()
    d = x.numel()
    flags = cost_mode_flags(E, d, s, torch.cuda.mem_get_info()[0])
    ws = E.workspace(d, s, flags=flags)
    launches0 = E.ecasq_kernel_launches()
    ms, outs, clocks = _timed_steps(args, lambda: E.ecasq_dp_pass(x, s, lams, flags=flags, ws=ws))
    st = E.native.ws_status(ws)
    p = st["p"]
    cand = len(lams) * candidates_per_multiplier(p, s)
    out = {"metric": "ECASQ DP pass: candidate evals/s", "value": args.steps * cand / (ms / 1000.0),
           "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
           "higher_is_better": True, "vs_baseline": None, "dtype": "f32 (fp64 exact stage)", "data": "synthetic",
           "config": {"workload": args.config + (" (first %d entries)" % d if args.prefix > 0 else ""),
                      "mode": "pass", "d": d, "p": p, "s": s, "lambdas": lams,
                      "cost_mode": cost_mode_name(E, flags)},
           "status": {"timeout": st["timeout"], "bound_viol": st["bound_viol"], "rescored": st["rescored"],
                      "tile_units_run": st["tiles_run"], "tile_units_skipped": st["tiles_skipped"],
                      "cost_tiles_fetched": st["tiles_fetched"], "band_members": st["members"],
                      "big_bands": st["big_bands"], "wide_bands": st["overflow"],
                      "executed_candidates": executed_candidates(st, p, s, len(lams))},
           "m": list(outs[-1][1]), "gpu_launches": E.ecasq_kernel_launches() - launches0, "clocks": clocks}
    print(json.dumps(out), flush=True)


def run_linear_mode(args, cfg, x_np):
    """The linear-space traceback (Sec. 5, last paragraph) of the configuration's vector (or
    its first --prefix entries) at the first multiplier of --lambdas: ms per call.  The
    throughput unit is the forward recurrence's candidate count (the splits' forward and
    backward passes roughly double the work)."""
    import torch
    import paper_2608_18147_gb300 as E
    s = cfg["s"]
    lam = float(args.lambdas.split(",")[0])
    if args.prefix > 0:
        x_np = x_np[:args.prefix]
    x = torch.as_tensor(x_np).cuda()
    d = x.numel()
    ws = torch.empty(int(E.lib().ecasq_workspace_size_linear(d)), dtype=torch.uint8, device="cuda")
    launches0 = E.ecasq_kernel_launches()
    ms, outs, clocks = _timed_steps(args, lambda: E.ecasq_dp_linear(x, s, lam, ws=ws))
    Q, met = outs[-1]
    p = E.native.ws_status(ws)["p"]
    cand = candidates_per_multiplier(p, s)
    out = {"metric": "ECASQ linear-space traceback: candidate evals/s of the forward recurrence", "unit": UNIT,
           "value": args.steps * cand / (ms / 1000.0), "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": ms / args.steps, "higher_is_better": True, "vs_baseline": None,
           "dtype": "f64", "data": "synthetic",
           "config": {"workload": args.config + (" (first %d entries)" % d if args.prefix > 0 else ""),
                      "mode": "linear", "d": d, "p": p, "s": s, "lambda": lam,
                      "workspace_mb": round(ws.numel() / 2 ** 20, 2)},
           "m": int(Q.numel()), "objective": float(met[0]),
           "gpu_launches": E.ecasq_kernel_launches() - launches0, "clocks": clocks}
    print(json.dumps(out), flush=True)


def opt_candidates(n, s, G, nL=1):
    """Candidates of the optimal DP's layers 3..s (Sec. 4): for each l, the finite
    predecessors k (k < nL at i = 3, i - 3 <= k < l above) times the outputs j > l, x G."""
    import numpy as np
    l = np.arange(n - 1, dtype=np.int64)
    c = 0
    for i in range(3, s + 1):
        nk = np.minimum(nL, l) if i == 3 else np.maximum(l - (i - 3), 0)
        c += int(np.sum(nk * (n - 1 - l)))
    return c * G


def run_opt_mode(args, cfg, x_np):
    import numpy as np
    import torch
    import paper_2608_18147_gb300 as E
    s = cfg["s"]
    d = x_np.size
    g = E.uniform_grid(x_np, args.grid)
    n = g.size
    lams = [0.0] + list(np.geomspace(1e-6, 1e2, 7))
    x = torch.as_tensor(x_np).cuda()
    gd = torch.as_tensor(g).cuda()
    ws = torch.empty(int(E.lib().ecasq_workspace_size_opt(d, n, s, len(lams))), dtype=torch.uint8, device="cuda")
    for _ in range(args.warmup):
        E.ecasq_opt_dp(x, s, lams, P=gd, ws=ws)
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    launches0 = E.ecasq_kernel_launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(int(os.environ.get("LOCAL_RANK", "0"))) as clk:
        ev0.record(stream)
        for _ in range(args.steps):
            Q, m, met = E.ecasq_opt_dp(x, s, lams, P=gd, ws=ws)
        ev1.record(stream)
        torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1) / args.steps
    cand = opt_candidates(n, s, len(lams))
    out = {"metric": "ECASQ optimal DP pass (Sec. 4): candidate evals/s", "value": cand / (ms / 1000.0),
           "unit": "candidate evals/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
           "ms_per_step": ms, "higher_is_better": True, "vs_baseline": None,
           "dtype": "f32 (fp64 band re-scoring)", "data": "synthetic",
           "config": {"workload": args.config, "mode": "opt", "d": d, "s": s, "grid": n, "multipliers": len(lams)},
           "pass": {"candidates": cand, "m": list(m), "optimum": met[:, 0].tolist(), "vnmse": (met[:, 1] / float(
               np.sum(x_np.astype(np.float64) ** 2))).tolist()},
           "gpu_launches": E.ecasq_kernel_launches() - launches0, "clocks": clk.summary()}
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    from paper_2608_18147_gb300 import workloads
    cfg = workloads.CONFIGS[args.config]
    x_np = workloads.make(args.config, 0)
    if args.impl == "reference":
        run_reference(args, cfg, x_np)
        return

    import numpy as np
    import torch
    import paper_2608_18147_gb300 as E
    if args.mode != "solve":
        run_other_mode(args, cfg, x_np)
        return

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    s, budget = cfg["s"], cfg["budgets"][0]
    # the stop rule of Sec. 6 (a round lowering J by at most refine_tol relative) ends the
    # refinement; the cap is only a safeguard (Student-t d = 2^17 stops after about 90 rounds)
    refine_rounds = 500 if cfg.get("refine") else 0
    refine_tol = cfg.get("refine_tol", 0.0)
    d = x_np.size
    x = torch.as_tensor(x_np).cuda()
    # resident interval costs when they fit in 60% of the free device memory
    flags = E.TIME_KERNELS
    flags |= cost_mode_flags(E, d, s, torch.cuda.mem_get_info()[0])
    ws = E.workspace(d, s, flags=flags)
    idx = torch.empty(d, dtype=torch.uint8, device="cuda")
    counts = torch.empty(s, dtype=torch.int32, device="cuda")
    qws = torch.empty(256, dtype=torch.uint8, device="cuda")

    def step(xin):
        Q, res = E.ecasq_solve(xin, s, budget_bits=budget, ws=ws, refine_max_rounds=refine_rounds,
                               refine_rel_tol=refine_tol, flags=flags)
        _, _, he = E.ecasq_quantize(xin, Q, seed=12345, ws=qws, idx=idx, counts=counts[:Q.numel()])
        return Q, res, he

    for _ in range(args.warmup):
        Q, res, he = step(x)
    barrier()
    stream = torch.cuda.current_stream()
    launches0 = E.ecasq_kernel_launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    results = []
    with ClockSampler(local) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            Q, res, he = step(x)
            results.append(res)
        ev1.record(stream)
        barrier()
    launches = E.ecasq_kernel_launches() - launches0
    ms = max_over_ranks(ev0.elapsed_time(ev1), dist, "cuda")
    cand_step = statistics.mean(r["candidates"] for r in results)
    value = whole_job_rate(world, args.steps * cand_step, ms)
    dp_ms = sum(r["dp_kernel_ms"] for r in results)
    dp_launches = sum(r["dp_kernel_launches"] for r in results)
    cand_total = sum(r["candidates"] for r in results)
    clocks = clk.summary()
    st = E.native.ws_status(ws)  # counters of the last solve
    last_p = results[-1]["p"]
    units = st["tiles_run"] + st["tiles_skipped"]
    run_frac = st["tiles_run"] / units if units else 1.0

    # roofline of the min-plus kernel against the FP32/ALU issue peak.  `achieved` counts
    # the candidates the kernel executed (the tile units it ran and its diagonal blocks),
    # not the algorithmic ones: the exact tile skip leaves most of eq. apx_rec unevaluated,
    # and the algorithmic rate is reported beside it as `effective`.
    last = results[-1]
    n_sm = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    peak = n_sm * FP32_LANES * SM_MAX_MHZ * 1e6 / 1e12
    last_launches = max(last["dp_kernel_launches"], 1)
    last_ms = last["dp_kernel_ms"]
    executed = executed_candidates(st, last_p, s, last["lambdas_evaluated"])
    achieved = OPS_PER_CANDIDATE * executed / (last_ms / 1000.0) / 1e12 if last_ms > 0 else None
    effective = OPS_PER_CANDIDATE * cand_total / (dp_ms / 1000.0) / 1e12 if dp_ms > 0 else None
    fetched_per_launch = st["tiles_fetched"] / last_launches
    traffic = (TRAFFIC_PER_FETCHED_TILE * fetched_per_launch
               if (flags & E.RESIDENT_COSTS) and TRAFFIC_PER_FETCHED_TILE else None)
    roofline = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TOP/s",
                "frac": (achieved / peak) if achieved else None, "traffic": traffic,
                "traffic_note": "bytes copied per launch, from HBM or L2 (an upper bound of its DRAM reads): the bytes of a "
                                "cost tile times the tiles this launch fetched",
                "tiles_fetched_per_launch": fetched_per_launch,
                "kernel": "k_wavefront",
                "peak_basis": "%d SMs (device attribute) x 128 FP32-pipe lanes (adds and mins share the issue "
                              "slots) x 2070 MHz max clock; of the 2-op count below" % n_sm,
                "avg_launch_ms": dp_ms / max(dp_launches, 1), "launches": dp_launches,
                "ops_basis": "executed: 2 ops (add, min) per candidate the kernel evaluated -- %d-column x %d-k "
                             "tile units it ran, times the s-2 layers, plus its diagonal blocks; "
                             "the FMA of C + lambda' Phi, which the far phase repeats per candidate, "
                             "is not counted" % (BJ, BK),
                "executed_candidates_per_launch": executed / last_launches,
                "effective": effective,
                "effective_frac": (effective / peak) if effective else None,
                "effective_note": "algorithmic rate: 2 ops for every candidate of eq. apx_rec (all layers, "
                                  "multipliers, k < j), including the ones the exact tile skip never evaluates",
                "executed_unit_frac": run_frac,
                "executed_note": "off-diagonal (multiplier, tile) units of s-2 layer tasks evaluated; the other tasks were "
                                 "skipped by an exact lower bound that proves they cannot change any minimum or band"}
    if achieved and clocks.get("sm_mhz"):
        roofline["frac_at_measured_clock"] = achieved / (n_sm * FP32_LANES * clocks["sm_mhz"] * 1e6 / 1e12)

    e2e = None
    if not args.no_e2e:
        x_host = torch.as_tensor(x_np).pin_memory()
        idx_host = torch.empty(d, dtype=torch.uint8).pin_memory()
        xdev = torch.empty_like(x)
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        cand_e = 0
        for _ in range(args.steps):
            xdev.copy_(x_host, non_blocking=True)
            Q, res, he = step(xdev)
            idx_host.copy_(idx, non_blocking=True)
            qh = Q.cpu()
            cand_e += res["candidates"]
        e1.record(stream)
        barrier()
        ms_e = max_over_ranks(e0.elapsed_time(e1), dist, "cuda")
        e2e = {"value": whole_job_rate(world, cand_e, ms_e), "unit": UNIT, "h2d_bytes_per_step": 4 * d,
               "d2h_bytes_per_step": d + 4 * int(qh.numel()), "ms_per_step": ms_e / args.steps}

    cb = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cb = cpu_baseline(x_np, cfg)

    if rank == 0:
        last = results[-1]
        out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
               "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
               "scaling": "weak", "vs_baseline": None, "dtype": "f32 (fp64 exact stage)", "data": "synthetic",
               "config": {"workload": args.config, "d": d, "s": s, "budget_bits": budget,
                          "refine": {"max_rounds": refine_rounds, "rel_tol": refine_tol},
                          "cost_mode": cost_mode_name(E, flags),
                          "workspace_gb": round(ws.numel() / 1e9, 2),
                          "l2": "working set larger than the 129 MB L2 (DP tables ~0.9 GB; resident costs "
                                "streamed once per pass); no flush",
                          "parallelism": "replicas" if world > 1 else "single GPU"},
               "solve": {"m": last["m"], "lambda": last["lambda"], "vnmse": last["vnmse"],
                         "h_surrogate": last["h_surrogate"], "h_exact": last["h_exact"],
                         "passes": last["passes"], "lambdas_evaluated": last["lambdas_evaluated"],
                         "refine_rounds": last["refine_rounds"], "refine_last_rel": last["refine_last_rel"],
                         "refine_stopped_by_rule": last["refine_rounds"] < refine_rounds,
                         "candidates_per_solve": last["candidates"],
                         "rescored_per_solve": last["rescored"], "dp_pass_ms": dp_ms / max(dp_launches, 1),
                         "tile_units_run": st["tiles_run"], "tile_units_skipped": st["tiles_skipped"],
                         "cost_tiles_fetched": st["tiles_fetched"],
                         "solves_per_s": world * args.steps / (ms / 1000.0)},
               "roofline": roofline, "cpu_baseline": cb, "e2e": e2e, "gpu_launches": launches,
               "clocks": clocks}
        print(json.dumps(out), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
