"""Benchmark: u-series energy + forces + potentials on the membrane-shaped slab.

One step = one evaluation of the 63,996-charge membrane slab (80 x 80 x 100 A,
64 x 64 x 80 grid, C1 b = 2 series) at every cutoff of the sweep
r_c = 8, 9, 10, 11, 12, 13 A, inputs resident in HBM.  value = atom-evals/s
(charges x evaluations / second; device time from CUDA events on the
evaluation stream; L2 flushed between steps by writing a 512 MB buffer).
e2e = the same metric through the host-buffer entry point (pinned host
buffers, copies and the synchronisation inside the timed region, L2 flushed
before every step, CUDA events around each step).

The timed form is the one chosen for the benchmark's accuracy bound (rms
relative force error <= 1e-4): per-axis convolutions as BF16x3 tensor-core
GEMMs, spreading with the paper's GSE-style parameters (sigma_s = 0.83 h, an
8-point stencil).  Its error against the FP64 oracle is measured in the same
run at r_c = 8, 10 and 13 A, and two plain FP32 forms are timed beside it: FP32
CUDA-core convolutions with the same spreading, and the tight FP32 form
(12-point stencil, sigma_s = h) used for the 1e-5 parity tests.  The
1,064,799-charge water box (r_c = 10 A, 176^3 grid) is timed in four forms as
well, and the serving stream of 512 independent systems.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference] [--serve-systems M] [--no-scale]

N > 1 (under torch.distributed.run): every rank evaluates its own replica of
the workload (independent systems, no collective), value sums all ranks over
the slowest rank's time.  --impl reference times the FP64 oracle on the host
cores instead (the reference arm): one full evaluation of the slab per step,
the same definition as the cpu_baseline of the GPU arm.
"""
from __future__ import annotations

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

METRIC = "u-series E+F atom-evals/s at rms rel force err ≤1e-4; serving p50/p99 ms"
UNIT = "atom-evals/s"
WORKLOAD = "membrane_slab"
SWEEP = (8.0, 9.0, 10.0, 11.0, 12.0, 13.0)
# kernels of one evaluation: bin_count, scan, place, cluster_build, near, spread, conv x, conv y, conv z, gather,
# combine
KERNELS_PER_EVAL = 11
FP32_PEAK_DERIVED_TFLOPS = 152 * 128 * 2 * 2.070e9 / 1e12   # SMs x FP32 lanes x 2 (FMA) x max SM clock
# algorithmic flops of one unordered pair inside r_c, the unit of the pair kernel's roofline: the midpoint of
# 30-50 flops for the arithmetic any pair kernel of Eq. 20 needs (the displacement and r^2, 1/r, F(r) and its
# derivative, the force on both atoms and both potentials), independent of how this kernel evaluates F
NEAR_FLOPS_PER_PAIR = 40
# DRAM bytes (read + write) per launch of the pair kernel over this sweep, averaged over its six launches (one
# per cutoff) in one ncu capture of `bench.py --steps 1 --warmup 3 --serve-systems 0 --no-scale`; None whenever
# the pair kernel has changed since that capture
NEAR_TRAFFIC_BYTES = None
# forms: (name, conv, spread_points, spread_sigma_over_h)
CHOSEN = ("bf16x3_gse8", 2, 8, 0.83)
COMPARATORS = (("fp32_gse8", 0, 8, 0.83), ("fp32_tight12", 0, 12, 1.0))


def measured_peaks():
    """HBM GB/s and dense BF16 TFLOP/s measured on this machine's GPUs (MEASURED_PEAKS.json), else the
    fallback figures of an earlier GB300 measurement."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            m = json.load(f)
        return {"hbm_gbs": float(m["hbm_gbs"]), "bf16_tflops": float(m["bf16_tflops"]), "source": "measured"}
    except (OSError, KeyError, ValueError):
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "source": "fallback"}


def stage_floors(n, pairs, info, grid, spread_points, hilo_products, peaks):
    """Lower bounds (ms) of one evaluation's stages from their algorithmic work and the peaks:
    bin 60 B/atom of HBM (positions in, cell ids, permutation, sorted and paired copies);
    near pairs x flops/pair at the FP32 peak; spread 2 P^3 and gather 8 P^3 flops per atom at the
    FP32 peak (one FMA per stencil point; value and three gradient components); conv the larger of
    its tensor flops (hilo_products x 2 N G n_axis per pass) at the BF16 peak and its grid bytes at the
    HBM peak (4 G in and 4 N G out on x, 4 N G both ways on y, 4 N G in and 4 G out on z)."""
    G = grid[0] * grid[1] * grid[2]
    N = info.n_terms
    fp32 = peaks["fp32_tflops"] * 1e12
    hbm = peaks["hbm_gbs"] * 1e9
    tc = peaks["bf16_tflops"] * 1e12
    f = {"bin": 60.0 * n / hbm,
         "near": pairs * NEAR_FLOPS_PER_PAIR / fp32,
         "spread": 2.0 * spread_points ** 3 * n / fp32,
         "gather": 8.0 * spread_points ** 3 * n / fp32}
    byts = {"conv_x": 4.0 * G + 4.0 * N * G, "conv_y": 8.0 * N * G, "conv_z": 4.0 * N * G + 4.0 * G}
    for ax, nx in zip(("conv_x", "conv_y", "conv_z"), grid):
        f[ax] = max(hilo_products * 2.0 * N * G * nx / tc, byts[ax] / hbm)
    return {k: 1e3 * v for k, v in f.items()}


def near_flops_per_pair(poly_degree: int, n_explicit: int) -> int:
    """The pair kernel's own arithmetic for one pair inside r_c, counted once per unordered pair (FMA = 2):
    displacement 3, r^2 5, rsqrt + Newton step 5, polynomial argument 2, Horner value and
    derivative 4 D, derivative scale 1, 1/r^3 2, force scale 3, forces on both atoms 12,
    potentials of both atoms 5; each explicit Gaussian adds exp (counted 8) + 5."""
    return 38 + 4 * poly_degree + 13 * n_explicit


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(x: float, device=None) -> float:
    """The largest value of x over all ranks (the slowest rank's time); x itself at world size 1.
    Works with any initialised torch.distributed backend (NCCL on GPUs, gloo on CPUs)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank: float, world_size: int, seconds_max: float) -> float:
    """Weak scaling: every rank processes units_per_rank; the job takes as long as its slowest rank."""
    return units_per_rank * world_size / seconds_max


class ClockSampler:
    """nvidia-smi clock/throttle samples (every 200 ms) while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, power, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
                power.append(float(parts[3]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "power_w_max": max(power) if power else None,
                "samples": len(sm),
                "reasons": sorted(reasons)}


def cpu_oracle_eval(w, r_c, targets=None):
    import oracle as O
    from tests.golden import paper_tables
    return O.evaluate(O.Series(*paper_tables()["table2_C1"]), r_c, w.box, w.xyzq[:, :3], w.xyzq[:, 3],
                      targets=targets)


def run_reference(args):
    """Reference arm: the FP64 oracle on the host cores, one full evaluation (energy, every force and
    potential) of the slab per step, the cutoff cycling through the sweep."""
    ws, rank, _ = _dist()
    if rank != 0:
        return
    import oracle as O
    from paper_1911_01377_gb300 import workloads as W
    w = W.get(WORKLOAD)
    times = []
    for step in range(args.warmup + args.steps):
        r_c = SWEEP[step % len(SWEEP)]
        t0 = time.perf_counter()
        cpu_oracle_eval(w, r_c)
        dt = time.perf_counter() - t0
        if step >= args.warmup:
            times.append(dt)
    total = sum(times)
    value = w.n * len(times) / total
    sample = (f"one full FP64 oracle evaluation (direct near sum + exact k-space far sum; energy, all forces and "
              f"potentials) of the {w.n}-charge slab per step, r_c cycling {SWEEP[0]:g}-{SWEEP[-1]:g} A")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / len(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": f"{WORKLOAD}: {w.n} charges, 80x80x100 A, r_c 8-13 A"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def _time_form(usr, torch, w, x, form, steps, warmup, flush, stream, cutoffs=SWEEP, stage_steps=3):
    """Device-time `steps` sweeps of one form with events around the pair kernel only (profiling level 2,
    so its launch duration is measured inside the timed region); then `stage_steps` more sweeps with every
    stage boundary recorded, outside the timed region, for the stage breakdown.  Returns (total ms, per-stage
    ms means, pair-kernel ms sums of the timed steps, contexts, outs, ens)."""
    name, conv, P, ratio = form[:4]
    extra = form[4] if len(form) > 4 else {}
    ctxs = [usr.USeries(w.box, w.grid, r_c, "C1_B2", max_atoms=w.n, conv=conv, spread_points=P,
                        spread_sigma_over_h=ratio, **extra) for r_c in cutoffs]
    outs = [torch.empty((w.n, 4), dtype=torch.float32, device=x.device) for _ in cutoffs]
    ens = [torch.empty(4, dtype=torch.float64, device=x.device) for _ in cutoffs]

    def step():
        for c, o, e in zip(ctxs, outs, ens):
            usr.usr_eval(c.ctx, w.n, x.data_ptr(), o.data_ptr(), e.data_ptr(), stream)

    for _ in range(warmup):
        flush.fill_(1.0)
        step()
    torch.cuda.synchronize()
    for c in ctxs:
        st = usr.usr_last_device_status(c.ctx)
        if st != 0:
            raise usr.UsrError(st, f"device status after warm-up ({name})")
        usr.usr_set_profiling(c.ctx, 2)
    near = [0.0 for _ in cutoffs]
    total = 0.0
    for k in range(steps):
        flush.fill_(float(k % 7))
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        e1.synchronize()
        total += e0.elapsed_time(e1)
        for i, c in enumerate(ctxs):
            near[i] += usr.usr_stage_times(c.ctx)[1]
    stage = [[0.0] * usr.USR_NSTAGES for _ in cutoffs]
    for c in ctxs:
        usr.usr_set_profiling(c.ctx, 1)
    for k in range(stage_steps):
        flush.fill_(float(k % 7))
        step()
        torch.cuda.synchronize()
        for i, c in enumerate(ctxs):
            for s_, v in enumerate(usr.usr_stage_times(c.ctx)):
                stage[i][s_] += v / stage_steps
    for c in ctxs:
        usr.usr_set_profiling(c.ctx, 0)
    return total, stage, near, ctxs, outs, ens


SCALE_FORMS = (CHOSEN, ("bf16x3_gse8_multilevel", 2, 8, 0.83, {"multilevel": 1}), ("tf32x3_gse8", 1, 8, 0.83),
               COMPARATORS[0], COMPARATORS[1])


def run_scale(usr, torch, steps, warmup, flush, stream):
    """Precision forms at scale: 354,933 waters (1,064,799 charges), L = 220 A, r_c = 10 A,
    176^3 grid; one evaluation per step per form, inputs resident, L2 flushed between steps.
    The errors of these forms against the FP64 oracle are checked by the scale parity tests."""
    from paper_1911_01377_gb300 import workloads as W
    w = W.get("water_1m")
    x = torch.from_numpy(w.xyzq).to(flush.device)
    forms = {}
    for form in SCALE_FORMS:
        tms, stage, _, cc, _, _ = _time_form(usr, torch, w, x, form, steps, warmup, flush, stream, cutoffs=(10.0,))
        forms[form[0]] = {"value": w.n * steps / (tms / 1e3), "unit": UNIT, "ms_per_eval": tms / steps,
                          "stage_ms": dict(zip(usr.STAGES, stage[0]))}
        for c in cc:
            c.close()
    return {"workload": f"water_1m: {w.n} charges (354933 3-site waters), cubic L=220 A, 176^3 grid, "
                        f"C1 b=2, r_c=10 A", "forms": forms}


def run_serving(usr, torch, count, seed=1911, slots=12, budget_gib=64.0, rate_frac=0.7):
    """Serving form: a stream of `count` independent water boxes (charges log-uniform in
    [2,000, 200,000], 0.1 per A^3, r_c = 9 A, ~1 A grids) through the continuous-batching
    server (the serving form: TF32x3, 10-point spreading), first all at once (capacity), then with Poisson arrivals at
    rate_frac x capacity (latency); and one system at a time with the plain FP32 form."""
    import numpy as np
    from paper_1911_01377_gb300 import workloads as W
    systems = list(W.serving_stream(seed, count))
    n_atoms = sum(s[3].shape[0] for s in systems)
    xs = [torch.from_numpy(s[3]).pin_memory() for s in systems]
    outs = [torch.empty((s[3].shape[0], 4), dtype=torch.float32).pin_memory() for s in systems]
    ens = [torch.empty(4, dtype=torch.float64).pin_memory() for _ in systems]
    form = W.SERVING_FORM
    params = [usr.make_params(b, g, rc, "C1_B2", max_atoms=x.shape[0], **form) for (b, g, rc, x) in systems]

    def serve(arrivals):
        srv = usr.Server(hbm_budget_bytes=budget_gib * (1 << 30), slots=slots)
        # warm every slot once with the largest system (allocations happen here, not in the timed run)
        big = int(np.argmax([x.shape[0] for x in xs]))
        for _ in range(slots):
            srv.submit(params[big], xs[big], outs[big], ens[big])
        srv.wait(600)
        srv.poll(4 * slots)
        t0 = time.perf_counter()
        for k in range(len(systems)):
            if arrivals is not None:
                while time.perf_counter() - t0 < arrivals[k]:
                    pass
            srv.submit(params[k], xs[k], outs[k], ens[k])
        srv.wait(600)
        wall = time.perf_counter() - t0
        res = srv.poll(len(systems) + 8)
        srv.close()
        lat = np.array([r[1] for r in res])
        bad = [r for r in res if r[2] != 0]
        return wall, lat, bad

    # capacity: the median of three all-at-once passes (each about 0.1 s of host wall clock)
    walls = []
    for _ in range(3):
        wall_k, lat_all, bad = serve(None)
        if bad:
            raise RuntimeError(f"serving failures: {bad[:3]}")
        walls.append(wall_k)
    wall = float(np.median(walls))
    capacity = n_atoms / wall
    rate = rate_frac * len(systems) / wall                 # requests per second
    rng = np.random.default_rng(seed + 1)
    arrivals = np.cumsum(rng.exponential(1.0 / rate, size=len(systems)))
    wall_p, lat, bad = serve(arrivals)
    if bad:
        raise RuntimeError(f"serving failures: {bad[:3]}")
    # one at a time (one context reconfigured per system, synchronous host-buffer calls), in the plain FP32
    # form and in the served form itself, so that the gain of batching alone is visible
    def one_at_a_time(**kw):
        big = int(np.argmax([x.shape[0] for x in xs]))
        c = usr.USeries(systems[big][0], systems[big][1], systems[big][2], "C1_B2", max_atoms=xs[big].shape[0],
                        **kw)
        c.eval_host(xs[big], outs[big], ens[big])
        t0 = time.perf_counter()
        for (b, g, rc, _), x, o, e in zip(systems, xs, outs, ens):
            c.reconfigure(b, g, rc, "C1_B2", max_atoms=x.shape[0], **kw)
            c.eval_host(x, o, e)
        t = time.perf_counter() - t0
        c.close()
        return t

    t_one = one_at_a_time()
    t_same = one_at_a_time(**form)
    return {"systems": len(systems), "charges": n_atoms, "slots": slots, "hbm_budget_gib": budget_gib,
            "form": "tf32x3_gse{spread_points}_w{spread_sigma_over_h:g}".format(**form),
            "capacity_atom_evals_per_s": capacity, "all_at_once_wall_s": wall,
            "all_at_once_passes_wall_s": walls,
            "poisson_rate_per_s": rate, "poisson_wall_s": wall_p,
            "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
            "throughput_atom_evals_per_s": n_atoms / wall_p,
            "one_at_a_time_fp32_atom_evals_per_s": n_atoms / t_one,
            "one_at_a_time_same_form_atom_evals_per_s": n_atoms / t_same,
            "speedup_vs_one_at_a_time_fp32": (n_atoms / wall) / (n_atoms / t_one),
            "speedup_vs_one_at_a_time_same_form": (n_atoms / wall) / (n_atoms / t_same),
            "latency": "submit to results in pinned host memory, host clock"}


def run_gpu(args):
    import numpy as np
    import torch

    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    from paper_1911_01377_gb300 import build as B
    B.build()
    import oracle as O
    from paper_1911_01377_gb300 import usr
    from paper_1911_01377_gb300 import workloads as W

    w = W.get(WORKLOAD)
    n = w.n
    x = torch.from_numpy(w.xyzq).to(dev)
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    # unordered pairs inside r_c per cutoff (pair-count pass, outside the timed region)
    pairs = []
    for r_c in SWEEP:
        c = usr.USeries(w.box, w.grid, r_c, "C1_B2", max_atoms=n)
        cnt, _ = c.debug_pairs(x)
        pairs.append(int(cnt.sum().item()) // 2)
        c.close()

    # the chosen form, timed with clocks sampled
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    ids = [v.strip() for v in vis.split(",") if v.strip()]
    sampler = ClockSampler(ids[local] if local < len(ids) else str(local))
    sampler.start()
    time.sleep(0.3)
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    t_wall0 = time.perf_counter()
    total_ms, stage_ms, near_ms, ctxs, outs, ens = _time_form(usr, torch, w, x, CHOSEN, args.steps, args.warmup,
                                                               flush, stream)
    torch.cuda.synchronize()
    t_wall = time.perf_counter() - t_wall0
    if ws > 1:
        torch.distributed.barrier()
    clocks = sampler.stop()
    total_ms = max_over_ranks(total_ms, dev)
    evals = n * len(SWEEP) * args.steps * ws
    value = whole_job_rate(n * len(SWEEP) * args.steps, ws, total_ms / 1e3)

    # end to end through the host-buffer entry point (pinned memory, copies inside the timed region), under
    # the same protocol as `value`: L2 flushed before every step, CUDA events around the step's six calls
    xh = torch.from_numpy(w.xyzq).pin_memory()
    oh = [torch.empty((n, 4), dtype=torch.float32).pin_memory() for _ in SWEEP]
    eh = [torch.empty(4, dtype=torch.float64).pin_memory() for _ in SWEEP]
    for _ in range(max(1, args.warmup)):
        flush.fill_(1.0)
        for c, o, e in zip(ctxs, oh, eh):
            usr.usr_eval_host(c.ctx, n, xh.data_ptr(), o.data_ptr(), e.data_ptr(), stream)
    torch.cuda.synchronize()
    t_e2e = 0.0
    for k in range(args.steps):
        flush.fill_(float(k % 7))
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for c, o, e in zip(ctxs, oh, eh):
            usr.usr_eval_host(c.ctx, n, xh.data_ptr(), o.data_ptr(), e.data_ptr(), stream)
        e1.record(stream)
        e1.synchronize()
        t_e2e += e0.elapsed_time(e1) / 1e3
    t_e2e = max_over_ranks(t_e2e, dev)
    e2e_value = whole_job_rate(n * len(SWEEP) * args.steps, ws, t_e2e)
    chosen_outs = [o.double().cpu().numpy() for o in outs]
    chosen_E = [float(e[0].item()) for e in ens]
    infos = [c.info for c in ctxs]
    for c in ctxs:
        c.close()

    # the plain FP32 comparators, same workload and protocol
    comps = {}
    for form in COMPARATORS:
        tms, _, _, cc, co, _ = _time_form(usr, torch, w, x, form, args.steps, args.warmup, flush, stream)
        comps[form[0]] = {"value": evals / ws / (tms / 1e3), "ms_per_step": tms / args.steps,
                          "out_rc8": co[0].double().cpu().numpy()}
        for c in cc:
            c.close()

    serving = run_serving(usr, torch, args.serve_systems) if args.serve_systems > 0 else None
    scale = run_scale(usr, torch, args.steps, args.warmup, flush, stream) if not args.no_scale else None
    fp32_peak = usr.usr_fp32_peak()     # measured FP32 FMA peak of this GPU (the pair kernel's denominator)

    if rank != 0:
        if ws > 1:
            torch.distributed.destroy_process_group()
        return
    # the dominant kernel (the pair kernel) and its roofline: its launch duration is the near stage's CUDA-event
    # time on the evaluation stream (events just before and after its launch), averaged over the timed steps
    per_stage = [sum(stage_ms[k][s] for k in range(len(SWEEP))) / len(SWEEP) for s in range(usr.USR_NSTAGES)]
    flops = sum(p * NEAR_FLOPS_PER_PAIR for p in pairs)                      # one launch per cutoff
    t_dom = sum(near_ms) / args.steps / 1e3
    achieved = flops / t_dom / 1e12
    peak_ok = fp32_peak > 0.0
    peak = fp32_peak if peak_ok else FP32_PEAK_DERIVED_TFLOPS
    roof = {"kernel": "near (k_near_half)", "bound": "alu", "achieved": achieved, "peak": peak,
            "unit": "TFLOP/s", "frac": achieved / peak, "traffic": NEAR_TRAFFIC_BYTES,
            "traffic_unit": "bytes per launch (DRAM read + write, ncu)",
            "peak_source": ("measured: register-only two-wide FFMA loop over all SMs (usr_fp32_peak), this run"
                            if peak_ok else "derived: 152 SMs x 128 FP32 lanes x 2 (FMA) x 2.07 GHz"),
            "peak_derived": FP32_PEAK_DERIVED_TFLOPS,
            "flops_per_pair": NEAR_FLOPS_PER_PAIR,
            "flops_per_pair_note": "algorithmic: 30-50 flops per pair inside r_c (Eq. 20's pair arithmetic), "
                                   "midpoint; the kernel's own arithmetic is "
                                   + ", ".join(str(near_flops_per_pair(i.poly_degree, i.n_explicit)) for i in infos[:1])
                                   + " per pair",
            "pairs_per_eval": pairs, "launch_ms_mean": 1e3 * t_dom / len(SWEEP)}

    # stage-wise floors of the chosen form, summed over the sweep, against the measured stage times
    peaks = measured_peaks()
    peaks["fp32_tflops"] = peak
    floors = [stage_floors(n, p, i, w.grid, CHOSEN[2], 3, peaks) for p, i in zip(pairs, infos)]
    floor_ms = {st: sum(fl[st] for fl in floors) / len(SWEEP) for st in usr.STAGES}
    eval_ms = total_ms / args.steps / len(SWEEP)
    stage_roof = {"floor_ms_mean": floor_ms, "measured_ms_mean": dict(zip(usr.STAGES, per_stage)),
                  "eval_ms_mean": eval_ms,
                  "frac_of_eval_time": sum(floor_ms.values()) / eval_ms,
                  "note": "the far stages run concurrently with the near stage (two streams), so the measured "
                          "stages add up to more than an evaluation; frac = sum of the floors / evaluation time",
                  "peaks": {"fp32_tflops": peak, "hbm_gbs": peaks["hbm_gbs"],
                            "bf16_tflops": peaks["bf16_tflops"],
                            "source": f"FP32 {'measured in this run' if peak_ok else 'derived'}; HBM and BF16 "
                                      f"{peaks['source']} (MEASURED_PEAKS.json)"}}

    # accuracy of every form against the FP64 oracle at r_c = 8 and of the chosen form at 10 and 13 (full evaluations)
    t0 = time.perf_counter()
    ref8 = cpu_oracle_eval(w, SWEEP[0])
    i10 = SWEEP.index(10.0)
    ref10 = cpu_oracle_eval(w, SWEEP[i10])
    ref13 = cpu_oracle_eval(w, SWEEP[-1])
    t_cpu = time.perf_counter() - t0
    acc = {CHOSEN[0]: {"rms_force_rel_err_rc8": O.rms_rel(chosen_outs[0][:, :3], ref8.F),
                       "rms_force_rel_err_rc10": O.rms_rel(chosen_outs[i10][:, :3], ref10.F),
                       "rms_force_rel_err_rc13": O.rms_rel(chosen_outs[-1][:, :3], ref13.F),
                       "energy_rel_err_rc8": abs(chosen_E[0] / ref8.E - 1.0),
                       "energy_rel_err_rc10": abs(chosen_E[i10] / ref10.E - 1.0),
                       "energy_rel_err_rc13": abs(chosen_E[-1] / ref13.E - 1.0)}}
    comparators = {}
    for name, v in comps.items():
        comparators[name] = {"value": v["value"], "unit": UNIT, "ms_per_step": v["ms_per_step"],
                             "rms_force_rel_err_rc8": O.rms_rel(v["out_rc8"][:, :3], ref8.F)}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None,
        "dtype": "f32 pairs, tf32x3 tensor-core spreading and bf16x3 convolutions with f32 accumulation, f64 energy",
        "data": "synthetic",
        "config": {"workload": f"{WORKLOAD}: {n} charges (2133 12-bead chains + 12800 waters), 80x80x100 A, "
                               f"64x64x80 grid, C1 b=2, r_c sweep 8-13 A (6 evals/step)",
                   "form": {"name": CHOSEN[0], "conv": "bf16x3", "spread_points": CHOSEN[2],
                            "spread_sigma_over_h": CHOSEN[3]},
                   "global_batch": n * len(SWEEP) * ws, "parallelism": f"replicas x{ws}",
                   "l2": "flushed between steps (512 MB write)", "wall_s_timed": t_wall},
        "accuracy": acc,
        "comparators": comparators,
        "serving": serving,
        "scale_1m": scale,
        "roofline": roof,
        "stage_ms_mean": dict(zip(usr.STAGES, per_stage)),
        "stage_roofline": stage_roof,
        "cpu_baseline": {"value": 3 * n / t_cpu, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle",
                         "sample": f"three full FP64 oracle evaluations (E, all forces and potentials) of the "
                                   f"{n}-charge slab, at r_c = 8, 10 and 13 A ({t_cpu:.1f} s in all)"},
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": 16 * n * len(SWEEP),
                "d2h_bytes_per_step": (16 * n + 32) * len(SWEEP)},
        "clocks": clocks,
        "gpu_launches": KERNELS_PER_EVAL * len(SWEEP) * args.steps,
    }
    print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--serve-systems", type=int, default=512,
                    help="systems in the serving stream (0 skips the serving measurement)")
    ap.add_argument("--no-scale", action="store_true",
                    help="skip the 1,064,799-charge water box (r_c = 10 A, 176^3 grid, every form)")
    args = ap.parse_args()
    if args.warmup < 3 and args.impl != "reference":
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
