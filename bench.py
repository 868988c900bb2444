"""Benchmark: Image Domain Gridding, grid + degrid throughput on one GB300.

One step = one pass of the whole hot path over the workload: idg_grid (plan's
subgrid images, taper and A-terms, subgrid FFT, adder into a zeroed grid)
followed by idg_degrid (splitter, subgrid IFFT, taper and A-terms, degridder)
from a model grid.  value = visibilities / (time of grid + degrid) in MVis/s,
with inputs resident in device memory.  e2e = the same metric through the
host-buffer C-ABI call that runs both directions (idg_grid_degrid_host) with the
copies from and to page-locked host memory inside the timed region.

Default workload: the LOFAR-like configuration (48 stations, 1128 baselines,
4096 x 1 s, 16 channels 130-146 MHz, 73.9 M visibilities, subgrid 32, grid
4096^2 x 4, A-terms every 128 timesteps).  Visibilities (2.37 GB) and grid
(0.54 GB) exceed the 129 MB L2, so no flush is needed between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

# Roofline of the gridder and degridder: FP32 FMA lanes.  Per visibility-pixel
# the algorithm needs 16 FMAs (4 complex multiply-adds) and 2 FMAs for the phase
# a*X + (b*Y + c*n'); sin and cos run on the SFU and, with packed f32x2 FMAs,
# issue slots are not the binding limit.  Every SM retires 128 FP32 FMAs per
# cycle, so the peak is SMs x 128 x f_max / 18 visibility-pixels per second.
FMA_PER_VISPIX = 18
LANES_PER_SM = 128
# Tensor-core forms: the complex multiply-adds run on the tensor cores and the
# CUDA cores generate the phasors.  Per visibility-pixel that takes at least 9
# issue slots: 2 FFMA for the phase, 1 FMUL for the sin/cos argument, 2 SFU
# (sin, cos) and 4 for the FP16 hi/lo split (2 packs, 2 mixed-precision fma).
# An SM issues 4 x 32 thread-instructions per clock.
ISSUE_PER_VISPIX_TC = 9
# DRAM bytes (read + write) per visibility-pixel of one launch, from the ncu
# capture of the separable kernels (the default at L = 32 where the plan is
# separable) on the LOFAR-like slice, one launch of all its subgrids, 4.731e9
# visibility-pixels: gridder 178.2 MB (visibilities and coordinates in; the
# atomically updated grid lines are still dirty in L2 when the launch ends), degridder
# 120.4 MB
# (grid lines and coordinates in, model visibilities out).  The traffic is
# proportional to the work, so it scales to a full launch by the units processed.
# Kernels without a capture of their current code report no traffic.
FUSED_VARIANT = "tcgen05_tmemA_ws_nt288_fused"
SEP_VARIANT = "tcgen05_separable_fused"
# Tensor-core work of the separable kernels at subgrid size L (kind::f16, M = 128, K = 16
# per MMA, 2 FLOP per multiply-add): the gridder issues N = 6 L + 2 L per group of 8
# visibilities (192 + 64 at L = 32), the degridder L / 8 K steps of 4 x N = 8 L per tile of
# 128 visibilities (at L = 32 and 24 in two rounds of two polarisations).
SEP_DEGRID_TILE = 128


def sep_grid_flop_per_group(L):
    return 2 * 128 * 16 * (6 * L + 2 * L)


def sep_degrid_flop_per_tile(L):
    return (L // 8) * 4 * 2 * 128 * 16 * (8 * L)

# Half of those products are the FP16 hi/lo split that keeps FP32 accuracy: the
# gridder's N = 256 columns are A_hi x [B_hi (128) | B0_lo (64)] and A_lo x B0_hi (64);
# the degridder's four products per K step are hi x hi of the m = 0 and the
# first-order w term plus the two lo corrections of the m = 0 term.  The method's own
# contraction (hi x hi) is the other half.
SEP_USEFUL_SHARE = 0.5
DTYPE_SEP = "f32 (fp16 hi/lo split tensor-core products, fp32 accumulate)"
DTYPE_MIXED = ("f32 (fp16 hi/lo split tensor-core products for subgrids within the separable bound and "
               "pieces, packed fp32 for the rest; fp32 accumulate)")
KERNEL_TRAFFIC = {
    "gridder": {SEP_VARIANT: 178.2e6 / 4.731e9},
    "degridder": {SEP_VARIANT: 120.4e6 / 4.731e9},
}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--config", default="lofar",
                    choices=["lofar", "lofar-slice", "tiny", "batched", "serving", "precision"])
    ap.add_argument("--rate", type=float, default=50.0, help="serving: Poisson arrival rate (jobs/s)")
    ap.add_argument("--jobs", type=int, default=None,
                    help="jobs of the batched (default 256) or serving (default 64) configuration")
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--cpu-seconds", type=float, default=10.0, help="target CPU time of the oracle sample")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-forms", action="store_true", help="skip the forms block of the default line")
    ap.add_argument("--step-only", action="store_true",
                    help="the grid + degrid step and its end-to-end number only: skip the image, calibration, "
                         "classical, stages and forms blocks of the default line")
    ap.add_argument("--shard", action="store_true",
                    help="with several ranks: split one plan's subgrids over them (one all-reduce per direction) "
                         "instead of running replicas")
    ap.add_argument("--case", default=None, choices=["image", "classical", "calibration", "stages", "lofar_slice"],
                    help="run one small profiling case alone (for ncu) instead of the benchmark")
    return ap.parse_args()


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if (args.impl == "gb300" and torch.cuda.is_available()) else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(world, x: float) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def sum_over_ranks(world, x: float) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def whole_job_rate(world, seconds_local: float, units_local: float) -> float:
    """Units per second of the whole job: the units all ranks processed over the
    slowest rank's time (each rank times the same bracketed region)."""
    return sum_over_ranks(world, units_local) / max_over_ranks(world, seconds_local)


def _cpulist(text: str) -> set:
    cpus = set()
    for part in text.strip().split(","):
        if not part:
            continue
        lo, _, hi = part.partition("-")
        cpus.update(range(int(lo), int(hi or lo) + 1))
    return cpus


class near_gpu_memory:
    """Within the block, run on the CPUs next to the GPU (its PCI device's
    local_cpulist in sysfs) so that page-locked host buffers allocated and filled
    there sit on the GPU's own host memory node (first-touch placement); the
    previous CPU set comes back on exit.  No-op where sysfs or affinity is not
    available.  Records the CPUs used in .cpus."""

    def __init__(self, device: int):
        self.device, self.saved, self.cpus = device, None, None

    def __enter__(self):
        import torch
        try:
            pr = torch.cuda.get_device_properties(self.device)
            bdf = f"{pr.pci_domain_id:04x}:{pr.pci_bus_id:02x}:{pr.pci_device_id:02x}.0"
            with open(f"/sys/bus/pci/devices/{bdf}/local_cpulist") as f:
                local = _cpulist(f.read())
            self.saved = os.sched_getaffinity(0)
            use = local & self.saved
            if use and use != self.saved:
                os.sched_setaffinity(0, use)
                self.cpus = f"{len(use)} of {len(self.saved)} allowed CPUs, local to {bdf}"
            else:
                self.cpus = (f"all {len(use)} allowed CPUs are local to {bdf}" if use else
                             f"none of the {len(self.saved)} allowed CPUs is local to {bdf}")
                self.saved = None
        except Exception:          # no sysfs entry, no affinity support, no device properties
            self.saved = None
        return self

    def __exit__(self, *exc):
        if self.saved is not None:
            os.sched_setaffinity(0, self.saved)
        return False


def make_workload(name):
    from paper_1909_07226_gb300 import synthetic as syn
    if name == "tiny":
        return syn.make_tiny()
    if name == "lofar-slice":
        # the LOFAR-like workload cut to its first 256 timesteps (two A-term
        # slots): still larger than L2, small enough for a detailed profile
        return syn.make_lofar(with_vis=True, n_t=256)
    return syn.make_lofar(with_vis=True)


def workload_config(wl, name):
    return {
        "workload": {"lofar": "LOFAR-like plain: 48 stations (1128 baselines), 4096 x 1 s, 16 ch 130-146 MHz, "
                              "subgrid 32, grid 4096^2 x 4 c64, A-terms every 128 t",
                     "lofar-slice": "LOFAR-like plain, first 256 of 4096 timesteps (profiling slice)",
                     "tiny": "Tiny plain: 8 stations, 64 x 10 s, 8 ch 140-148 MHz, subgrid 24, grid 512^2 x 4 c64"}[name],
        "n_vis": int(wl.n_vis), "n_baselines": int(wl.n_bl), "n_timesteps": int(wl.n_t),
        "n_channels": int(wl.n_chan), "subgrid_size": int(wl.subgrid_size), "grid_size": int(wl.grid_size),
        "kernel_size": float(wl.kernel_size), "max_timesteps_per_subgrid": int(wl.max_timesteps),
        "aterm_slots": int(wl.n_slots), "w_step": float(wl.w_step),
        "l2": "inputs larger than L2 (visibilities and grid), no flush",
    }


# ---------------------------------------------------------------------------
# clocks sampled during the timed region


class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.proc = None
        self.sel = []
        try:
            import torch
            props = torch.cuda.get_device_properties(device_index)
            uuid = str(getattr(props, "uuid", "") or "")
            if uuid:
                self.sel = ["-i", uuid if uuid.startswith("GPU-") else "GPU-" + uuid]
        except Exception:
            self.sel = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200", *self.sel], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, smax, pw, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
                pw.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "samples": len(sm),
                "power_w_max": max(pw) if pw else None, "reasons": sorted(reasons)}


# ---------------------------------------------------------------------------
# the oracle on the host cores (CPU baseline and the reference arm)


def oracle_sample(wl, op, target_s: float, seed: int = 0):
    """Time the FP64 oracle's grid + degrid on a deterministic sample of the
    workload's subgrids sized to about target_s seconds.  Returns (MVis/s,
    description, seconds)."""
    from oracle import oracle as O
    from paper_1909_07226_gb300 import synthetic as syn
    n = op.n_sub
    L = wl.subgrid_size
    model = syn.random_grid(np.random.default_rng(seed), 1, 2 * L)   # local model patch source
    kp = op.desc[:, O.D_KP].astype(np.int64)

    def run(ids):
        sub_desc = op.desc[ids].copy()
        # place the sampled subgrids on a private small grid so the oracle's
        # adder and splitter stay O(L^2) per subgrid
        sub_desc[:, O.D_Q0] = 0
        sub_desc[:, O.D_R0] = 0
        sub_desc[:, O.D_LAYER] = 0
        p_s = O.OraclePlan(sub_desc, 0, 1, op.k_min)
        wl_s = _SubWorkload(wl, grid_size=2 * L)
        t0 = time.perf_counter()
        img = O.subgrid_images(wl, O.OraclePlan(op.desc, 0, op.n_w, op.k_min), ids)
        uv = O.dft2(img, -1)
        O.add(wl_s, p_s, uv)
        t1 = time.perf_counter()
        sp = O.split(wl_s, p_s, model)
        im = O.dft2(sp, +1)
        O.degrid_images(wl, O.OraclePlan(op.desc, 0, op.n_w, op.k_min), im, ids)
        t2 = time.perf_counter()
        return t2 - t0

    # calibrate on two subgrids per host core (the oracle runs one subgrid per
    # OpenMP thread), then size the sample
    rng = np.random.default_rng(seed)
    cal = np.sort(rng.choice(n, size=min(n, 2 * (os.cpu_count() or 1)), replace=False)).astype(np.int32)
    tc = run(cal)
    per_vis = tc / max(1, int(kp[cal].sum()))
    want_vis = target_s / max(per_vis, 1e-12)
    mean_kp = float(kp.mean())
    m = int(min(n, max(4, want_vis / mean_kp)))
    ids = np.sort(rng.choice(n, size=m, replace=False)).astype(np.int32)
    dt = run(ids)
    nvis = int(kp[ids].sum())
    desc = (f"{m} of {n} subgrids drawn uniformly (seed {seed}), {nvis} visibilities, "
            f"grid + degrid in FP64 on all host cores")
    return nvis / dt / 1e6, desc, dt


class _SubWorkload:
    """View of a workload with a different grid size (for the oracle sample)."""

    def __init__(self, wl, grid_size):
        self._wl = wl
        self.grid_size = grid_size

    def __getattr__(self, k):
        return getattr(self._wl, k)


# ---------------------------------------------------------------------------


def run_reference(args, world, rank):
    if rank != 0:
        return
    from oracle import oracle as O
    O.build()
    wl = make_workload(args.config)
    op = O.plan(wl)
    cfg = workload_config(wl, args.config)
    for _ in range(args.warmup):
        oracle_sample(wl, op, min(args.cpu_seconds, 2.0), seed=1)
    vals, secs, descs = [], [], []
    for k in range(args.steps):
        v, d, s = oracle_sample(wl, op, args.cpu_seconds, seed=100 + k)
        vals.append(v)
        secs.append(s)
        descs.append(d)
    value = float(np.mean(vals))
    cores = os.cpu_count()
    rec = {
        "impl": "reference", "metric": "grid+degrid MVis/s", "value": value, "unit": "MVis/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * float(np.mean(secs)), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": cfg,
        "cpu_baseline": {"value": value, "unit": "MVis/s", "cores": cores, "kind": "oracle",
                         "sample": descs[0] + " (one sample per step)"},
        "e2e": {"value": value, "unit": "MVis/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(rec))


def run_gb300(args, world, rank, local):
    import torch
    from paper_1909_07226_gb300 import build as lib_build
    from paper_1909_07226_gb300 import idg
    from paper_1909_07226_gb300 import synthetic as syn

    torch.cuda.set_device(local)
    lib_build.build()
    idg.load()
    wl = make_workload(args.config)
    t0 = time.perf_counter()
    plan = idg.plan_from_workload(wl)
    plan_s = time.perf_counter() - t0
    dev = torch.device("cuda", local)
    vis = torch.from_numpy(wl.vis).to(dev)
    aterms = torch.from_numpy(wl.aterms).to(dev)
    taper = torch.from_numpy(wl.taper).to(dev)
    flags = None if wl.flags is None else torch.from_numpy(wl.flags).to(dev)
    model_h = syn.random_grid(np.random.default_rng(7), plan.n_w_layers, wl.grid_size)
    model = torch.from_numpy(model_h).to(dev)
    grid = torch.empty((plan.n_w_layers, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device=dev)
    vis_out = torch.empty_like(vis)
    stream = torch.cuda.current_stream(dev)

    sharded = args.shard and world > 1

    def step():
        if sharded:
            # one plan over all ranks: each grids and degrids its range of subgrids, one
            # all-reduce per direction (strong scaling; every rank ends with the whole result)
            from paper_1909_07226_gb300 import shard
            shard.grid(plan, vis, flags, aterms, taper, grid, stream=stream)
            shard.degrid(plan, model, flags, aterms, taper, vis_out, stream=stream)
            return
        grid.zero_()                       # Algorithm 1 starts from V = 0
        idg.grid(plan, vis, flags, aterms, taper, grid, stream)
        idg.degrid(plan, model, flags, aterms, taper, vis_out, stream)

    for _ in range(max(3, args.warmup)):
        step()
    torch.cuda.synchronize()
    sampler = ClockSampler(local)
    sampler.start()
    idg.profile_enable(True)
    idg.profile_read(reset=True)
    barrier(world)
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        step()
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    clocks = sampler.stop()
    idg.profile_enable(False)
    prof = idg.profile_read(reset=True)
    ms_local = ev0.elapsed_time(ev1)
    ms_total = max_over_ranks(world, ms_local)
    ms_step = ms_total / args.steps
    # replicas: every rank processes the whole workload; sharded: the ranks share one
    value = whole_job_rate(world, ms_local * 1e-3, float(wl.n_vis) * args.steps / (world if sharded else 1)) / 1e6

    # end to end through the host-buffer C-ABI calls (measured right after the device-buffer
    # steps, before the blocks below fill the device with their own buffers)
    with near_gpu_memory(local) as placement:
        vis_h = torch.empty(vis.shape, dtype=torch.complex64, pin_memory=True)
        vis_h.copy_(torch.from_numpy(wl.vis))
        model_p = torch.empty(model.shape, dtype=torch.complex64, pin_memory=True)
        model_p.copy_(torch.from_numpy(model_h))
        grid_h = torch.empty(grid.shape, dtype=torch.complex64, pin_memory=True)
        grid_h.zero_()
        visout_h = torch.empty(vis.shape, dtype=torch.complex64, pin_memory=True)
        visout_h.zero_()
    aterms_h = torch.from_numpy(wl.aterms)
    taper_h = torch.from_numpy(wl.taper)
    flags_h = None if wl.flags is None else torch.from_numpy(wl.flags)

    def e2e_step():
        # both directions in one pipelined call: the grid copies overlap the other direction
        idg.grid_degrid_host(plan, vis_h, model_p, flags_h, aterms_h, taper_h, grid_h, visout_h, stream)

    e2e_step()
    torch.cuda.synchronize()
    barrier(world)
    t0 = time.perf_counter()
    for _ in range(args.e2e_steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_value = whole_job_rate(world, time.perf_counter() - t0, float(wl.n_vis) * args.e2e_steps) / 1e6
    nvis = wl.n_vis
    fl = 0 if wl.flags is None else wl.flags.nbytes
    # in: visibilities, model grid, flags, A-terms, taper; out: grid, model visibilities
    h2d = nvis * 32 + model_h.nbytes + fl + wl.aterms.nbytes + wl.taper.nbytes
    d2h = grid_h.numel() * 8 + nvis * 32

    # kernels: achieved against their rooflines
    props = torch.cuda.get_device_properties(local)
    n_sm = props.multi_processor_count
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        pass
    f_max_mhz = float(peaks.get("sm_max_mhz", 2070.0))
    hbm_peak = float(peaks.get("hbm_gbs", 6800.0))
    hbm_src = "measured" if "hbm_gbs" in peaks else "fallback"
    alu_peak = n_sm * LANES_PER_SM * f_max_mhz * 1e6 / FMA_PER_VISPIX / 1e9       # G vis-pix / s
    tc_peak = n_sm * LANES_PER_SM * f_max_mhz * 1e6 / ISSUE_PER_VISPIX_TC / 1e9
    fma_basis = (f"{n_sm} SMs x {LANES_PER_SM} FP32 FMA lanes x {f_max_mhz:.0f} MHz / {FMA_PER_VISPIX} FMA "
                 f"per visibility-pixel")
    tc_basis = (f"{n_sm} SMs x {LANES_PER_SM} issue slots x {f_max_mhz:.0f} MHz / {ISSUE_PER_VISPIX_TC} "
                f"phasor-generation instructions per visibility-pixel (multiply-adds on the tensor cores)")
    bf16_peak = float(peaks.get("bf16_tflops", 1900.0))
    bf16_src = "measured burst" if "bf16_tflops" in peaks else "fallback"
    kp = plan.export()[:, 9].astype(np.int64)                 # K_p per subgrid (descriptor field 9)
    sep_flop = {"gridder": float(((kp + 7) // 8).sum()) * sep_grid_flop_per_group(wl.subgrid_size),
                "degridder": float((-(-kp // SEP_DEGRID_TILE)).sum()) * sep_degrid_flop_per_tile(wl.subgrid_size)}
    kernels = {}
    for k, d in prof.items():
        if d["launches"] == 0:
            continue
        ent = {"launches": d["launches"] // args.steps, "ms_per_step": d["ms"] / args.steps,
               "share": d["ms"] / ms_total if ms_total > 0 else None}
        if k in ("gridder", "degridder"):
            ach = d["work"] / (d["ms"] * 1e-3) / 1e9
            var = idg.kernel_variants(k, wl.subgrid_size)[idg.plan_get_kernel_variant(plan, k)]
            # a step without adder (splitter) launches ran a fused tensor-core kernel: the separable
            # one where the plan allows it, else the direct one (transform and adder in the same CTA)
            if prof["adder" if k == "gridder" else "splitter"]["launches"] == 0:
                var = SEP_VARIANT if plan.stats.separable else FUSED_VARIANT
            if var == SEP_VARIANT:
                tfl = sep_flop[k] * args.steps / (d["ms"] * 1e-3) / 1e12
                ent.update(bound="tensor", achieved=tfl, peak=bf16_peak, unit="TFLOP/s", frac=tfl / bf16_peak,
                           variant=var, peak_basis=f"dense bf16 tensor rate ({bf16_src}); FP16 runs at the same rate",
                           useful_frac=SEP_USEFUL_SHARE * tfl / bf16_peak,
                           useful_basis="hi x hi products only (the method's contraction); the rest is the FP16 "
                                        "hi/lo split for FP32 accuracy",
                           achieved_vispix=ach, vispix_unit="Gvispix/s", frac_of_fp32_fma_peak=ach / alu_peak)
            else:
                tc = var.startswith("tcgen05")
                pk = tc_peak if tc else alu_peak
                ent.update(bound="alu", achieved=ach, peak=pk, unit="Gvispix/s", frac=ach / pk, variant=var,
                           peak_basis=tc_basis if tc else fma_basis, frac_of_fp32_fma_peak=ach / alu_peak)
        elif k in ("adder", "splitter"):
            ach = d["work"] / (d["ms"] * 1e-3) / 1e9
            ent.update(bound="hbm", achieved=ach, peak=hbm_peak, unit="GB/s", frac=ach / hbm_peak)
        kernels[k] = ent
    dom = max(("gridder", "degridder"), key=lambda k: prof[k]["ms"])
    traffic = None
    L = wl.subgrid_size
    per_vispix = KERNEL_TRAFFIC.get(dom, {}).get(kernels[dom]["variant"]) if L == 32 else None
    if per_vispix is not None:
        traffic = per_vispix * prof[dom]["work"] / prof[dom]["launches"]
    roof = {"kernel": dom, "variant": kernels[dom]["variant"], "bound": kernels[dom]["bound"],
            "achieved": kernels[dom]["achieved"], "peak": kernels[dom]["peak"],
            "unit": kernels[dom]["unit"], "frac": kernels[dom]["frac"], "traffic": traffic,
            "traffic_basis": "ncu dram bytes per visibility-pixel of the slice capture x visibility-pixels per launch"
            if traffic is not None else None,
            "peak_basis": kernels[dom]["peak_basis"], "frac_of_fp32_fma_peak": kernels[dom]["frac_of_fp32_fma_peak"],
            "hbm_peak_basis": hbm_src}
    if "useful_frac" in kernels[dom]:
        roof["useful_frac"] = kernels[dom]["useful_frac"]
        roof["useful_basis"] = kernels[dom]["useful_basis"]
    if "achieved_vispix" in kernels[dom]:
        roof["achieved_vispix"] = kernels[dom]["achieved_vispix"]
        roof["flop_basis"] = ("MMA FLOP issued: gridder 2*128*16*8L per group of 8 visibilities, degridder "
                              "(L/8)*4*2*128*16*8L per tile of 128 (FP16 hi/lo split products included)")
    gpu_launches = int(sum(d["launches"] for d in prof.values()))

    # image-side steps, outside the grid + degrid step: the whole grid to the image and
    # back (idg_image_from_grid / idg_grid_from_image, PSWF window of the taper).  Each call
    # reads and writes the N x N x 4 complex64 image twice (row pass, column pass) per w-layer.
    image_steps = None
    if wl.grid_size in (16, 32, 64, 128, 256, 512, 1024, 2048, 4096) and not args.step_only:
        win, _ = idg.taper_window(wl.subgrid_size, float(wl.kernel_size), idg.TAPER_PSWF)
        img = torch.empty((wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device=dev)
        im_ms = {}
        for name, fn in (("image_from_grid", lambda: idg.image_from_grid(plan, grid, win, img, stream)),
                         ("grid_from_image", lambda: idg.grid_from_image(plan, img, win, grid, stream))):
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(5):
                fn()
            e1.record(stream)
            torch.cuda.synchronize()
            im_ms[name] = e0.elapsed_time(e1) / 5
        idg.device_errors(stream)
        im_bytes = 4.0 * plan.n_w_layers * wl.grid_size ** 2 * 32
        image_steps = {name: {"ms": ms, "achieved": im_bytes / (ms * 1e-3) / 1e9, "peak": hbm_peak, "unit": "GB/s",
                              "frac": im_bytes / (ms * 1e-3) / 1e9 / hbm_peak} for name, ms in im_ms.items()}
        image_steps["bytes_per_call"] = im_bytes
        image_steps["basis"] = ("4 x n_w x N^2 x 32 B per call (row and column pass, read and write), "
                                f"against the {hbm_src} copy bandwidth")

    # calibration (idg_aterm_gradient) on the same workload
    calib = None if args.step_only else calibration_rate(idg, torch, dev, plan, wl, model, vis, flags, aterms, taper,
                                                         stream, hbm_peak)
    extras = args.config == "lofar" and not args.step_only

    # classical gridding with oversampled A/W-projection kernels rebuilt per subgrid (the
    # paper's comparison, Sect. 2) beside image domain gridding, on the precision
    # workload's A-term cadence (slots of 16 timesteps), first 256 timesteps
    classical = classical_comparison(idg, syn, torch, dev, stream, hbm_peak) if extras else None

    # the adder and the splitter as their own launches over every subgrid (the fused
    # kernels above do not launch them)
    stages = stage_rates(idg, torch, dev, plan, vis, flags, aterms, taper, grid, stream, hbm_peak) if extras else None

    # the deployment forms on small fixed cases: batched against per-job calls on 16 jobs,
    # serving against per-job FIFO at 50 jobs/s, errors of the precision forms
    forms = None
    if extras and not args.no_forms:
        b16 = batched_compare(idg, syn, torch, dev, 16, 3, 3, seed=1916)
        forms = {"batched_16_jobs": {k: b16[k] for k in ("n_vis", "plain_mvis_per_s", "batched_mvis_per_s",
                                                         "batched_over_plain", "classes")},
                 "serving_50_per_s": serving_point(idg, syn, torch),
                 "precision_errors": precision_errors(idg, syn, torch, dev, stream)}

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        from oracle import oracle as O
        O.build()
        op = O.plan(wl)
        v, desc, secs = oracle_sample(wl, op, args.cpu_seconds)
        cpu = {"value": v, "unit": "MVis/s", "cores": os.cpu_count(), "kind": "oracle", "sample": desc,
               "seconds": secs}

    if rank == 0:
        rec = {
            "metric": "grid+degrid MVis/s", "value": value, "unit": "MVis/s", "n_gpus": world,
            "steps": args.steps, "warmup": max(3, args.warmup), "ms_per_step": ms_step,
            "higher_is_better": True, "scaling": "strong" if sharded else "weak", "vs_baseline": None,
            "dtype": DTYPE_SEP if plan.stats.separable else "f32",
            "data": "synthetic", "config": workload_config(wl, args.config),
            "roofline": roof, "kernels": kernels,
            "e2e": {"value": e2e_value, "unit": "MVis/s", "h2d_bytes_per_step": int(h2d),
                    "d2h_bytes_per_step": int(d2h), "steps": args.e2e_steps,
                    "host_buffers_placed_from_cpus": placement.cpus},
            "gpu_launches": gpu_launches, "clocks": clocks, "cpu_baseline": cpu, "image_steps": image_steps,
            "calibration": calib, "classical": classical, "stages": stages, "forms": forms,
            "plan": {"n_subgrids": plan.n_subgrids, "seconds": plan_s},
            "parallelism": ("sharded subgrids, one all-reduce per direction" if sharded else "replicas")
            if world > 1 else "single GPU",
        }
        print(json.dumps(rec))


def calibration_rate(idg, torch, dev, plan, wl, model, vis, flags, aterms, taper, stream, hbm_peak):
    """One idg_aterm_gradient call on the workload (the residuals, cost and A-term
    gradient of the model grid against the observed visibilities): a degrid and a
    grid pass of every visibility plus the residual and gradient kernels."""
    resid = torch.empty_like(vis)
    agrad = torch.zeros(aterms.shape, dtype=torch.complex64, device=dev)
    cost = torch.zeros(1, dtype=torch.float64, device=dev)

    def calib_call():
        idg.aterm_gradient(plan, model, vis, flags, aterms, taper, resid, agrad, cost, stream)

    for _ in range(3):
        calib_call()
    torch.cuda.synchronize()
    idg.profile_enable(True)
    idg.profile_read(reset=True)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    n_cal = 5
    e0.record(stream)
    for _ in range(n_cal):
        calib_call()
    e1.record(stream)
    torch.cuda.synchronize()
    cprof = idg.profile_read(reset=True)
    idg.profile_enable(False)
    idg.device_errors(stream)
    cal_ms = e0.elapsed_time(e1) / n_cal
    calib = {"ms": cal_ms, "mvis_per_s": wl.n_vis / (cal_ms * 1e-3) / 1e6,
             "launches": int(sum(d["launches"] for d in cprof.values())) // n_cal, "kernels": {}}
    for k, d in cprof.items():
        if d["launches"] == 0:
            continue
        ent = {"ms_per_call": d["ms"] / n_cal, "launches": d["launches"] // n_cal}
        if k in ("calib_residual", "calib_gradient", "splitter"):
            ach = d["work"] / (d["ms"] * 1e-3) / 1e9
            ent.update(bound="hbm", achieved=ach, peak=hbm_peak, unit="GB/s", frac=ach / hbm_peak)
        elif k in ("gridder", "degridder"):
            ent.update(achieved_vispix=d["work"] / (d["ms"] * 1e-3) / 1e9, vispix_unit="Gvispix/s")
        calib["kernels"][k] = ent
    calib["basis"] = ("one idg_aterm_gradient call: splitter, inverse transform and degridder (stage kernels), "
                      "residual kernel (96 B per visibility), gridder of the residuals, gradient kernel (256 B per "
                      "subgrid pixel); MVis/s = visibilities per call / call time")
    return calib


def stage_rates(idg, torch, dev, plan, vis, flags, aterms, taper, grid, stream, hbm_peak):
    """The adder and the splitter as separate launches over every subgrid of the
    plan (chunks of 16384 subgrid images, 512 MiB at L = 32): algorithmic bytes
    96 B per subgrid pixel for the adder (subgrid read, grid read and written)
    and 64 B for the splitter (grid read, subgrid written), per CUDA events."""
    L = plan.stats.subgrid_size
    n = plan.n_subgrids
    chunk = min(n, 16384)
    sub = torch.zeros((chunk, L, L, 4), dtype=torch.complex64, device=dev)
    idg.grid_subgrids(plan, 0, chunk, vis, flags, aterms, taper, sub, stream)
    out = {}
    for name, fn in (("adder", lambda f, c: idg.add_subgrids(plan, f, c, sub[:c], grid, stream)),
                     ("splitter", lambda f, c: idg.split_subgrids(plan, f, c, grid, sub[:c], stream))):
        def one_pass():
            for f in range(0, n, chunk):
                fn(f, min(chunk, n - f))
        one_pass()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        reps = 3
        e0.record(stream)
        for _ in range(reps):
            one_pass()
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        byts = (96.0 if name == "adder" else 64.0) * n * L * L
        out[name] = {"ms": ms, "launches": (n + chunk - 1) // chunk, "bytes": byts, "bound": "hbm",
                     "achieved": byts / (ms * 1e-3) / 1e9, "peak": hbm_peak, "unit": "GB/s",
                     "frac": byts / (ms * 1e-3) / 1e9 / hbm_peak}
    out["basis"] = (f"all {n} subgrids of the workload through idg_add_subgrids / idg_split_subgrids in chunks of "
                    f"{chunk}; adder 96 B and splitter 64 B per subgrid pixel (algorithmic), against the measured copy "
                    "bandwidth; overlapping subgrids share grid lines in L2")
    return out


def precision_errors(idg, syn, torch, dev, stream, n_t=32):
    """Error of every precision form against the FP64 oracle on the precision
    workload's first n_t timesteps (the whole grid and every visibility)."""
    from oracle import oracle as O
    O.build()
    forms = {"direct_sincos": dict(),
             "channel_recurrence": dict(precision_mode=idg.PHASOR_RECURRENCE),
             "compensated_adder": dict(adder_mode=idg.ADDER_COMPENSATED),
             "sorted_adder": dict(adder_mode=idg.ADDER_SORTED),
             "tc_split_transform": dict(fft_mode=idg.FFT_TC_SPLIT)}
    sl = syn.make_lofar(with_vis=True, n_t=n_t, slot_len=16, name="precision")
    op = O.plan(sl)
    ref_grid = O.grid(sl, op)
    model_h = syn.random_grid(np.random.default_rng(7), op.n_w, sl.grid_size)
    ref_vis = O.degrid(sl, op, model_h)
    d = dict(vis=torch.from_numpy(sl.vis).to(dev), at=torch.from_numpy(sl.aterms).to(dev),
             tp=torch.from_numpy(sl.taper).to(dev), model=torch.from_numpy(model_h).to(dev))
    out = {"workload": f"precision workload (A-terms every 16 timesteps), first {n_t} timesteps: {op.n_sub} "
                       f"subgrids, {sl.n_vis} visibilities, every pixel and visibility against the oracle"}
    for name, kw in forms.items():
        p = idg.plan_from_workload(sl, **kw)
        g = torch.zeros(ref_grid.shape, dtype=torch.complex64, device=dev)
        idg.grid(p, d["vis"], None, d["at"], d["tp"], g, stream)
        v = torch.zeros(sl.vis.shape, dtype=torch.complex64, device=dev)
        idg.degrid(p, d["model"], None, d["at"], d["tp"], v, stream)
        gg = g.cpu().numpy().astype(np.complex128)
        vv = v.cpu().numpy().astype(np.complex128)
        out[name] = {"grid_rel_rms": float(np.linalg.norm(gg - ref_grid) / np.linalg.norm(ref_grid)),
                     "grid_max_err_rel": float(np.max(np.abs(gg - ref_grid)) / np.max(np.abs(ref_grid))),
                     "vis_rel_rms": float(np.linalg.norm(vv - ref_vis) / np.linalg.norm(ref_vis)),
                     "vis_max_err_rel": float(np.max(np.abs(vv - ref_vis)) / np.max(np.abs(ref_vis)))}
        p.destroy()
    return out


def serving_point(idg, syn, torch, n_jobs=16, rate=50.0):
    """Serving engine vs per-job FIFO on one Poisson trace (latency and MVis/s)."""
    from paper_1909_07226_gb300 import serving
    wls = syn.make_batched_jobs(n_jobs, seed=1913, scale_t=0.25)
    kinds = ("cycle", "grid", "degrid")
    serving.Engine(budget_bytes=150 << 30).run(serving.make_trace(
        syn.make_batched_jobs(3, seed=7, scale_t=0.1), 1000.0, kinds, seed=7))
    torch.cuda.synchronize()
    srv = serving.Engine(budget_bytes=150 << 30, max_slots=32, graph=False).run(
        serving.make_trace(wls, rate, kinds))
    fifo = serving.run_plain_fifo(serving.make_trace(wls, rate, kinds))
    keep = ("grid_degrid_mvis_per_s", "latency_p50_s", "latency_p99_s", "makespan_s")
    return {"rate_jobs_per_s": rate, "jobs": n_jobs, "serving": {k: srv[k] for k in keep},
            "plain_fifo": {k: fifo[k] for k in keep},
            "workload": f"{n_jobs} requests from the batched distribution (timesteps scaled by 0.25), kinds "
                        f"cycle (5 major cycles) / grid / degrid"}


CLASSICAL_SUPPORT, CLASSICAL_OVERSAMPLE = 8, 16
# W-projection plane spacing: half a plane of w error is 2 pi (dw / 2) |n'| <= 0.07 rad
# at the corner of the LOFAR-like image (|n'| = 4.2e-4)
CLASSICAL_W_PLANE = 50.0


def classical_comparison(idg, syn, torch, dev, stream, hbm_peak):
    wl = syn.make_lofar(n_t=256, slot_len=16, name="precision")
    plan = idg.plan_from_workload(wl)
    M, O_ = CLASSICAL_SUPPORT, CLASSICAL_OVERSAMPLE
    S = wl.grid_size * wl.cell_size
    vis = torch.from_numpy(wl.vis).to(dev)
    at = torch.from_numpy(wl.aterms).to(dev)
    at_m = torch.from_numpy(syn.aterms_on_subgrid(wl.screens, M, S).astype(np.complex64)).to(dev)
    tap = torch.from_numpy(wl.taper).to(dev)
    g = torch.zeros((plan.n_w_layers, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device=dev)
    out = {"workload": f"LOFAR-like, first 256 timesteps, A-terms every 16 timesteps ({plan.n_subgrids} subgrids, "
                       f"{wl.n_vis} visibilities)",
           "support": M, "oversample": O_, "w_plane_step": CLASSICAL_W_PLANE}
    for name, fn in (("idg_grid", lambda: idg.grid(plan, vis, None, at, tap, g, stream)),
                     ("classical_grid", lambda: idg.classical_grid(plan, M, O_, CLASSICAL_W_PLANE, vis, None, at_m,
                                                                  None, g, stream))):
        for _ in range(2):
            fn()
        torch.cuda.synchronize()
        idg.profile_enable(True)
        idg.profile_read(reset=True)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(3):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        prof = idg.profile_read(reset=True)
        idg.profile_enable(False)
        idg.device_errors(stream)
        ms = e0.elapsed_time(e1) / 3
        ent = {"ms": ms, "mvis_per_s": wl.n_vis / (ms * 1e-3) / 1e6}
        if name == "classical_grid":
            kb = prof["classical_kernels"]
            ent["kernel_build_ms"] = kb["ms"] / 3
            ent["kernel_bytes_per_call"] = kb["work"] / 3
            ent["kernel_build"] = {"bound": "hbm", "achieved": kb["work"] / (kb["ms"] * 1e-3) / 1e9, "peak": hbm_peak,
                                   "unit": "GB/s", "frac": kb["work"] / (kb["ms"] * 1e-3) / 1e9 / hbm_peak}
            ent["gridding_ms"] = prof["classical_grid"]["ms"] / 3
            ent["kernel_build_share"] = kb["ms"] / max(kb["ms"] + prof["classical_grid"]["ms"], 1e-9)
            ent["launches"] = (kb["launches"] + prof["classical_grid"]["launches"]) // 3
        out[name] = ent
    out["classical_over_idg_time"] = out["classical_grid"]["ms"] / out["idg_grid"]["ms"]
    return out


def batched_compare(idg, syn, torch, dev, n_jobs, steps, warmup, seed=None):
    """The same uneven jobs gridded and degridded (a) one after another with
    idg_grid / idg_degrid (plain per-job form) and (b) as one batch (one persistent
    launch per subgrid size, subgrids kept in shared memory, graph replay).
    Returns (rec, n_vis, ms_plain, ms_batch, info)."""
    jobs = syn.make_batched_jobs(n_jobs, seed=seed)
    t0 = time.perf_counter()
    plans = [idg.plan_from_workload(w) for w in jobs]
    plan_s = time.perf_counter() - t0
    gen = torch.Generator(device=dev)
    gen.manual_seed(1912)
    bufs = []
    for w, p in zip(jobs, plans):
        vis = torch.randn((w.n_bl, w.n_t, w.n_chan, 4), dtype=torch.complex64, device=dev, generator=gen)
        flags = (torch.rand((w.n_bl, w.n_t, w.n_chan), device=dev, generator=gen) < w.flag_p).to(torch.uint8)
        grid = torch.zeros((p.n_w_layers, w.grid_size, w.grid_size, 4), dtype=torch.complex64, device=dev)
        bufs.append(dict(vis=vis, vis_out=vis, flags=flags, aterms=None, taper=torch.from_numpy(w.taper).to(dev),
                         grid=grid))
    n_vis = float(sum(w.n_vis for w in jobs))
    stream = torch.cuda.current_stream(dev)

    def plain_step():
        for p, b in zip(plans, bufs):
            b["grid"].zero_()
            idg.grid(p, b["vis"], b["flags"], None, b["taper"], b["grid"], stream)
            idg.degrid(p, b["grid"], b["flags"], None, b["taper"], b["vis_out"], stream)

    batch = idg.Batch(plans, bufs, graph=True)
    trials = batch.autotune(stream)             # the batch's own shapes per class (trials add into the grids)

    def batch_step():
        for b in bufs:
            b["grid"].zero_()
        batch.grid(stream)
        batch.degrid(stream)

    def timed(fn, n):
        for _ in range(max(3, warmup)):
            fn()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(n):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / n

    ms_plain = timed(plain_step, max(1, steps // 2))
    ms_batch = timed(batch_step, steps)
    info = batch.info()
    classes = {}
    for w, p in zip(jobs, plans):
        c = classes.setdefault(f"L{w.subgrid_size}", {"jobs": 0, "vis": 0, "separable_jobs": 0,
                                                      "separable_vis_fraction": 0.0})
        c["jobs"] += 1
        c["vis"] += int(w.n_vis)
        c["separable_jobs"] += int(p.stats.separable)
        # visibilities (planned) in subgrids that the separable kernels take
        c["separable_vis_fraction"] += p.stats.n_vis_sep
    for c in classes.values():
        c["separable_vis_fraction"] /= max(1, c["vis"])
    # per class: the plain per-job form of that class's jobs alone (grid + degrid)
    for name, c in classes.items():
        sel = [(p, b) for w, p, b in zip(jobs, plans, bufs) if f"L{w.subgrid_size}" == name]
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for p, b in sel:
            b["grid"].zero_()
            idg.grid(p, b["vis"], b["flags"], None, b["taper"], b["grid"], stream)
            idg.degrid(p, b["grid"], b["flags"], None, b["taper"], b["vis_out"], stream)
        e1.record(stream)
        torch.cuda.synchronize()
        c["plain_ms"] = e0.elapsed_time(e1)
        c["plain_mvis_per_s"] = c["vis"] / c["plain_ms"] / 1e3
    batch.destroy()
    return {"n_vis": int(n_vis), "work_items": info["n_items"], "work_classes": info["n_launches"],
            "plain_mvis_per_s": n_vis / ms_plain / 1e3, "batched_mvis_per_s": n_vis / ms_batch / 1e3,
            "plain_ms": ms_plain, "batched_ms": ms_batch, "batched_over_plain": ms_plain / ms_batch,
            "classes": classes, "plan_seconds": plan_s, "autotune_trial_ms": trials}


def run_batched(args, world, rank, local):
    """The uneven batch (config B): the same jobs gridded and degridded
    (a) one after another with idg_grid / idg_degrid (plain per-job form) and
    (b) as one batch: per subgrid size a separable and a direct work class, each
    one persistent launch or one tensor-core launch per job (programmatic
    dependent launches), subgrids kept in shared memory, the launch sequence
    replayed from a CUDA graph."""
    import torch
    from paper_1909_07226_gb300 import build as lib_build
    from paper_1909_07226_gb300 import idg
    from paper_1909_07226_gb300 import synthetic as syn

    torch.cuda.set_device(local)
    lib_build.build()
    idg.load()
    dev = torch.device("cuda", local)
    sampler = ClockSampler(local)
    sampler.start()
    args.jobs = args.jobs or 256
    r = batched_compare(idg, syn, torch, dev, args.jobs, args.steps, args.warmup)
    clocks = sampler.stop()
    rec = {
        "metric": "grid+degrid MVis/s (batched form vs plain per-job form)", "value": r["batched_mvis_per_s"],
        "unit": "MVis/s", "n_gpus": 1, "steps": args.steps, "warmup": max(3, args.warmup),
        "ms_per_step": r["batched_ms"], "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": DTYPE_MIXED, "data": "synthetic",
        "config": {"workload": f"Batched uneven: {args.jobs} snapshot jobs, U{{12..64}} stations, U{{64..1024}} t, "
                               f"U{{4..32}} ch of 0.2 MHz in 100-200 MHz, 0-20% flags, L in {{16,24,32}}, "
                               f"N in {{1024,2048,4096}}", "jobs": args.jobs, "n_vis": r["n_vis"],
                   "work_items": r["work_items"], "work_classes": r["work_classes"],
                   "graph": True, "l2": "inputs larger than L2, no flush"},
        "plain_per_job": {"value": r["plain_mvis_per_s"], "unit": "MVis/s", "ms_per_step": r["plain_ms"]},
        "batched_over_plain": r["batched_over_plain"], "classes": r["classes"],
        "clocks": clocks, "plan_seconds": r["plan_seconds"],
    }
    print(json.dumps(rec))


def run_serving(args, world, rank, local):
    """Serving (config S): a Poisson stream of requests drawn from the
    batched distribution ("cycle": 5 major cycles of degrid -> residual -> grid,
    "grid", "degrid"), served by the continuous-batching engine, and the same
    trace served one job at a time by the plain per-job form."""
    import torch
    from paper_1909_07226_gb300 import build as lib_build
    from paper_1909_07226_gb300 import idg, serving
    from paper_1909_07226_gb300 import synthetic as syn

    torch.cuda.set_device(local)
    lib_build.build()
    idg.load()
    args.jobs = args.jobs or 64
    wls = syn.make_batched_jobs(args.jobs, seed=1913)
    kinds = ("cycle", "grid", "degrid")
    sampler = ClockSampler(local)
    # warm up kernels, pools and graphs on a few jobs
    serving.Engine(budget_bytes=150 << 30).run(serving.make_trace(
        syn.make_batched_jobs(4, seed=7, scale_t=0.25), 1000.0, kinds, seed=7))
    torch.cuda.synchronize()
    sampler.start()
    points = []
    for rate in (args.rate, 4.0 * args.rate):
        eng = serving.Engine(budget_bytes=150 << 30, max_slots=32, graph=False)
        srv = eng.run(serving.make_trace(wls, rate, kinds))
        fifo = serving.run_plain_fifo(serving.make_trace(wls, rate, kinds))
        points.append({"rate_jobs_per_s": rate, "serving": srv, "plain_fifo": fifo,
                       "engine": {"iterations": eng.iterations, "max_active_jobs": eng.max_active,
                                  "host_batch_build_s": eng.host_batch_s}})
    clocks = sampler.stop()
    srv = points[0]["serving"]
    rec = {
        "metric": "grid+degrid MVis/s and latency (serving form vs plain per-job FIFO)",
        "value": srv["grid_degrid_mvis_per_s"],
        "unit": "MVis/s", "n_gpus": 1, "steps": 1, "warmup": 1, "ms_per_step": 1e3 * srv["makespan_s"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": DTYPE_MIXED, "data": "synthetic",
        "config": {"workload": f"Serving: Poisson arrivals, {args.jobs} requests from the batched "
                               f"distribution, kinds {list(kinds)} (uniform), 5 major cycles per cycle job, "
                               f"150 GB admission budget, 32 slots; rates {args.rate} and {4 * args.rate} jobs/s",
                   "jobs": args.jobs},
        "points": points, "clocks": clocks,
    }
    print(json.dumps(rec))


def run_precision(args, world, rank, local):
    """Precision forms (config P): the LOFAR-like workload with A-terms
    refreshed every 16 timesteps.  For every form: grid+degrid MVis/s on the
    full workload, and the error against the FP64 oracle of the full grid and of
    all visibilities on the first 256 timesteps (which the oracle redoes)."""
    import torch
    from oracle import oracle as O
    from paper_1909_07226_gb300 import build as lib_build
    from paper_1909_07226_gb300 import idg
    from paper_1909_07226_gb300 import synthetic as syn

    torch.cuda.set_device(local)
    lib_build.build()
    idg.load()
    O.build()
    forms = {"direct_sincos": dict(precision_mode=idg.PHASOR_SINCOS),
             "channel_recurrence": dict(precision_mode=idg.PHASOR_RECURRENCE),
             "direct_sincos+compensated_adder": dict(precision_mode=idg.PHASOR_SINCOS,
                                                     adder_mode=idg.ADDER_COMPENSATED),
             "channel_recurrence+compensated_adder": dict(precision_mode=idg.PHASOR_RECURRENCE,
                                                          adder_mode=idg.ADDER_COMPENSATED),
             "direct_sincos+tc_split_transform": dict(precision_mode=idg.PHASOR_SINCOS,
                                                      fft_mode=idg.FFT_TC_SPLIT),
             "direct_sincos+sorted_adder": dict(precision_mode=idg.PHASOR_SINCOS, adder_mode=idg.ADDER_SORTED)}
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    out = {}
    # accuracy on the slice, against the oracle
    sl = syn.make_lofar(with_vis=True, n_t=256, slot_len=16, name="precision")
    op = O.plan(sl)
    ref_grid = O.grid(sl, op)
    model_h = syn.random_grid(np.random.default_rng(7), op.n_w, sl.grid_size)
    ref_vis = O.degrid(sl, op, model_h)
    d_vis = torch.from_numpy(sl.vis).to(dev)
    d_at = torch.from_numpy(sl.aterms).to(dev)
    d_tp = torch.from_numpy(sl.taper).to(dev)
    d_model = torch.from_numpy(model_h).to(dev)
    for name, kw in forms.items():
        p = idg.plan_from_workload(sl, **kw)
        g = torch.zeros(ref_grid.shape, dtype=torch.complex64, device=dev)
        idg.grid(p, d_vis, None, d_at, d_tp, g, stream)
        v = torch.zeros(sl.vis.shape, dtype=torch.complex64, device=dev)
        idg.degrid(p, d_model, None, d_at, d_tp, v, stream)
        gg = g.cpu().numpy().astype(np.complex128)
        vv = v.cpu().numpy().astype(np.complex128)
        out[name] = {"grid_rel_rms": float(np.linalg.norm(gg - ref_grid) / np.linalg.norm(ref_grid)),
                     "grid_max_err_rel": float(np.max(np.abs(gg - ref_grid)) / np.max(np.abs(ref_grid))),
                     "vis_rel_rms": float(np.linalg.norm(vv - ref_vis) / np.linalg.norm(ref_vis)),
                     "vis_max_err_rel": float(np.max(np.abs(vv - ref_vis)) / np.max(np.abs(ref_vis)))}
        p.destroy()
    del d_vis, d_at, d_model
    # throughput on the full workload
    wl = syn.make_lofar(with_vis=True, slot_len=16, name="precision")
    vis = torch.from_numpy(wl.vis).to(dev)
    aterms = torch.from_numpy(wl.aterms).to(dev)
    taper = torch.from_numpy(wl.taper).to(dev)
    n_w = 1
    model = torch.from_numpy(syn.random_grid(np.random.default_rng(7), n_w, wl.grid_size)).to(dev)
    grid = torch.empty((n_w, wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device=dev)
    vis_out = torch.empty_like(vis)
    sampler = ClockSampler(local)
    sampler.start()
    n_sub = None
    direct_separable = False
    for name, kw in forms.items():
        p = idg.plan_from_workload(wl, **kw)
        n_sub = p.n_subgrids
        if name == "direct_sincos":
            direct_separable = bool(p.stats.separable)

        def step():
            grid.zero_()
            idg.grid(p, vis, None, aterms, taper, grid, stream)
            idg.degrid(p, model, None, aterms, taper, vis_out, stream)

        for _ in range(max(3, args.warmup)):
            step()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(args.steps):
            step()
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / args.steps
        out[name]["mvis_per_s"] = wl.n_vis / ms / 1e3
        out[name]["ms_per_step"] = ms
        # after the timed steps: one grid call under the library's per-kernel event profile
        idg.profile_enable(True)
        try:
            idg.profile_read(reset=True)
            grid.zero_()
            idg.grid(p, vis, None, aterms, taper, grid, stream)
            torch.cuda.synchronize()
            out[name]["grid_stage_ms"] = {k: round(v["ms"], 3) for k, v in idg.profile_read(reset=True).items()
                                          if v["launches"]}
        finally:
            idg.profile_enable(False)
        p.destroy()
    clocks = sampler.stop()
    best = max(out.values(), key=lambda r: r["mvis_per_s"])
    rec = {"metric": "grid+degrid MVis/s per precision form, with error vs the FP64 oracle",
           "value": out["direct_sincos"]["mvis_per_s"], "unit": "MVis/s", "n_gpus": 1, "steps": args.steps,
           "warmup": max(3, args.warmup), "ms_per_step": out["direct_sincos"]["ms_per_step"],
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": DTYPE_SEP if direct_separable else DTYPE_MIXED, "data": "synthetic",
           "config": {"workload": "Precision: LOFAR-like with A-terms every 16 timesteps (256 slots); accuracy on "
                                  "the first 256 timesteps against the FP64 oracle", "n_vis": int(wl.n_vis),
                      "n_subgrids": n_sub},
           "forms": out, "best_form_mvis_per_s": best["mvis_per_s"], "clocks": clocks}
    print(json.dumps(rec))


def run_case(args, local):
    """One small profiling case, run once after one warm-up: the block of the default
    line named by --case, on a workload sized for an ncu capture (a few GB on the
    device, inputs larger than L2).  Prints the case's own times."""
    import torch
    from paper_1909_07226_gb300 import build as lib_build
    from paper_1909_07226_gb300 import idg
    from paper_1909_07226_gb300 import synthetic as syn

    torch.cuda.set_device(local)
    lib_build.build()
    idg.load()
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream(dev)
    case = args.case
    if case == "classical":
        wl = syn.make_lofar(n_t=256, slot_len=16, name="precision")
    else:
        wl = syn.make_lofar(n_t=256)
    plan = idg.plan_from_workload(wl)
    vis = torch.from_numpy(wl.vis).to(dev)
    at = torch.from_numpy(wl.aterms).to(dev)
    tap = torch.from_numpy(wl.taper).to(dev)
    shape = (plan.n_w_layers, wl.grid_size, wl.grid_size, 4)
    model = torch.from_numpy(syn.random_grid(np.random.default_rng(7), plan.n_w_layers, wl.grid_size)).to(dev)
    grid = torch.zeros(shape, dtype=torch.complex64, device=dev)
    if case == "image":
        win, _ = idg.taper_window(wl.subgrid_size, float(wl.kernel_size), idg.TAPER_PSWF)
        img = torch.empty((wl.grid_size, wl.grid_size, 4), dtype=torch.complex64, device=dev)
        fns = [lambda: idg.image_from_grid(plan, model, win, img, stream),
               lambda: idg.grid_from_image(plan, img, win, grid, stream)]
    elif case == "classical":
        M = CLASSICAL_SUPPORT
        at_m = torch.from_numpy(syn.aterms_on_subgrid(wl.screens, M, wl.grid_size * wl.cell_size)
                                .astype(np.complex64)).to(dev)
        fns = [lambda: idg.classical_grid(plan, M, CLASSICAL_OVERSAMPLE, CLASSICAL_W_PLANE, vis, None, at_m, None,
                                          grid, stream)]
    elif case == "calibration":
        resid = torch.empty_like(vis)
        agrad = torch.zeros(at.shape, dtype=torch.complex64, device=dev)
        fns = [lambda: idg.aterm_gradient(plan, model, vis, None, at, tap, resid, agrad, None, stream)]
    elif case == "stages":
        n = plan.n_subgrids
        sub = torch.zeros((n, wl.subgrid_size, wl.subgrid_size, 4), dtype=torch.complex64, device=dev)
        idg.grid_subgrids(plan, 0, n, vis, None, at, tap, sub, stream)
        fns = [lambda: idg.add_subgrids(plan, 0, n, sub, grid, stream),
               lambda: idg.split_subgrids(plan, 0, n, grid, sub, stream)]
    else:                                   # lofar_slice: the composite calls the bench times
        vout = torch.empty_like(vis)
        fns = [lambda: idg.grid(plan, vis, None, at, tap, grid, stream),
               lambda: idg.degrid(plan, model, None, at, tap, vout, stream)]
    out = {}
    for rep in range(2):
        for i, fn in enumerate(fns):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn()
            e1.record(stream)
            torch.cuda.synchronize()
            out[f"call{i}_ms"] = e0.elapsed_time(e1)
    idg.device_errors(stream)
    print(json.dumps({"case": case, "n_subgrids": plan.n_subgrids, "n_vis": int(wl.n_vis), **out}))


def main():
    args = parse()
    world, rank, local = dist_setup(args)
    try:
        if args.impl == "reference":
            run_reference(args, world, rank)
        elif args.case:
            run_case(args, local)
        elif args.config == "batched":
            run_batched(args, world, rank, local)
        elif args.config == "serving":
            run_serving(args, world, rank, local)
        elif args.config == "precision":
            run_precision(args, world, rank, local)
        else:
            run_gb300(args, world, rank, local)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
