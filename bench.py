"""Throughput benchmark of the lock-exchange LBM step on GB300.

Workload (one bench step): 100 time steps of the 2048 x 128 x 256 lock-exchange
box, D3Q19 BGK-Smagorinsky + D3Q7 scalar, FP32 storage (H = x0 = 256,
u_b = 0.03, Re = 30000, Sc = 1, C_s = 0.17), followed by one diagnostics pass
(front, F_w, FP64 budgets) - the logging interval of the paper's runs.  The
state (7 GB) is far larger than L2, so no flush is needed between steps.

Prints one JSON line (rank 0): MNUPS over all ranks, the end-to-end figure
through host buffers, the HBM roofline of the step kernel, the FP64 oracle
timed on the host cores, side measurements (16-bit storage, cumulant model,
adjoint / forward ratio) and the SM clocks seen during the timed region.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

INNER = 100                     # time steps per bench step
WORKLOADS = {
    # the 67 M-node box the headline number is quoted on
    "config3": dict(nx=2048, ny=128, nz=256, H=256, x0=256, u_b=0.03, Re=30000.0),
    # a 4.2 M-node box (436 MB in FP32, larger than L2) for profiler captures
    "profile": dict(nx=512, ny=128, nz=64, H=64, x0=64, u_b=0.03, Re=30000.0 / 4),
}
WORKLOAD = dict(WORKLOADS["config3"])
def bytes_per_node(model="bgk", storage="fp32", scalar="q7") -> int:
    """Algorithmic bytes of one node update: every population read once and
    written once (AA in place), (Q + NS) populations of 4 or 2 bytes; with
    16-bit storage the scalar's rest population (D3Q7, D3Q27) is FP32."""
    q = 19 if model == "bgk" else 27
    ns = {"q7": 7, "q6": 6, "q27": 27}[scalar]
    if storage == "fp32":
        return (q + ns) * 2 * 4
    return (q + ns) * 2 * 2 + (4 if scalar != "q6" else 0)
PROFILE = os.path.join(ROOT, "profiles", "aa_step_bgk_fp32_traffic.md")
# the sources that define the headline step kernel (bgk_chain_kernel) and the plan
# of its launches, which decides its traffic
KERNEL_SOURCES = ["paper_2112_08479_gb300/csrc/lbm_aux.cu",
                  "paper_2112_08479_gb300/csrc/lbm_bgk.cu",
                  "paper_2112_08479_gb300/csrc/lbm_bgk_collide.cuh",
                  "paper_2112_08479_gb300/csrc/lbm_chain.cuh",
                  "paper_2112_08479_gb300/csrc/lbm_internal.h",
                  "paper_2112_08479_gb300/csrc/lbm_lanes.cuh",
                  "paper_2112_08479_gb300/csrc/lbm_pair.cuh",
                  "paper_2112_08479_gb300/csrc/lbm_common.cuh"]


def kernel_hash() -> str:
    h = hashlib.sha256()
    for s in KERNEL_SOURCES:
        with open(os.path.join(ROOT, s), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def profiled_traffic(nodes: int):
    """DRAM bytes (read + write) per time step from the committed ncu summary:
    of the captured launch divided by its steps when it ran on a box of `nodes`
    nodes, else the per-node figure scaled to `nodes`.  (None, why) when the
    kernel changed since the capture."""
    try:
        txt = open(PROFILE).read()
    except OSError:
        return None, "no profile"
    m = re.search(r"kernel_source_hash:\s*([0-9a-f]+)", txt)
    if not m or m.group(1) != kernel_hash():
        return None, "kernel changed since the capture"
    full = re.search(r"dram_bytes_per_(?:step|launch):\s*([0-9.eE+-]+)", txt)
    box = re.search(r"box_nodes:\s*([0-9]+)", txt)
    if full and box and int(box.group(1)) == nodes:
        return float(full.group(1)), "ncu capture of this box (per step of the captured launches)"
    b = re.search(r"dram_bytes_per_node_update:\s*([0-9.eE+-]+)", txt)
    if not b:
        return None, "no per-node figure"
    return float(b.group(1)) * nodes, "per-node figure of a smaller box scaled by nodes"


NOMINAL_HBM_GBS = 8000.0


def measured_peak_hbm():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


# ---------------------------------------------------------------------------
class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.fh = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=self.fh, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        self.t0 = self.t1 = None

    def mark_start(self):
        self.t0 = time.time()

    def mark_end(self):
        self.t1 = time.time()

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.3)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.flush()
        self.fh.seek(0)
        rows = [r.split(",") for r in self.fh.read().strip().splitlines() if r.strip()]
        os.unlink(self.fh.name)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                mhz = float(r[1]); mx = float(r[2]); pw = float(r[3])
            except (ValueError, IndexError):
                continue
            if pw > 300.0:  # under load
                sm.append(mhz)
                smax.append(mx)
                for name, v in zip(names, r[5:9]):
                    if v.strip().lower() == "active":
                        reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "samples_under_load": len(sm), "reasons": sorted(reasons)}


# ---------------------------------------------------------------------------
def dist_setup(backend=None):
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch
        import torch.distributed as dist
        backend = backend or ("nccl" if torch.cuda.is_available() else "gloo")
        if backend == "nccl":
            torch.cuda.set_device(local)
            dist.init_process_group(backend, device_id=torch.device("cuda", local))
        else:
            dist.init_process_group(backend)
    return ws, rank, local


def device_index(local: int) -> int:
    """GPU of this rank: LOCAL_RANK, or 0 when fewer GPUs than ranks exist
    (ranks sharing one GPU through host-staged gloo exchanges)."""
    import torch
    n = torch.cuda.device_count()
    return local if local < n else 0


def barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(v: float, ws: int) -> float:
    if ws == 1:
        return v
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([v], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---------------------------------------------------------------------------
def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def host_mem_available() -> int | None:
    """Bytes the process may still allocate: MemAvailable, bounded by the
    cgroup (v2) limit when one is set."""
    avail = None
    try:
        with open("/proc/meminfo") as fh:
            for line in fh:
                if line.startswith("MemAvailable:"):
                    avail = int(line.split()[1]) * 1024
    except OSError:
        pass
    try:
        lim = open("/sys/fs/cgroup/memory.max").read().strip()
        cur = int(open("/sys/fs/cgroup/memory.current").read().strip())
        if lim != "max":
            room = int(lim) - cur
            avail = room if avail is None else min(avail, room)
    except (OSError, ValueError):
        pass
    return avail


ORACLE_BYTES_PER_NODE = (19 + 7) * 8 * 2 + 8   # f, Phi and their post-collision copies, chi0


def oracle_box(nz_max: int | None = None):
    """The workload's lock-exchange box for the FP64 oracle (BGK-Smagorinsky
    D3Q19 + D3Q7), or its lower z-slab of nz_max layers when the full box does
    not fit in the host memory; returns (params, f, phi, nz)."""
    import oracle as O
    nx, ny, nz = WORKLOAD["nx"], WORKLOAD["ny"], WORKLOAD["nz"]
    avail = host_mem_available()
    if avail is not None:
        fit = int(0.6 * avail / (ORACLE_BYTES_PER_NODE * nx * ny))
        nz = max(2, min(nz, fit))
    if nz_max is not None:
        nz = max(2, min(nz, nz_max))
    u_b, H, Re = WORKLOAD["u_b"], WORKLOAD["H"], WORKLOAD["Re"]
    nu = u_b * H / Re
    p = O.OracleParams(nx, ny, nz, model=0, nu=nu, D=nu, cs_smag=0.17, gprime=u_b * u_b / H)
    f, phi = O.init(p, O.lock_chi0(nx, ny, nz, WORKLOAD["x0"], 1e-3, 2112))
    return p, f, phi, nz


def box_label(nz: int) -> str:
    nx, ny, full = WORKLOAD["nx"], WORKLOAD["ny"], WORKLOAD["nz"]
    if nz == full:
        return f"the full {nx}x{ny}x{full} workload box"
    return (f"the lower {nz} of {full} z-layers of the {nx}x{ny}x{full} workload box "
            "(host memory)")


def time_oracle(steps: int, threads: int, nz_max: int | None = None):
    """The FP64 C oracle as it stands (node loops on `threads` host threads)
    stepping the workload box (all lattice parameters of the workload) in
    place; returns (MNUPS, seconds, nz, threads used)."""
    import oracle as O
    O.build()
    used = O.set_threads(threads)
    p, f, phi, nz = oracle_box(nz_max)
    t = time.perf_counter()
    O.run_inplace(p, steps, f, phi)
    dt = time.perf_counter() - t
    return p.nx * p.ny * nz * steps / dt / 1e6, dt, nz, used


def oracle_baselines():
    """cpu_baseline of the GPU arm: the oracle on every host core over two
    time steps of the workload box, and on one thread over one step of a
    16-layer z-slab of it (about 10-30 s of CPU work together)."""
    cores = host_cores()
    v, dt, nz, used = time_oracle(2, cores)
    main = {"value": v, "unit": "MNUPS", "cores": used, "kind": "oracle",
            "sample": f"2 time steps of {box_label(nz)} (BGK-Smagorinsky D3Q19 + D3Q7, FP64, "
                      f"{used} threads), {dt:.1f} s"}
    v1, dt1, nz1, _ = time_oracle(1, 1, nz_max=16)
    single = {"value": v1, "unit": "MNUPS", "cores": 1, "kind": "oracle",
              "sample": f"1 time step of {box_label(nz1)} (FP64, single thread), {dt1:.1f} s"}
    return main, single


def run_reference(args, ws, rank):
    """Reference arm: the FP64 oracle as it stands on the host cores, one
    time step of the workload box per bench step (shrunk to a z-slab when
    the host memory or a few minutes of run time require it)."""
    if rank != 0:
        return
    import oracle as O
    O.build()
    cores = O.set_threads(host_cores())
    p, f, phi, nz = oracle_box()
    # bound the whole run to a few minutes: time one step first
    t = time.perf_counter()
    O.run_inplace(p, 1, f, phi)
    t1 = time.perf_counter() - t
    budget = 200.0
    total = args.steps + max(args.warmup - 1, 0)
    if t1 * total > budget:
        nz_s = max(2, int(nz * budget / (t1 * total)))
        del f, phi
        p, f, phi, nz = oracle_box(nz_s)
    for _ in range(max(args.warmup - 1, 0)):
        O.run_inplace(p, 1, f, phi)
    t = time.perf_counter()
    for _ in range(args.steps):
        O.run_inplace(p, 1, f, phi)
    dt = time.perf_counter() - t
    v = p.nx * p.ny * nz * args.steps / dt / 1e6
    cfg = config_dict(ws)
    if nz != WORKLOAD["nz"]:
        cfg["sample"] = box_label(nz)
    line = {"metric": "MNUPS (lattice node updates per second / 1e6), fused LBM step",
            "value": v, "unit": "MNUPS", "impl": "reference", "n_gpus": 0, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": cfg,
            "cpu_baseline": {"value": v, "unit": "MNUPS", "cores": cores, "kind": "oracle",
                             "sample": f"one time step of {box_label(nz)} per bench step "
                                       f"(BGK-Smagorinsky D3Q19 + D3Q7, FP64, {cores} threads)"},
            "e2e": {"value": v, "unit": "MNUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def config_dict(ws, model="bgk", storage="fp32", slabs=False, scalar="q7"):
    fluid = "D3Q19 BGK-Smagorinsky" if model == "bgk" else "D3Q27 cumulant"
    lat = {"q7": "D3Q7", "q6": "D3Q6", "q27": "D3Q27 FCM"}[scalar]
    return {"workload": f"lock-exchange {WORKLOAD['nx']}x{WORKLOAD['ny']}x{WORKLOAD['nz']}, "
                        f"{fluid} + {lat} scalar, {storage.upper()} storage, Re={WORKLOAD['Re']:g}, "
                        "100 steps + diagnostics per bench step",
            "nodes": WORKLOAD["nx"] * WORKLOAD["ny"] * WORKLOAD["nz"],
            "steps_per_bench_step": INNER,
            "parallelism": f"x-slabs x{ws} (one box, halo exchange)" if slabs else f"replicas x{ws}",
            "l2": "inputs larger than L2 (state >= 436 MB), no flush"}


# ---------------------------------------------------------------------------
def make_lattice(model="bgk", storage="fp32", scalar="q7", flags=0, **over):
    from paper_2112_08479_gb300 import lbm
    w = dict(WORKLOAD)
    w.update(over)
    p = lbm.lock_exchange(w["nx"], w["ny"], w["nz"], H=w["H"], x0=w["x0"], u_b=w["u_b"],
                          Re=w["Re"], model=model, storage=storage, scalar=scalar, flags=flags)
    return lbm.Lattice(p, device="cuda")


def step_launches(p, sms, n):
    """Step kernels that lbm_step launches for n steps of a whole box p (lbm_params)
    on a device of sms SMs: launches of several steps, then one per step left."""
    from paper_2112_08479_gb300 import lbm
    k = 0
    while n and (together := lbm.lbm_step_plan(p, sms, n)["steps"]):
        k, n = k + 1, n - together
    return k + n


def timed_loop(lat, steps, warmup, torch, inner=INNER, with_diag=True, kernel_events=True):
    """Returns (total seconds, mean step-kernel seconds, launches)."""
    s = lat.stream
    for _ in range(warmup):
        lat.step(inner)
        if with_diag:
            lat.diag()
    torch.cuda.synchronize()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(steps)]
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    t0.record(s)
    for k in range(steps):
        evs[k][0].record(s)
        lat.step(inner)
        evs[k][1].record(s)
        if with_diag:
            lat.diag()
    t1.record(s)
    torch.cuda.synchronize()
    total = t0.elapsed_time(t1) / 1e3
    kern = sum(a.elapsed_time(b) for a, b in evs) / 1e3 / (steps * inner)
    # (slabs step one by one)
    per_call = inner
    if getattr(lat, "peer", None) is None:
        sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
        per_call = step_launches(lat.params.c(), sms, inner)
    launches = steps * (per_call + (2 if with_diag else 0))
    return total, kern, launches


def side_variant(torch, model, storage, scalar="q7", steps=3, flags=0):
    lat = make_lattice(model, storage, scalar, flags=flags)
    total, kern, _ = timed_loop(lat, steps, 1, torch, with_diag=False)
    n = lat.N
    mnups = n / kern / 1e6
    gbs = bytes_per_node(model, storage, scalar) * n / kern / 1e9
    del lat
    torch.cuda.empty_cache()
    return {"mnups": mnups, "ms_per_time_step": kern * 1e3, "achieved_gbs": gbs}


def adjoint_ratio(torch, dims=(256, 32, 64), K=100, model="bgk", nseg=4, reps=2):
    """Forward step vs one reverse step on a lock-exchange box (default the
    256 x 32 x 64 differentiation box, H = nz, Re = 2000): the reverse sweep
    of the autograd backward (objective.reverse_sweep: recompute of each
    K-step segment from its checkpoint + adjoint steps, the next segment's
    recompute overlapped with the current sweep on a second stream) over
    nseg segments, and the same sweep without the overlap."""
    from paper_2112_08479_gb300 import lbm
    from paper_2112_08479_gb300.objective import reverse_sweep
    nx, ny, nz = dims
    p = lbm.lock_exchange(nx, ny, nz, H=nz, x0=nz, u_b=0.03, Re=2000.0, model=model)
    lat = lbm.Lattice(p, device="cuda")
    S = p.Q + p.NS
    s = lat.stream
    n = nseg * K
    lat.step(200)
    ckpts = torch.empty(nseg, S, p.N, device="cuda")
    lat.objective_forward(n, K, ckpts, None)
    lam = torch.zeros(S, p.N, device="cuda")
    tmp = torch.empty(S, p.N, device="cuda")
    dcs = torch.zeros(1, dtype=torch.float64, device="cuda")

    def fwd():
        lat.step(n)

    def rev():
        reverse_sweep(lat, ckpts, n, K, lam, tmp, dcs, 1.0, overlap=True)

    def rev_seq():
        reverse_sweep(lat, ckpts, n, K, lam, tmp, dcs, 1.0, overlap=False)

    out = {}
    for name, fn in (("forward", fwd), ("reverse", rev), ("reverse_sequential", rev_seq)):
        fn()
        torch.cuda.synchronize()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(s)
        for _ in range(reps):
            fn()
        b.record(s)
        torch.cuda.synchronize()
        out[name] = a.elapsed_time(b) / reps / n
    del lat, ckpts, lam, tmp
    torch.cuda.empty_cache()
    model_name = "BGK-Smagorinsky" if model == "bgk" else "cumulant"
    return {"workload": f"{nx}x{ny}x{nz} {model_name} FP32, {nseg} segments of K={K}",
            "fwd_ms_per_step": out["forward"], "adj_ms_per_step": out["reverse"],
            "ratio": out["reverse"] / out["forward"],
            "ratio_without_overlap": out["reverse_sequential"] / out["forward"]}


def run_ours(args, ws, rank, local):
    import torch
    from paper_2112_08479_gb300 import lbm
    lbm.load()
    local = device_index(local)
    torch.cuda.set_device(local)
    sampler = ClockSampler(torch.cuda.current_device() if ws == 1 else local)

    slabs = ws > 1 and args.decomp == "slab"
    if slabs:
        # one box cut into x-slabs, one per rank (strong scaling)
        from paper_2112_08479_gb300 import slab
        w = WORKLOAD
        p = lbm.lock_exchange(w["nx"], w["ny"], w["nz"], H=w["H"], x0=w["x0"], u_b=w["u_b"],
                              Re=w["Re"], model=args.model, storage=args.storage,
                              scalar=args.scalar)
        lat = slab.SlabLattice(p, rank, ws, device=f"cuda:{local}")
        nodes_total = p.N
    else:
        lat = make_lattice(args.model, args.storage, args.scalar)
        nodes_total = lat.N * ws
    N = lat.N
    barrier(ws)
    torch.cuda.synchronize()
    sampler.mark_start()
    total, kern, launches = timed_loop(lat, args.steps, args.warmup, torch)
    sampler.mark_end()
    barrier(ws)
    tmax = max_over_ranks(total, ws)
    value = nodes_total * INNER * args.steps / tmax / 1e6
    if slabs:
        # per bench step: each odd step is bracketed by two exchanges of a pack
        # and an unpack per touching face; the slab diagnostics add the
        # column maxima (2 launches) and the front of the gathered columns
        faces = sum(1 for f in (0, 1) if lat.peer[f] is not None)
        launches += args.steps * ((INNER // 2) * 2 * 2 * faces + 3)
    d = lat.diag()

    # end to end through the public API with host buffers: the step's scalar
    # field comes from pinned host memory, the diagnostics go back to the host
    import numpy as np
    lo, hi = (lat.local.x_offset, lat.local.x_offset + lat.local.nx) if slabs else (0, WORKLOAD["nx"])
    chi0 = torch.from_numpy(
        np.where(np.arange(lo, hi) < WORKLOAD["x0"], 1.0, 0.0).astype(np.float32)
    ).repeat(WORKLOAD["ny"] * WORKLOAD["nz"]).pin_memory()
    assert chi0.numel() == N
    s = lat.stream
    # each step's field is uploaded on a copy stream into one of two device
    # buffers while the previous step computes (the upload of step k + 1
    # overlaps step k; the first upload is inside the timed region)
    copy_stream = torch.cuda.Stream(device=s.device)
    bufs = [torch.empty(N, dtype=torch.float32, device=s.device) for _ in range(2)]
    done = [torch.cuda.Event(), torch.cuda.Event()]

    def upload(k):
        with torch.cuda.stream(copy_stream):
            bufs[k % 2].copy_(chi0, non_blocking=True)
            done[k % 2].record(copy_stream)

    def e2e_run(nsteps):
        upload(0)
        for k in range(nsteps):
            if k + 1 < nsteps:
                upload(k + 1)
            s.wait_event(done[k % 2])
            lat.set_scalar(bufs[k % 2])
            lat.step(INNER)
            lat.diag()                  # device -> host: the step's result

    e2e_run(max(1, args.warmup))
    torch.cuda.synchronize()
    barrier(ws)
    t0 = time.perf_counter()
    e2e_run(args.steps)
    torch.cuda.synchronize()
    e2e_t = max_over_ranks(time.perf_counter() - t0, ws)
    e2e = {"value": nodes_total * INNER * args.steps / e2e_t / 1e6, "unit": "MNUPS",
           "h2d_bytes_per_step": int(chi0.numel() * 4),
           "d2h_bytes_per_step": int(__import__("ctypes").sizeof(lbm.lbm_diagnostics))}
    clocks = sampler.stop()
    del lat
    torch.cuda.empty_cache()

    peak, peak_kind = measured_peak_hbm()
    bpn = bytes_per_node(args.model, args.storage, args.scalar)
    achieved = bpn * N / kern / 1e9
    headline = ((args.model, args.storage, args.scalar) == ("bgk", "fp32", "q7")
                and args.workload == "config3")
    shared = args.storage == "fp32" and args.scalar != "q27" and not slabs   # several steps a launch
    if args.storage == "fp32":
        kname = ("cumulant_step_kernel" if args.scalar == "q27"
                 else f"{args.model}_{'chain' if shared else 'pair'}_kernel")
    else:
        kname = "bgk_step2_kernel" if args.model == "bgk" else "cumulant_step_kernel"
        if args.scalar == "q7" and WORKLOAD["nx"] % 4 == 0:
            kname = f"{args.model}_even4_kernel + {kname}"
    traffic, tsrc = profiled_traffic(N) if headline else (None, "not captured for this variant")
    # a launch of several steps passes its state through HBM once per sweep of steps, so
    # frac (state bytes of every step over the copy rate) may exceed 1 and HBM is not
    # its bound; frac_dram has the bytes that ncu counted
    roof = {"bound": "latency and issue" if shared else "hbm",
            "kernel": f"{kname} (AA even/odd, {args.storage.upper()})",
            "achieved": achieved, "peak": peak, "peak_kind": peak_kind, "unit": "GB/s",
            "frac": achieved / peak, "traffic": traffic, "traffic_source": tsrc,
            "algorithmic_bytes_per_step": bpn * N, "mean_step_ms": kern * 1e3,
            # the same step time against the DRAM bytes ncu counted, and the
            # algorithmic rate against the nominal 8 TB/s of the part
            "achieved_dram": traffic / kern / 1e9 if traffic else None,
            "frac_dram": traffic / kern / 1e9 / peak if traffic else None,
            "frac_nominal": achieved / NOMINAL_HBM_GBS}

    extra = {}
    if rank == 0 and ws == 1 and not args.no_side and args.workload == "config3":
        variants = {}
        for model, storage, scalar in (("bgk", "fp16s", "q7"), ("bgk", "bf16s", "q7"),
                                       ("cumulant", "fp32", "q7"), ("cumulant", "fp16s", "q7"),
                                       ("cumulant", "bf16s", "q7"),
                                       ("bgk", "fp32", "q6"), ("cumulant", "fp32", "q27")):
            r = side_variant(torch, model, storage, scalar)
            r["hbm_frac"] = r.pop("achieved_gbs") / peak
            variants[f"{model}_{storage}" + ("" if scalar == "q7" else f"_{scalar}")] = r
        # the opt-in TMA-staged form of the cumulant FP16 step (bulk copies
        # through shared memory), for comparison with the default kernel
        from paper_2112_08479_gb300 import lbm as _l
        r = side_variant(torch, "cumulant", "fp16s", flags=_l.LBM_FLAG_TMA_STAGED)
        r["hbm_frac"] = r.pop("achieved_gbs") / peak
        variants["cumulant_fp16s_tma_staged"] = r
        extra["variants"] = variants
        extra["adjoint"] = adjoint_ratio(torch)
        extra["adjoint_cumulant"] = adjoint_ratio(torch, model="cumulant")
        extra["adjoint_1024x64x128"] = adjoint_ratio(torch, (1024, 64, 128), K=20, nseg=3, reps=1)
        extra["adjoint_cumulant_1024x64x128"] = adjoint_ratio(torch, (1024, 64, 128), K=20,
                                                             model="cumulant", nseg=3, reps=1)
    cpu = cpu1 = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        cpu, cpu1 = oracle_baselines()

    if rank == 0:
        line = {"metric": "MNUPS (lattice node updates per second / 1e6), fused LBM step",
                "value": value, "unit": "MNUPS", "n_gpus": ws, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": tmax / args.steps * 1e3,
                "higher_is_better": True, "scaling": "strong" if slabs else "weak",
                "vs_baseline": None,
                "dtype": "f32", "data": "synthetic (lock-exchange initial condition)",
                "config": config_dict(ws, args.model, args.storage, slabs, args.scalar), "e2e": e2e,
                "gpu_launches": launches,
                "roofline": roof, "cpu_baseline": cpu, "cpu_baseline_single_thread": cpu1,
                "clocks": clocks,
                "diag_at_end": {"front": d["front"], "Fw": d["Fw"], "step": d["step"]}}
        line.update(extra)
        print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-side", action="store_true", help="skip the side measurements")
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle timing")
    ap.add_argument("--workload", default="config3", choices=sorted(WORKLOADS))
    ap.add_argument("--model", default="bgk", choices=["bgk", "cumulant"])
    ap.add_argument("--storage", default="fp32", choices=["fp32", "fp16s", "bf16s"])
    ap.add_argument("--scalar", default="q7", choices=["q7", "q6", "q27"],
                    help="scalar lattice: D3Q7, D3Q6 (BGK only) or D3Q27 FCM (cumulant only)")
    ap.add_argument("--backend", default=None, choices=["nccl", "gloo"],
                    help="torch.distributed backend for N > 1 (default: nccl with GPUs)")
    ap.add_argument("--decomp", default="slab", choices=["slab", "replicas"],
                    help="N > 1: one box cut into x-slabs with a halo exchange (strong "
                         "scaling), or an independent box per rank (weak scaling)")
    ap.add_argument("--adjoint-only", default=None, metavar="NX,NY,NZ",
                    help="only time the adjoint sweep against the forward step on this "
                         "lock-exchange box (--model, --adjoint-k) and print it")
    ap.add_argument("--adjoint-k", type=int, default=100)
    args = ap.parse_args()
    if args.adjoint_only:
        import torch
        from paper_2112_08479_gb300 import lbm
        lbm.load()
        dims = tuple(int(v) for v in args.adjoint_only.split(","))
        print(json.dumps({"adjoint": adjoint_ratio(torch, dims, args.adjoint_k, args.model)}),
              flush=True)
        return
    WORKLOAD.clear()
    WORKLOAD.update(WORKLOADS[args.workload])
    ws, rank, local = dist_setup(args.backend)
    if args.impl == "reference":
        run_reference(args, ws, rank)
    else:
        run_ours(args, ws, rank, local)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
