#!/usr/bin/env python
"""SU3_Bench link multiply on GB300: HBM GB/s and site-updates/s at L=64.

One step = one pass of the operation c[i].link[j] = a[i].link[j] x b[j] over the whole L=64
lattice (16,777,216 sites, FP64 AoS, the paper's method and the benchmark's input format), one
su3_mult launch through the C ABI with a and c resident in HBM (19.3 GB per step, far larger than
the 129 MB L2, so no flush is needed). After the timed steps the same lattice is run in every
reduced form (FP32/FP16/BF16 storage, two-row, SoA/AoSoA) for the speedup-at-error table, the
batched 96-lattice workload, the end-to-end host-buffer path and the CPU oracle baseline.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl native|reference]

Under torchrun (N > 1) every rank runs its own L=64 lattice (replicas: sites are independent, no
data-path collective; weak scaling); only the timing uses a barrier and a max over ranks. With
--shard the ranks instead split ONE L=64 lattice into contiguous slabs of sites (strong scaling,
still without a data-path collective). The CPU baseline, the per-form, batched and adjacent-op legs
run at N = 1 only; at N > 1 the line carries the timed step and the end-to-end leg.
"""
import os

# The CPU oracle's OpenMP threads are pinned one per core, packed (set before any library starts
# an OpenMP runtime); with the default local allocation policy their first touch keeps the
# oracle's output on the NUMA node of the cores it runs on.
os.environ.setdefault("OMP_PROC_BIND", "close")
os.environ.setdefault("OMP_PLACES", "cores")
# the cores this process may use, read before an OpenMP runtime binds the main thread to one core
CPUS_ALLOWED = sorted(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else []

import argparse
import ctypes
import json
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "SU(3) link-mult HBM GB/s & site-updates/s at L=64 vs peak; low-prec speedup at error"
FLOP_PER_SITE = 864  # paper convention: 4 links x 27 complex MACs x (4 mul + 4 add)
SEED = 2103


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--L", type=int, default=64)
    ap.add_argument("--quick", action="store_true", help="headline only: no forms/batched/e2e/cpu legs")
    ap.add_argument("--arith", default="native", choices=["native", "f32pair", "hybrid"],
                    help="arithmetic of the FP64 AoS step (native = FP64 accuracy)")
    ap.add_argument("--dtype", default="f64", choices=["f64", "f32", "f16", "bf16"],
                    help="storage type of the timed step (other than f64: with --quick, for profiling)")
    ap.add_argument("--stride", type=int, default=0,
                    help="AoS site stride in bytes of the timed step's a and c, wider than the links "
                         "(640: the paper's padded FP64 Site); with --quick, for profiling")
    ap.add_argument("--form", default="",
                    help="with --quick: time this form alone, named as the tuner names forms "
                         "(dtype-repr-layout[-arith][-p<stride>], e.g. f64-2to18-aos-f32pair)")
    ap.add_argument("--shard", action="store_true",
                    help="N > 1: split one lattice into contiguous slabs of sites, one per rank (strong "
                         "scaling) instead of one lattice per rank (replicas, weak scaling)")
    ap.add_argument("--launch", default="",
                    help="launch configuration of the timed step instead of the tuned one, e.g. "
                         "block=256,tile_sites=64,stages=3,ctas_per_sm=2,threads_per_link=1")
    return ap.parse_args()


def parse_launch(text):
    """'k=v,k=v' -> dict of the su3_launch_cfg fields (ints); raises on unknown keys."""
    keys = ("block", "tile_sites", "stages", "ctas_per_sm", "native_permille", "threads_per_link")
    out = {}
    for item in filter(None, (t.strip() for t in text.split(","))):
        k, _, v = item.partition("=")
        if k not in keys:
            raise SystemExit("--launch: unknown field %r (fields: %s)" % (k, ", ".join(keys)))
        out[k] = int(v)
    return out


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d.get("hbm_gbs", 6800.0), d.get("sm_max_mhz", 2070.0), "measured"
    return 6800.0, 2070.0, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 100 ms while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        self.lines = []
        if self.proc:
            self.proc.terminate()
            out, _ = self.proc.communicate(timeout=10)
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in getattr(self, "lines", []):
            f = [x.strip() for x in l.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def flop_per_site(repr_in, repr_out):
    """Flops of one site update by the paper's count (8 per complex multiply-add): 864 for the
    full product, 576 for rows 0-1 only (two-row in and out), 1056 for two-row in, full out (the
    rebuilt row 2 of a adds 2 complex multiply-adds per element, 48 flops per link)."""
    import paper_2103_00571_gb300 as su3
    if repr_in == su3.FULL18:
        return FLOP_PER_SITE
    return 576 if repr_out == su3.TWOROW12 else FLOP_PER_SITE + 4 * 48


def slab(n_sites, world, rank):
    """Rank `rank`'s contiguous slab of one lattice split over `world` ranks: (first site, sites).
    Sizes differ by at most one site (the first n_sites % world ranks take one more), the slabs are
    disjoint and cover the lattice in rank order; sites are independent, so no rank needs another's
    data (the paper splits sites equally over threads, §Performance on Xeon)."""
    base, rem = divmod(n_sites, world)
    return rank * base + min(rank, rem), base + (1 if rank < rem else 0)


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        backend = "nccl" if args.impl == "native" else "gloo"
        if backend == "nccl":
            # each rank's GPU must be current before NCCL binds the process group to a device
            import torch
            torch.cuda.set_device(local)
        dist.init_process_group(backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch
        import torch.distributed as dist
        if dist.get_backend() == "nccl":
            dist.barrier(device_ids=[torch.cuda.current_device()])
        else:
            dist.barrier()


def max_over_ranks(x, world, device=None):
    """Max of a float over ranks (the whole job is as slow as its slowest rank)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---- the CPU baseline leg: the oracle, as it stands, on the host cores --------------------------

def _cpulist(text):
    out = set()
    for part in filter(None, text.strip().split(",")):
        lo, _, hi = part.partition("-")
        out.update(range(int(lo), int(hi or lo) + 1))
    return out


def host_info():
    """The host the CPU baseline runs on: CPU model, the cores this process may use, the NUMA
    nodes those cores belong to, and the OpenMP binding of the oracle's threads."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for l in out.splitlines():
            if l.startswith("Model name:"):
                model = l.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    if not model:
        try:
            with open("/proc/cpuinfo") as f:
                for l in f:
                    if l.lower().startswith(("model name", "cpu part")):
                        model = l.split(":", 1)[1].strip()
                        break
        except OSError:
            pass
    cpus = CPUS_ALLOWED
    nodes = []
    base = "/sys/devices/system/node"
    if os.path.isdir(base):
        for n in sorted(os.listdir(base)):
            if n.startswith("node") and n[4:].isdigit():
                try:
                    with open(os.path.join(base, n, "cpulist")) as f:
                        if _cpulist(f.read()) & set(cpus):
                            nodes.append(int(n[4:]))
                except OSError:
                    pass
    return {"cpu_model": model, "cpus_allowed": len(cpus), "numa_nodes_of_cpus": nodes,
            "omp_proc_bind": os.environ.get("OMP_PROC_BIND"), "omp_places": os.environ.get("OMP_PLACES"),
            "memory": "first touch by the pinned OpenMP threads under the default local allocation policy, "
                      "so pages land on the NUMA node(s) of those cores"}


def batched_refs(gen, oracle, n=96):
    """Oracle outputs of every lattice of the 96-lattice batch (part of the CPU-baseline leg: the
    batched leg's error report compares against them)."""
    ext = gen.extents(SEED, n)
    out = []
    for k in range(n):
        V = int(np.prod(ext[k]))
        out.append(oracle.mult(gen.sites(SEED, k, V), gen.bmat(SEED, k, V)))
    return out


def cpu_baseline_leg(a_host, b, V_sample, min_seconds=10.0):
    """Times the FP64 oracle (plain OpenMP loop over sites) on the first V_sample sites of the
    lattice, repeating passes until ~min_seconds of CPU work. Returns (summary, reference c of the
    sample) - the reference output is what the forms' error report compares against."""
    import oracle
    a = np.ascontiguousarray(a_host[: V_sample * 72])
    ref = oracle.mult(a, b)  # first touch of c and a warm pass
    t0 = time.perf_counter()
    passes = 0
    while True:
        oracle.mult(a, b)
        passes += 1
        el = time.perf_counter() - t0
        if el >= min_seconds:
            break
    gbs = 1152.0 * V_sample * passes / el / 1e9
    cores = oracle.threads()
    # one core, shorter sample (the paper's strong-scaling baseline point)
    oracle.set_threads(1)
    t1 = time.perf_counter()
    n1 = 0
    while time.perf_counter() - t1 < 2.0:
        oracle.mult(a[: 65536 * 72], b)
        n1 += 1
    el1 = time.perf_counter() - t1
    oracle.set_threads(cores)
    # references of the adjacent operations on the same sample, for their error report
    v = np.linspace(-0.5, 0.5, 24)
    extra = {"an": oracle.mult_an(a, b), "na": oracle.mult_na(a, b), "v": v,
             "mv": oracle.mat_vec(a, v), "mv_adj": oracle.mat_vec(a, v, adjoint=True)}
    import su3_inputs as gen
    extra["batched"] = batched_refs(gen, oracle)
    summary = {"value": round(gbs, 3), "unit": "GB/s", "cores": cores, "kind": "oracle", "host": host_info(),
               "one_core_GBps": round(1152.0 * 65536 * n1 / el1 / 1e9, 3),
               "site_updates_per_s": round(V_sample * passes / el, 1),
               "sample": "%d sites (the first %d of the L=64 lattice) x %d passes, %.1f s, FP64, plain C "
                         "OpenMP loop over sites (the paper's VersionX form)" % (V_sample, V_sample, passes, el)}
    return summary, ref, extra


def run_reference(args, world, rank):
    """--impl reference: the oracle timed on the host cores, each step a bounded sample."""
    if rank != 0:
        return
    import oracle
    import su3_inputs as gen
    V = args.L ** 4
    Vs = min(V, 1 << 20)
    a = gen.sites(SEED, 0, V, first_site=0, count=Vs)
    b = gen.bmat(SEED, 0, V)
    for _ in range(args.warmup):
        oracle.mult(a, b)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.mult(a, b)
    el = time.perf_counter() - t0
    gbs = 1152.0 * Vs * args.steps / el / 1e9
    line = {"impl": "reference", "metric": METRIC, "value": round(gbs, 3), "unit": "GB/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(el / args.steps * 1e3, 3),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "L=64 FP64 AoS SU3_Bench link multiply; each reference step is a bounded "
                                   "sample of %d sites of it" % Vs, "lattice": "%d^4" % args.L, "seed": SEED},
            "site_updates_per_s": round(Vs * args.steps / el, 1),
            "cpu_baseline": {"value": round(gbs, 3), "unit": "GB/s", "cores": oracle.threads(), "kind": "oracle",
                             "sample": "%d sites per step x %d steps" % (Vs, args.steps)},
            "e2e": {"value": round(gbs, 3), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---- the GPU legs -------------------------------------------------------------------------------

LAST_LAUNCH_MS = []  # per-launch times of the most recent time_launches call


def time_launches(h, torch, fn, n, stream):
    """Per-launch CUDA events on the launching stream; returns (total ms, mean ms per launch)."""
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n)]
    first = torch.cuda.Event(enable_timing=True)
    last = torch.cuda.Event(enable_timing=True)
    first.record(stream)
    for e0, e1 in evs:
        e0.record(stream)
        fn()
        e1.record(stream)
    last.record(stream)
    last.synchronize()
    per = [e0.elapsed_time(e1) for e0, e1 in evs]
    LAST_LAUNCH_MS[:] = per
    return first.elapsed_time(last), sum(per) / len(per)


def traffic_record():
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(p):
        return {}
    with open(p) as f:
        return json.load(f)


# the sources that define the single-lattice AoS kernels (the ones the traffic records describe)
AOS_KERNEL_SOURCES = ("su3_device.cuh", "su3_internal.h", "su3_stream.cuh", "su3_stream.cu", "su3_stream_padded.cu")


def code_only(text):
    """C/C++/CUDA source with comments removed and whitespace runs collapsed (string and character
    literals kept as they are), so that editing a comment leaves the digest alone."""
    out, i, n = [], 0, len(text)
    while i < n:
        c = text[i]
        if c in "\"'":  # a literal: copy it through its closing quote, honouring escapes
            j = i + 1
            while j < n and text[j] != c:
                j += 2 if text[j] == "\\" else 1
            out.append(text[i:j + 1])
            i = j + 1
        elif text.startswith("//", i):
            i = text.find("\n", i)
            i = n if i < 0 else i
        elif text.startswith("/*", i):
            j = text.find("*/", i + 2)
            i = n if j < 0 else j + 2
            out.append(" ")
        else:
            out.append(c)
            i += 1
    return " ".join("".join(out).split())


def source_digest():
    """Digest of the AoS kernels' code (comments and layout ignored): a traffic record taken under
    another digest is stale."""
    import hashlib
    d = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2103_00571_gb300", "csrc")
    for n in AOS_KERNEL_SOURCES:
        with open(os.path.join(csrc, n), encoding="utf-8") as f:
            d.update((n + "\n" + code_only(f.read())).encode())
    return d.hexdigest()[:16]


FORMS = [
    # name, dtype, repr_in, repr_out, layout[, arith]
    ("f64-f32pair-aos", 0, 0, 0, 0, 1), ("f64-f32pair-aosoa32", 0, 0, 0, 1, 1), ("f64-f32pair-2row-aos", 0, 1, 1, 0, 1),
    ("f32-aos", 1, 0, 0, 0), ("f16-aos", 2, 0, 0, 0), ("bf16-aos", 3, 0, 0, 0),
    ("f64-2row-aos", 0, 1, 1, 0), ("f32-2row-aos", 1, 1, 1, 0), ("f16-2row-aos", 2, 1, 1, 0),
    ("f64-2row-to-full-aos", 0, 1, 0, 0), ("f64-f32pair-2row-to-full-aos", 0, 1, 0, 0, 1),
    ("f64-soa", 0, 0, 0, 2), ("f32-soa", 1, 0, 0, 2), ("f16-soa", 2, 0, 0, 2),
    ("f64-aosoa32", 0, 0, 0, 1), ("f32-aosoa32", 1, 0, 0, 1), ("bf16-aosoa32", 3, 0, 0, 1),
]
TOL = {(0, 0): 1e-13, (0, 1): 1e-12, (1, 0): 2e-6, (1, 1): 5e-6, (2, 0): 5e-3, (2, 1): 5e-3, (3, 0): 3e-2,
       (3, 1): 3e-2}


def run_native(args, world, rank, local):
    import torch

    import paper_2103_00571_gb300 as su3
    import su3_inputs as gen
    from paper_2103_00571_gb300 import tune
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    h = su3.Handle(local)
    tuned = tune.apply_cached(h)
    hbm_peak, sm_max, peak_src = peaks()
    L = args.L
    V_lattice = L ** 4
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    if args.shard:  # one lattice (id 0), this rank's slab of it
        first, V = slab(V_lattice, world, rank)
        lattice_id, sites_all = 0, V_lattice
    else:  # one lattice per rank
        first, V = 0, V_lattice
        lattice_id, sites_all = rank, world * V_lattice
    stream = torch.cuda.current_stream()

    # inputs: this rank's sites, generated on the host into pinned memory (also the e2e source)
    a_host = torch.empty(V * 72, dtype=torch.float64, pin_memory=True)
    gen.sites(SEED, lattice_id, V_lattice, first_site=first, count=V, out=a_host.numpy())
    b = gen.bmat(SEED, lattice_id, V_lattice)
    a_dev = a_host.to(dev)
    c_dev = torch.empty_like(a_dev)
    if (args.dtype != "f64" or args.stride or args.form) and not args.quick:
        raise SystemExit("--dtype other than f64, --stride and --form time that form alone: use them with --quick")
    if args.form:  # any form the tuner names; its storage type, arithmetic and stride replace the flags
        d64, dc = tune.parse_pair(args.form, V)
        args.dtype = {su3.F64: "f64", su3.F32: "f32", su3.F16: "f16", su3.BF16: "bf16"}[d64.dtype]
        args.arith = {su3.NATIVE: "native", su3.F32PAIR: "f32pair", su3.HYBRID: "hybrid"}[d64.arith]
        args.stride = d64.site_stride_bytes
    arith = {"native": su3.NATIVE, "f32pair": su3.F32PAIR, "hybrid": su3.HYBRID}[args.arith]
    dt = {"f64": su3.F64, "f32": su3.F32, "f16": su3.F16, "bf16": su3.BF16}[args.dtype]
    if not args.form:
        d64 = su3.Desc(dt, su3.FULL18, su3.AOS, V, args.stride, arith if dt == su3.F64 else su3.NATIVE)
        dc = d64
    a_step, c_step = a_dev, c_dev
    if args.form or dt != su3.F64 or args.stride:
        a_step = torch.empty(su3.array_bytes(d64), dtype=torch.uint8, device=dev)
        c_step = torch.empty(su3.array_bytes(dc), dtype=torch.uint8, device=dev)
        h.pack(a_dev, d64, a_step, stream)
    if args.launch:
        h.set_launch_cfg_for(d64, dc, **parse_launch(args.launch))
    step = lambda: h.mult(d64, a_step, b, dc, c_step, stream)  # noqa: E731

    for _ in range(args.warmup):
        step()
    h.sync(stream)
    n_before = h.launch_count()
    barrier(world)
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        total_ms, per_launch_ms = time_launches(h, torch, step, args.steps, stream)
        torch.cuda.synchronize()
    launch_ms = sorted(LAST_LAUNCH_MS)
    barrier(world)
    h.sync(stream)
    launches = h.launch_count() - n_before
    total_ms = max_over_ranks(total_ms, world, dev)
    site_bytes = float(su3.site_update_bytes(dt, d64.repr, dc.repr))
    bytes_per_step = site_bytes * V
    value = sites_all * site_bytes * args.steps / (total_ms * 1e-3) / 1e9
    sups = sites_all * args.steps / (total_ms * 1e-3)
    clocks = clk.summary()

    # roofline of the dominant kernel (the FP64 AoS kernel is the whole step); its template's
    # threads per link: 1, or 3 when the launch splits links into rows
    tpl = 3 if h.get_launch_cfg_for(d64, dc)["threads_per_link"] == 3 else 1
    # An upper bound of the FP64 product's rate, TFLOP/s by the paper's count: its wide multiply-adds (18 for
    # an output real, five or six of a row's six) back to back at 32 per clock and SM, the FP64 pipe's share
    # beside them. The other integer instructions share the multiply-adds' issue, so it cannot be reached.
    flop_site = flop_per_site(d64.repr, dc.repr)
    rows_site = 12 if dc.repr == su3.FULL18 else 8
    fp64_peak = sms * 32 * flop_site / (18 * (5 if d64.repr == dc.repr else 6) * rows_site) * sm_max * 1e6 / 1e12
    fp64_share = 1 / 6 if d64.repr == dc.repr else 192 / flop_site  # of the flops, on the FP64 pipe
    achieved_tf = flop_site * V / (per_launch_ms * 1e-3) / 1e12
    achieved_gbs = bytes_per_step / (per_launch_ms * 1e-3) / 1e9
    try:  # the FP64 pipe's sustained rate, measured on this device by a diagnostic FMA kernel
        fp64_measured = h.measure_fp64_rate(8192)
    except su3.Su3Error:
        fp64_measured = None
    pad = ",p%d" % args.stride if args.stride else ""  # padded sites: the kernel of their own
    padded = "true" if args.stride else "false"
    ops = "%d,%d" % (9 if d64.repr == su3.FULL18 else 6, 3 if dc.repr == su3.FULL18 else 2)  # elements in, rows out
    if args.form and (d64.repr, dc.repr) != (su3.FULL18, su3.FULL18):
        pad = ",%s" % args.form  # no traffic record is kept for the two-row forms
    tr = traffic_record().get("su3_aos_kernel<f64,full%s>" % pad, {})
    traffic = None
    if tr and tr.get("source_digest") == source_digest():
        traffic = tr["bytes_per_site"] * V
    hbm_roof = {"achieved": round(achieved_gbs, 1), "peak": hbm_peak, "unit": "GB/s",
                "frac": round(achieved_gbs / hbm_peak, 4), "peak_source": peak_src + " hbm_gbs"}
    if dt != su3.F64:
        tr = traffic_record().get("su3_aos_kernel<%s,full%s>" % (args.dtype, pad), {})
        traffic = tr["bytes_per_site"] * V if tr and tr.get("source_digest") == source_digest() else None
        roofline = dict(hbm_roof, bound="hbm", traffic=traffic,
                        kernel="su3_aos_kernel<NativeOp<%s,%s>, %d, AOS, %s>" % (args.dtype.upper(), ops, tpl, padded))
    elif args.arith == "native":
        roofline = {"bound": "alu", "achieved": round(achieved_tf, 4), "peak": round(fp64_peak, 4),
                    "unit": "TFLOP/s", "frac": round(achieved_tf / fp64_peak, 4), "traffic": traffic,
                    "kernel": "su3_aos_kernel<NativeOp<F64,%s>, %d, AOS, %s>" % (ops, tpl, padded),
                    "peak_source": "%d SMs (this device) x %.0f MHz (max SM clock) x 32 wide multiply-adds/clk, 18 for an "
                                   "output real in fixed point; an upper bound: the other integer instructions share "
                                   "their issue" % (sms, sm_max),
                    "peak_measured": round(fp64_measured, 4) if fp64_measured else None,
                    "frac_of_measured": round(achieved_tf * fp64_share / fp64_measured, 4) if fp64_measured else None,
                    "peak_measured_source": "the FP64 pipe alone, and the share of the flops that it does (one output "
                                            "real of six, or row 2's rebuild) against it: su3_measure_fp64_rate, 8 "
                                            "independent DFMA chains per thread, 2,048 threads per SM, CUDA events",
                    "arithmetic": "FP64 FMAs, and 61-bit fixed point with one rounding (half the error on random SU(3))",
                    "hbm": hbm_roof}
    else:
        tr = traffic_record().get("su3_aos_kernel<f64,full,%s%s>" % (args.arith, pad), {})
        traffic = tr["bytes_per_site"] * V if tr and tr.get("source_digest") == source_digest() else None
        roofline = dict(hbm_roof, bound="hbm", traffic=traffic,
                        kernel="su3_aos_kernel<%s<%s>, %d, AOS, %s>" % ("PairF64Op" if args.arith == "f32pair" else "HybridF64Op", ops,
                                                                            tpl, padded))

    line = {"metric": METRIC, "value": round(value, 2), "unit": "GB/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(total_ms / args.steps, 4), "higher_is_better": True,
            "scaling": "strong" if args.shard else "weak", "vs_baseline": None,
            "dtype": ({"native": "f64", "f32pair": "f32x2 (FP64 storage)", "hybrid": "f64 + f32x2"}[args.arith]
                      if dt == su3.F64 else "%s storage, f32 math" % args.dtype),
            "data": "synthetic",
            "config": {"workload": "L=%d %s AoS SU3_Bench link multiply (c[i][j] = a[i][j] x b[j], "
                                   "%d sites, %d B read + %d B written per site)%s%s"
                                   % (L, args.dtype.upper(), V_lattice, 4 * su3.link_bytes(dt, d64.repr),
                                      4 * su3.link_bytes(dt, dc.repr),
                                      ", split into %d slabs of contiguous sites" % world if args.shard else "",
                                      ", sites padded to %d B (links only are read and written)" % args.stride
                                      if args.stride else ""),
                       "lattice": "%d^4" % L,
                       "form": args.form or ((("f64-full18-aos-" + args.arith) if dt == su3.F64 else args.dtype + "-full18-aos")
                                             + ("-p%d" % args.stride if args.stride else "")),
                       "seed": SEED,
                       "inputs": "random SU(3) (Gram-Schmidt on Gaussian rows), one lattice per GPU",
                       "l2": "inputs larger than L2 (%.1f GB touched per step vs 129 MB L2): no flush"
                             % (bytes_per_step / 1e9),
                       "launch_cfg": h.get_launch_cfg_for(d64, dc), "tuned": bool(tuned) and not args.launch,
                       "parallelism": ("slab shards" if args.shard else "replicas") if world > 1 else "single GPU",
                       "sms": sms},
            "site_updates_per_s": round(sups, 1),
            "gflops": round(flop_site * sups / 1e9, 2),
            "roofline": roofline, "gpu_launches": launches, "clocks": clocks,
            "launch_ms": {"mean": round(per_launch_ms, 4), "median": round(launch_ms[len(launch_ms) // 2], 4),
                          "min": round(launch_ms[0], 4), "max": round(launch_ms[-1], 4)}}

    if world == 1 and not args.quick:
        # CPU baseline leg (oracle, as it stands, on the host cores; bounded sample) and the
        # per-form legs: single-GPU runs only, so that N > 1 holds its GPUs for the timed step alone
        V_sample = min(V, 1 << 20)
        cpu, ref, extra = cpu_baseline_leg(a_host.numpy(), b, V_sample)
        line["cpu_baseline"] = cpu
        # speedup at error of every form on the same lattice
        line["forms"] = forms_leg(h, torch, su3, a_dev, b, V, stream, value, ref, V_sample, hbm_peak=hbm_peak)
        line["paper_site640"] = site640_leg(h, torch, su3, a_dev, b, V, stream, ref, V_sample)
        line["adjacent_ops"] = adjacent_leg(h, torch, su3, a_dev, b, V, stream, extra, V_sample)
        fp64_err = sample_error(torch, c_dev, ref, V_sample)
        line["forms"]["f64-aos-" + args.arith] = {"GBps": round(value / world, 1), "site_updates_per_s": round(sups / world, 1),
                                    "speedup_vs_f64": 1.0, "max_err": fp64_err[0], "rms_err": fp64_err[1],
                                    "tol": 1e-13, "ok": fp64_err[0] <= 1e-13}
        # the fastest FP64-accurate form (FP64 in and out, within the FP64 tolerance) beside the
        # plain method's headline: FP64 storage with FP32-pair arithmetic, AoS
        fa = line["forms"].get("f64-f32pair-aos")
        if fa:
            tr = traffic_record().get("su3_aos_kernel<f64,full,f32pair>", {})
            line["fp64_accurate"] = {
                "form": "f64-f32pair-aos", "GBps": fa["GBps"], "site_updates_per_s": fa["site_updates_per_s"],
                "speedup_vs_f64": fa["speedup_vs_f64"], "max_err": fa["max_err"], "tol": fa["tol"], "ok": fa["ok"],
                "roofline": {"bound": "hbm", "achieved": fa["GBps"], "peak": hbm_peak, "unit": "GB/s",
                             "frac": round(fa["GBps"] / hbm_peak, 4), "peak_source": peak_src + " hbm_gbs",
                             "traffic": tr["bytes_per_site"] * V if tr and tr.get("source_digest") == source_digest() else None,
                             "kernel": "su3_aos_kernel<PairF64Op<9,3>, 1, AOS, false>"}}
    if not args.quick:
        line["e2e"] = e2e_leg(h, torch, su3, a_host, b, V, args, stream, world, dev, a_dev, c_dev, sites_all)
        if world == 1:
            line["batched"] = batched_leg(h, torch, su3, gen, extra["batched"])
    elif rank == 0:
        line["e2e"] = None
    if rank == 0:
        line["summary"] = summary(line)  # last key: the compact digest ends the line
        print(json.dumps(line), flush=True)
    h.close()


def summary(line):
    """The line's key figures in about 1.3 kB: the headline with both roofline fractions, the
    fastest FP64-accurate form, every form as [GB/s, G site/s, max error] and whether all are
    within their tolerances, the paper's 640-byte Site, the batch and the end-to-end path."""
    rf = line["roofline"]
    out = {"headline": {"form": line["config"]["form"], "GBps": line["value"],
                        "Gsite_per_s": round(line["site_updates_per_s"] / 1e9, 3),
                        "frac": rf["frac"], "bound": rf["bound"],
                        "hbm_frac": rf.get("hbm", {}).get("frac", rf["frac"] if rf["bound"] == "hbm" else None)}}
    fa = line.get("fp64_accurate")
    if fa:
        out["fp64_accurate"] = {"form": fa["form"], "GBps": fa["GBps"], "hbm_frac": fa["roofline"]["frac"],
                                "max_err": float("%.3g" % fa["max_err"]), "tol": fa["tol"], "ok": fa["ok"]}
    if "forms" in line:
        out["forms"] = {n: [round(f["GBps"]), round(f["site_updates_per_s"] / 1e9, 2), float("%.2g" % f["max_err"])]
                        for n, f in line["forms"].items()}
        out["forms_within_tol"] = all(f["ok"] for f in line["forms"].values())
    p640 = line.get("paper_site640")
    if p640:
        out["site640_Gsite_per_s"] = {k: round(v["site_updates_per_s"] / 1e9, 2) for k, v in p640.items()}
    bt = line.get("batched")
    if bt:
        out["batched"] = {n: [bt[n]["ms"], round(bt[n]["site_updates_per_s"] / 1e9, 3), bt[n]["ok"]]
                          for n in ("graph_persistent", "graph_persistent_f64_as_f32pair", "per_lattice_loop")
                          if n in bt}
    e2e = line.get("e2e")
    if e2e:
        out["e2e"] = {"GBps": e2e["value"], "path": e2e.get("path"), "vs_copies_only": e2e.get("vs_copies_only"),
                      "matches_device_step": e2e.get("matches_device_step")}
    cpu = line.get("cpu_baseline")
    if cpu:
        out["cpu_oracle_GBps"] = cpu["value"]
    return out


def sample_error(torch, c_dev_f64, ref, V_sample):
    got = c_dev_f64[: V_sample * 72].cpu().numpy()
    d = np.abs(got - ref)
    return float(d.max()), float(np.sqrt(np.mean(d * d)))


def forms_leg(h, torch, su3, a_dev, b, V, stream, f64_gbs, ref, V_sample, reps=10, hbm_peak=None):
    """Every reduced form on the same lattice: site-updates/s, algorithmic GB/s, speedup over the
    FP64 kernel and error against the oracle; plus the form's pack (FP64 AoS -> form) and unpack
    (form -> FP64 AoS) throughput, which stay outside the timed step."""
    out = {}
    f64_sups = f64_gbs * 1e9 / 1152.0
    scratch = torch.empty(V * 72, dtype=torch.float64, device=a_dev.device)  # unpack target
    for name, dt, ri, ro, lay, *ar in FORMS:
        arith = ar[0] if ar else 0
        da = su3.Desc(dt, ri, lay, V, 0, arith)
        dc = su3.Desc(dt, ro, lay, V, 0, arith)
        abuf = torch.empty(su3.array_bytes(da), dtype=torch.uint8, device=a_dev.device)
        cbuf = torch.empty(su3.array_bytes(dc), dtype=torch.uint8, device=a_dev.device)
        h.pack(a_dev, da, abuf, stream)
        fn = lambda: h.mult(da, abuf, b, dc, cbuf, stream)  # noqa: E731
        for _ in range(3):
            fn()
        h.sync(stream)
        total, per = time_launches(h, torch, fn, reps, stream)
        h.sync(stream)
        sups = V / (per * 1e-3)
        gbs = su3.site_update_bytes(dt, ri, ro) * sups / 1e9
        # pack and unpack of this form, timed apart from the step (3 launches each)
        _, pack_ms = time_launches(h, torch, lambda: h.pack(a_dev, da, abuf, stream), 3, stream)
        _, unpack_ms = time_launches(h, torch, lambda: h.unpack(dc, cbuf, scratch, stream), 3, stream)
        h.sync(stream)
        # error on the CPU-baseline sample (first V_sample sites), vs the oracle; the last unpack
        # left the whole lattice in FP64 AoS
        c64 = scratch[: V_sample * 72]
        err = sample_error(torch, c64, ref, V_sample)
        tol = TOL[(dt, 1 if (ri == 1 and ro == 1) or (ri == 1) else 0)]
        out[name] = {"GBps": round(gbs, 1), "site_updates_per_s": round(sups, 1),
                     "speedup_vs_f64": round(sups / f64_sups, 3), "max_err": err[0], "rms_err": err[1],
                     "tol": tol, "ok": err[0] <= tol, "ms": round(per, 4), "launch_cfg": h.get_launch_cfg_for(da, dc),
                     "pack_GBps": round((576 * V + su3.array_bytes(da)) / (pack_ms * 1e-3) / 1e9, 1),
                     "unpack_GBps": round((su3.array_bytes(dc) + 576 * V) / (unpack_ms * 1e-3) / 1e9, 1)}
        if hbm_peak:
            out[name]["hbm_frac"] = round(gbs / hbm_peak, 4)  # of the measured HBM copy peak
        if arith == su3.F32PAIR:
            out[name]["note"] = ("FP64 in, FP64 out, arithmetic in FP32 pairs: input magnitudes below 2^-74 "
                                 "(zeros included) act as values below 2^-73, so b = I gives c == a only "
                                 "to within 1e-22 rather than bit for bit")
        del abuf, cbuf
        torch.cuda.empty_cache()
    return out


def site640_leg(h, torch, su3, a_dev, b, V, stream, ref, V_sample, reps=10):
    """The paper's own FP64 Site: 4 links plus coordinates, index, parity and padding to 640 bytes
    (§Background), so a site update moves 2 x 640 B by the paper's accounting while the kernel
    reads and writes only the 576 link bytes of each site (2-D tensor copies of whole tiles)."""
    d = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V, 640)
    abuf = torch.empty(su3.array_bytes(d), dtype=torch.uint8, device=a_dev.device)
    cbuf = torch.zeros_like(abuf)
    h.pack(a_dev, d, abuf, stream)
    res = {}
    for arith, name in ((su3.NATIVE, "native"), (su3.F32PAIR, "f32pair")):
        dd = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V, 640, arith)
        fn = lambda: h.mult(dd, abuf, b, dd, cbuf, stream)  # noqa: E731
        for _ in range(3):
            fn()
        h.sync(stream)
        _, per = time_launches(h, torch, fn, reps, stream)
        sups = V / (per * 1e-3)
        c64 = torch.empty(V_sample * 72, dtype=torch.float64, device=a_dev.device)
        h.unpack(su3.Desc(su3.F64, su3.FULL18, su3.AOS, V_sample, 640), cbuf, c64, stream)
        h.sync(stream)
        err = sample_error(torch, c64, ref, V_sample)
        res[name] = {"site_updates_per_s": round(sups, 1), "paper_GBps_2x640B": round(1280 * sups / 1e9, 1),
                     "link_GBps_1152B": round(1152 * sups / 1e9, 1), "ms": round(per, 4), "max_err": err[0],
                     "tol": 1e-13, "ok": err[0] <= 1e-13}
    del abuf, cbuf
    torch.cuda.empty_cache()
    return res


def adjacent_leg(h, torch, su3, a_dev, b, V, stream, extra, V_sample, reps=10):
    """a b^dagger, a^dagger b, a v and a^dagger v over the same lattice (AOS), FP64 and FP32:
    site-updates/s, algorithmic GB/s (link bytes read + output bytes written) and error."""
    res = {}
    vec = torch.empty(V * 24, dtype=torch.float64, device=a_dev.device)
    for dt, dname, arith in ((su3.F64, "f64", su3.NATIVE), (su3.F64, "f64-f32pair", su3.F32PAIR),
                             (su3.F32, "f32", su3.NATIVE)):
        rb = 8 if dt == su3.F64 else 4
        d = su3.Desc(dt, su3.FULL18, su3.AOS, V, 0, arith)
        abuf = a_dev if dt == su3.F64 else torch.empty(su3.array_bytes(d), dtype=torch.uint8, device=a_dev.device)
        if dt != su3.F64:
            h.pack(a_dev, d, abuf, stream)
        cbuf = torch.empty(su3.array_bytes(d), dtype=torch.uint8, device=a_dev.device)
        wbuf = torch.empty(V * 24 * rb, dtype=torch.uint8, device=a_dev.device)
        cases = [("a_bdag", lambda: h.mult_op(su3.OP_NA, d, abuf, b, d, cbuf, stream), 72 * rb, "na"),
                 ("adag_b", lambda: h.mult_op(su3.OP_AN, d, abuf, b, d, cbuf, stream), 72 * rb, "an"),
                 ("a_v", lambda: h.mat_vec(d, abuf, extra["v"], wbuf, False, stream), 24 * rb, "mv"),
                 ("adag_v", lambda: h.mat_vec(d, abuf, extra["v"], wbuf, True, stream), 24 * rb, "mv_adj")]
        for name, fn, out_bytes, key in cases:
            for _ in range(3):
                fn()
            h.sync(stream)
            _, per = time_launches(h, torch, fn, reps, stream)
            h.sync(stream)
            sups = V / (per * 1e-3)
            if key in ("na", "an"):
                c64 = torch.empty(V_sample * 72, dtype=torch.float64, device=a_dev.device)
                h.unpack(su3.Desc(dt, su3.FULL18, su3.AOS, V_sample), cbuf, c64, stream)
                h.sync(stream)
                got = c64.cpu().numpy()
            else:
                raw = wbuf[: V_sample * 24 * rb].cpu().numpy()
                got = raw.view(np.float64 if rb == 8 else np.float32).astype(np.float64)
            diff = np.abs(got - extra[key])
            tol = 1e-13 if dt == su3.F64 else 2e-6
            res["%s-%s-aos" % (dname, name)] = {
                "site_updates_per_s": round(sups, 1), "GBps": round((72 * rb + out_bytes) * sups / 1e9, 1),
                "ms": round(per, 4), "max_err": float(diff.max()), "tol": tol, "ok": bool(diff.max() <= tol)}
        del cbuf, wbuf
        if dt != su3.F64:
            del abuf
    del vec
    torch.cuda.empty_cache()
    return res


def cudart():
    """The CUDA runtime library the process already uses (libsu3 links it), for plain copies."""
    for name in ("libcudart.so.13", "libcudart.so.12", "libcudart.so"):
        try:
            rt = ctypes.CDLL(name)
        except OSError:
            continue
        rt.cudaMemcpyAsync.restype = ctypes.c_int
        rt.cudaMemcpyAsync.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int,
                                       ctypes.c_void_p]
        return rt
    return None


def e2e_leg(h, torch, su3, a_host, b, V, args, stream, world, dev, a_dev=None, c_dev=None, sites_all=None):
    """The same step through the host-buffer entry point with pinned a and c: every byte of a
    crosses the host link to the GPU and every byte of c back inside the timed region (libsu3 takes
    its direct path: the kernel streams both over the link). For context, each step is followed by
    the same bytes moved by plain concurrent copies with no kernel, timed separately (what the link
    gives at that moment), and the staged path (chunked copies through HBM) is timed afterwards, as
    is the default path on ordinary (unpinned) arrays: direct where the device reads pageable host
    memory coherently, staged elsewhere."""
    d64 = su3.Desc(su3.F64, su3.FULL18, su3.AOS, V)
    c_host = torch.empty(V * 72, dtype=torch.float64, pin_memory=True)
    h.mult_host(d64, a_host.data_ptr(), b, d64, c_host.data_ptr(), stream)  # warm (staging buffers)
    k = max(3, min(args.steps, 5))
    rt = cudart()
    copies = a_dev is not None and c_dev is not None and rt is not None
    s_in, s_out = (torch.cuda.Stream(), torch.cuda.Stream()) if copies else (None, None)
    ring = torch.empty(3 * (64 << 20), dtype=torch.uint8, device=dev) if copies else None
    el = cel = 0.0
    barrier(world)
    for _ in range(k):
        t0 = time.perf_counter()
        h.mult_host(d64, a_host.data_ptr(), b, d64, c_host.data_ptr(), stream)
        el += time.perf_counter() - t0
        if copies:
            # the same bytes through plain copies and no kernel: a's sites H2D and back D2H into
            # c_host in 64 MB pieces through a 3-slot device ring, on two streams ordered by events
            # (the staged path's copy pattern; raw cudaMemcpyAsync, since torch's copy_ of these
            # pinned tensors measured far below the link)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            piece = 64 << 20
            done_in = [torch.cuda.Event() for _ in range(3)]
            done_out = [torch.cuda.Event() for _ in range(3)]
            for i, off in enumerate(range(0, V * 576, piece)):
                slot = i % 3
                n = ctypes.c_size_t(min(piece, V * 576 - off))
                buf = ctypes.c_void_p(ring.data_ptr() + slot * piece)
                if i >= 3:
                    s_in.wait_event(done_out[slot])
                rt.cudaMemcpyAsync(buf, ctypes.c_void_p(a_host.data_ptr() + off), n, 1, ctypes.c_void_p(s_in.cuda_stream))
                done_in[slot].record(s_in)
                s_out.wait_event(done_in[slot])
                rt.cudaMemcpyAsync(ctypes.c_void_p(c_host.data_ptr() + off), buf, n, 2, ctypes.c_void_p(s_out.cuda_stream))
                done_out[slot].record(s_out)
            torch.cuda.synchronize()
            cel += time.perf_counter() - t0
    path = {su3.HOST_DIRECT: "direct", su3.HOST_STAGED: "staged"}.get(h.last_host_path(), "none")
    el = max_over_ranks(el, world, dev)
    sites_all = world * V if sites_all is None else sites_all
    gbs = 1152.0 * sites_all * k / el / 1e9
    out = {"value": round(gbs, 2), "unit": "GB/s", "h2d_bytes_per_step": 576 * V, "d2h_bytes_per_step": 576 * V,
           "steps": k, "ms_per_step": round(el / k * 1e3, 3), "path": path,
           "api": "su3_mult_host with pinned host a and c: the direct path (the kernel streams a in and c out "
                  "over the host link, no staging copies)" if path == "direct" else
                  "su3_mult_host (host a and c; chunked H2D / kernel / D2H overlapped on 3 streams)"}
    if copies:
        cel = max_over_ranks(cel, world, dev)
        out["copies_only_GBps"] = round(1152.0 * sites_all * k / cel / 1e9, 2)
        out["vs_copies_only"] = round(gbs / out["copies_only_GBps"], 3)
    if c_dev is not None and args.arith == "native":
        # the timed path's result (the copies above reused c_host, so it is computed once more) on
        # 65,536 sampled sites, bit for bit against the device-resident step's c (same arithmetic)
        h.mult_host(d64, a_host.data_ptr(), b, d64, c_host.data_ptr(), stream)
        idx = np.sort(np.random.default_rng(1).choice(V, min(V, 65536), replace=False))
        got = c_host.view(V, 72)[torch.from_numpy(idx)].numpy()
        want = c_dev.view(V, 72)[torch.from_numpy(idx).to(c_dev.device)].cpu().numpy()
        out["matches_device_step"] = bool(np.array_equal(got, want))
    # for context: the same calls forced through the staged (chunked copy) path
    h.set_host_path(su3.HOST_STAGED)
    try:
        t0 = time.perf_counter()
        for _ in range(2):
            h.mult_host(d64, a_host.data_ptr(), b, d64, c_host.data_ptr(), stream)
        sel = max_over_ranks(time.perf_counter() - t0, world, dev)
    finally:
        h.set_host_path(su3.HOST_AUTO)
    out["staged_path_GBps"] = round(1152.0 * sites_all * 2 / sel / 1e9, 2)
    # ordinary pageable a and c (no pinning): on a device that reads pageable host memory
    # coherently through the host's page tables, the default path streams them as they stand; the
    # pages are touched on the host first, as an application's own arrays would be (single-GPU
    # runs only: at N > 1 the ranks' extra host copies would add up to hundreds of GB)
    if world > 1:
        del c_host
        return out
    a_page = a_host.numpy().copy()
    c_page = np.zeros_like(a_page)
    h.mult_host(d64, a_page, b, d64, c_page, stream)  # warm
    barrier(world)
    t0 = time.perf_counter()
    for _ in range(2):
        h.mult_host(d64, a_page, b, d64, c_page, stream)
    pel = max_over_ranks(time.perf_counter() - t0, world, dev)
    out["pageable"] = {"GBps": round(1152.0 * sites_all * 2 / pel / 1e9, 2),
                       "path": {su3.HOST_DIRECT: "direct", su3.HOST_STAGED: "staged"}.get(h.last_host_path(), "none"),
                       "device_reads_pageable_memory": h.pageable_host_access(),
                       "same_bits_as_pinned": bool(np.array_equal(c_page, c_host.numpy()))}
    del a_page, c_page
    del c_host
    return out


def batched_leg(h, torch, su3, gen, refs, reps=20):
    """96 lattices, extents uniform over {4, 6, ..., 24}, FP64 (even) / FP32 (odd): one persistent
    launch replayed from a CUDA graph vs a loop of per-lattice su3_mult launches. After each
    variant's timing every lattice's whole output is compared with the oracle's (`refs`): the max
    error per storage type, against 1e-13 (FP64, native or in FP32 pairs) and 2e-6 (FP32)."""
    ext = gen.extents(SEED, 96)
    items, keep, per = [], [], []
    total_sites = 0
    for k in range(96):
        V = int(np.prod(ext[k]))
        total_sites += V
        dt = su3.F64 if k % 2 == 0 else su3.F32
        d = su3.Desc(dt, su3.FULL18, su3.AOS, V)
        a64 = torch.from_numpy(gen.sites(SEED, k, V)).cuda()
        abuf = torch.empty(su3.array_bytes(d), dtype=torch.uint8, device="cuda")
        h.pack(a64, d, abuf)
        cbuf = torch.empty_like(abuf)
        bk = gen.bmat(SEED, k, V)
        keep += [abuf, cbuf]
        items.append(su3.BatchItem(d, abuf.data_ptr(), cbuf.data_ptr(), (ctypes.c_double * 72)(*bk)))
        per.append((d, abuf, bk, cbuf))
    s = torch.cuda.current_stream()

    def batched():
        h.mult_batched(items, s, use_graph=True)

    def loop():
        for d, abuf, bk, cbuf in per:
            h.mult(d, abuf, bk, d, cbuf, s)

    # the same batch with its FP64 lattices in FP32-pair arithmetic
    items_pair = []
    for it in items:
        d = it.desc
        dp = su3.Desc(d.dtype, d.repr, d.layout, d.n_sites, d.site_stride_bytes,
                      su3.F32PAIR if d.dtype == su3.F64 else su3.NATIVE)
        items_pair.append(su3.BatchItem(dp, it.a_dev, it.c_dev, it.b))

    def batched_pair():
        h.mult_batched(items_pair, s, use_graph=True)

    res = {}
    for name, fn in (("graph_persistent", batched), ("per_lattice_loop", loop),
                     ("graph_persistent_f64_as_f32pair", batched_pair)):
        for _ in range(3):
            fn()
        h.sync(s)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(s)
        for _ in range(reps):
            fn()
        e1.record(s)
        e1.synchronize()
        ms = e0.elapsed_time(e1) / reps
        res[name] = {"ms": round(ms, 4), "site_updates_per_s": round(total_sites / (ms * 1e-3), 1)}
        h.sync(s)
        errs = {"f64": 0.0, "f32": 0.0}
        for k, (d, abuf, bk, cbuf) in enumerate(per):
            o = torch.empty(d.n_sites * 72, dtype=torch.float64, device="cuda")
            h.unpack(d, cbuf, o, s)
            h.sync(s)
            diff = np.abs(o.cpu().numpy() - refs[k])
            key = "f64" if d.dtype == su3.F64 else "f32"
            errs[key] = max(errs[key], float(np.nan_to_num(diff, nan=np.inf).max()))
            cbuf.fill_(0xFF)  # NaN bytes: the next variant must rewrite every output
        res[name]["max_err"] = errs
        res[name]["ok"] = errs["f64"] <= 1e-13 and errs["f32"] <= 2e-6
    h.sync(s)
    res["speedup"] = round(res["per_lattice_loop"]["ms"] / res["graph_persistent"]["ms"], 3)
    res["lattices"] = 96
    res["total_sites"] = total_sites
    res["batched_cfg"] = h.get_batched_cfg()
    return res


def main():
    args = parse()
    world, rank, local = dist_setup(args)
    if args.impl == "reference":
        run_reference(args, world, rank)
    else:
        run_native(args, world, rank, local)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
