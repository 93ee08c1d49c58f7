#!/usr/bin/env python
"""Benchmark of the RPA hot path on GB300.

Default workload (slab): a step is one whole RPA correlation-energy job of
the slab dual-grid workload (complex128, coarse 3x3x1 q-grid without Gamma
plus 4 near-Gamma points, dense 6x6x1 K_reg = 12 q x 36 k pairs, N_aux = 768,
N_occ = 32, N_virt = 480, 16 imaginary frequencies): chi0 for every
(q, omega), the V side, the Cholesky log-det and the quadrature, through the
C ABI (rpa_energy) with inputs resident in HBM.  The mixed (split-precision
chi0) path is timed, and one step of the plain FP64 path is timed beside it
with |dE_c| and the per-term error between the two; a short Poisson stream
of served jobs gives the p50/p99 latency beside it.  Prints one JSON line.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--prec fp64|mixed]
    python bench.py --workload periodic2d  # the 2-D periodic job (4x4x1, N_aux 512, 20 frequencies)
    python bench.py --workload batch     # 64 uneven instances per step (rpa_energy_batch)
    python bench.py --workload serving   # Poisson stream of jobs (rpa_submit), p50/p99 latency
    python bench.py --workload periodic2d-ao  # the same job given as PADF + MO coefficients
    python bench.py --impl reference ... # the CPU oracle as reference arm

Under torchrun (N > 1) every rank runs its own job on its own GPU (weak
scaling, no collective on the data path); rank 0 prints.  With --q-shard one
job is split over the ranks by q-blocks instead (strong scaling, one
all-reduce of the integrand table per job).
"""
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

T_START = time.perf_counter()


def log(msg):
    """Progress note on stderr (stdout carries only the JSON line)."""
    sys.stderr.write("[bench %7.1f s] %s\n" % (time.perf_counter() - T_START, msg))
    sys.stderr.flush()


METRIC = "χ0 TFLOP/s & E_c jobs/s, mixed vs FP64 at |ΔE_c|≤1µHa; p50/p99 job latency"
FP64_PEAK_TFLOPS = 152 * 4 * 2.070e9 / 1e12  # 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz = 1.259


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--prec", default="auto", choices=["auto", "fp64", "mixed"])
    ap.add_argument("--slices", type=int, default=0,
                    help="BF16 digit slices of the mixed path (2-4; 0: library default)")
    ap.add_argument("--chi0-freq", type=int, default=0, choices=[0, 1, 2],
                    help="mixed chi0: 0 frequency-batched when it saves work (library default), 1 every frequency "
                         "contracted, 2 always frequency-batched")
    ap.add_argument("--cap-gb", type=float, default=0.0,
                    help="periodic2d/slab: the context's HBM cap (bounds the workspace; profiling small cases)")
    ap.add_argument("--n-q", type=int, default=0, help="profiling only: restrict the job to its first n q-points")
    ap.add_argument("--tail-case", action="store_true",
                    help="profiling only: the job's q-points, N_aux and frequencies (the V side and log-det "
                         "launches at full shape) with N_occ 4, N_virt 24 and, for slab, a 3x3x1 k-grid")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--q-shard", action="store_true",
                    help="periodic2d/slab: one job split over the ranks by q-blocks (strong scaling) instead of "
                         "one job per rank")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--workload", default="slab", choices=["periodic2d", "slab", "batch", "serving",
                                                                   "periodic2d-ao"])
    ap.add_argument("--lat-jobs", type=int, default=40,
                    help="periodic2d/slab: jobs of the short served stream whose p50/p99 latency joins the line "
                         "(0: none)")
    ap.add_argument("--no-fp64", action="store_true", help="periodic2d: skip the FP64 comparison step")
    ap.add_argument("--n-inst", type=int, default=64, help="batch: instances per step")
    ap.add_argument("--ao-scale", type=int, default=1,
                    help="periodic2d-ao, profiling only: divide basis, fit, occupied and virtual counts by this")
    ap.add_argument("--ao-projector", type=float, default=0.0,
                    help="periodic2d-ao: regularise the MO coefficients with the periodic projector at this eps_d")
    ap.add_argument("--ao-lattice", type=int, default=0,
                    help="periodic2d-ao: give the PADF coefficients per lattice vector (|a|,|b| <= this) instead "
                         "of per k-point; the library forms the lattice sums")
    ap.add_argument("--serve-jobs", type=int, default=200, help="serving: jobs in the stream")
    ap.add_argument("--serve-load", type=float, default=0.8, help="serving: arrival rate / measured capacity")
    ap.add_argument("--serve-cap-gb", type=float, default=120.0, help="serving: HBM admission cap")
    return ap.parse_args()


def workload(n_q=0, name="periodic2d", tail_case=False):
    from paper_2505_06021_gb300 import synth

    if tail_case:  # the job's q-points, N_aux and frequencies with a tiny C (profiling the tail)
        p = (synth.config2(n_occ=4, n_virt=24, k_dims=(3, 3, 1)) if name == "slab" else
             synth.config1(n_occ=4, n_virt=24))
    else:
        p = synth.config2() if name == "slab" else synth.config1()
    if n_q:
        g = p.grid
        g.pair_k, g.pair_kq, g.w_q = g.pair_k[:n_q], g.pair_kq[:n_q], g.w_q[:n_q]
        g.qpts = g.qpts[:n_q]
    return p


def config_of(p, prec, n_q_override, name="periodic2d", tail_case=False):
    if name == "slab":
        desc = ("slab-dual-c128: slab dual k-grid, complex128, coarse 3x3x1 q-grid without Gamma + 4 near-Gamma "
                "points, dense 6x6x1 K_reg (12 q x 36 k pairs), N_aux=%d, N_occ=%d, N_virt=%d, %d imaginary "
                "frequencies" % (p.n_aux, p.n_occ, p.n_virt, p.n_w))
    else:
        desc = ("periodic2d-c128: 2-D periodic, complex128, 4x4x1 k and q grids (16 q x 16 k pairs), "
                "N_aux=%d, N_occ=%d, N_virt=%d, %d imaginary frequencies" % (p.n_aux, p.n_occ, p.n_virt, p.n_w))
    return {
        "workload": desc + ("" if not n_q_override else " [first %d q only: profiling case]" % n_q_override) +
                    (" [tail profiling case: N_occ %d, N_virt %d, %d k per q]" % (p.n_occ, p.n_virt, p.n_k)
                     if tail_case else ""),
        "n_q": p.n_q, "n_k": p.n_k, "n_aux": p.n_aux, "n_occ": p.n_occ, "n_virt": p.n_virt, "n_w": p.n_w,
        "chi0_prec": prec,
        "l2": "inputs larger than L2 (C alone is %.1f GB per job vs 129 MB L2)" % (p.c_bytes() / 1e9),
        "parallelism": "one job per GPU (weak scaling)",
    }


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.th = threading.Thread(target=self._read, daemon=True)
            self.th.start()
        except Exception:
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
        except Exception:
            self.proc.kill()
        self.th.join(timeout=2)
        sm, mx, reasons, pw = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
                pw.append(float(f[3]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm), "power_w_max": max(pw) if pw else None}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist

        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist

        dist.barrier()


def allreduce_max(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist

    t = torch.tensor([x], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def allreduce_sum(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist

    t = torch.tensor([x], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def oracle_terms(p, name):
    """The (q, omega) terms the oracle samples on the large workloads: 2-D
    periodic q in {Gamma, 5} x omega in {0, 10, 19}; slab dual grid q in
    {first regular, first near-Gamma} x omega in {0, 8, 15}."""
    import numpy as np

    if name == "slab":
        ng = np.asarray(p.grid.near_gamma, bool)
        qs = [int(np.argmin(ng)), int(np.argmax(ng))]
        ws = [0, p.n_w // 2, p.n_w - 1]
    else:
        qs = [0, min(5, p.n_q - 1)]
        ws = [0, p.n_w // 2, p.n_w - 1]
    return [(q, w) for q in qs for w in ws]


class OracleSampler:
    """Times the oracle as it stands (the plain FP64 definition, OpenMP over
    rows) on the host cores.  V(q)^1/2 (single-threaded Jacobi) is formed once
    per sampled q, outside the sampled steps; a step is one (q, omega) term of
    the stated subset with its chi0 over one k-pair (the pairs cycle from step
    to step), then the sandwich and the Cholesky log-det of the full N x N
    matrices.  A whole job is extrapolated as
    n_q T_vhalf + n_q n_w (n_k T_chi0(one pair) + T_tail)."""

    def __init__(self, p, name, n_vhalf=None):
        import oracle

        oracle.build()
        self.p, self.terms = p, oracle_terms(p, name)
        self.threads = oracle.max_threads()
        self.Vh, self.vhalf_s = {}, []
        qs = sorted(set(q for q, _ in self.terms))
        for q in qs[:n_vhalf] if n_vhalf else qs:
            t0 = time.perf_counter()
            self.Vh[q] = oracle.vhalf(p.V(q))
            self.vhalf_s.append(time.perf_counter() - t0)
        self.terms = [(q, w) for q, w in self.terms if q in self.Vh]
        self._C = {}
        self.chi_s, self.tail_s = [], []

    def step(self, i):
        import oracle

        p = self.p
        q, w = self.terms[i % len(self.terms)]
        j = (i // len(self.terms)) % p.n_k
        if (q, j) not in self._C:
            self._C[(q, j)] = p.C(q, j)
        eo, ev = p.eps_pair(q, j)
        t0 = time.perf_counter()
        chi = oracle.chi0([self._C[(q, j)]], [eo], [ev], p.grid.zeta_k, float(p.omega[w]))
        t1 = time.perf_counter()
        Pi = oracle.sandwich(self.Vh[q], chi)
        oracle.logdet(Pi)
        t2 = time.perf_counter()
        self.chi_s.append(t1 - t0)
        self.tail_s.append(t2 - t1)
        return t2 - t0

    def job_s(self):
        p = self.p
        return (p.n_q * statistics.median(self.vhalf_s) +
                p.n_q * p.n_w * (p.n_k * statistics.median(self.chi_s) + statistics.median(self.tail_s)))

    def record(self):
        js = self.job_s()
        return {"value": 1.0 / js, "unit": "jobs/s", "cores": self.threads, "kind": "oracle",
                "sample": "terms %s (q, w) of the job, each step chi0 over one k-pair (pairs cycling) + V^1/2 "
                          "sandwich + Cholesky log-det at full N, OpenMP over rows; V(q)^1/2 Jacobi once per sampled "
                          "q (single thread, outside the steps); whole job extrapolated as n_q*T_vhalf + "
                          "n_q*n_w*(n_k*T_chi0_pair + T_tail)" % self.terms,
                "extrapolated_job_s": js, "vhalf_s": statistics.median(self.vhalf_s),
                "chi0_one_pair_s": statistics.median(self.chi_s), "tail_s": statistics.median(self.tail_s),
                "steps_sampled": len(self.chi_s)}


def gpu_local_cpus(dev_index):
    """CPUs of the NUMA node the GPU hangs off (from sysfs), restricted to the
    ones this process may use; (node, cpus) or (None, None) if unknown."""
    try:
        out = subprocess.run(["nvidia-smi", "-i", str(dev_index), "--query-gpu=pci.bus_id", "--format=csv,noheader"],
                             capture_output=True, text=True, timeout=20).stdout.strip()
        dom, bus, rest = out.split(":")
        addr = "%04x:%s:%s" % (int(dom, 16), bus.lower(), rest.lower())
        node = int(open("/sys/bus/pci/devices/%s/numa_node" % addr).read().strip())
        if node < 0:
            return None, None
        cpus = set()
        for part in open("/sys/devices/system/node/node%d/cpulist" % node).read().strip().split(","):
            a, _, b = part.partition("-")
            cpus.update(range(int(a), int(b or a) + 1))
        cpus &= os.sched_getaffinity(0)
        return (node, cpus) if cpus else (node, None)
    except Exception:
        return None, None


class near_gpu:
    """Runs the enclosed host allocations (pinning, first touch) on the CPUs of
    the GPU's NUMA node, so that pinned inputs are local to the GPU's host link."""

    def __init__(self, dev_index):
        self.node, self.cpus = gpu_local_cpus(dev_index)

    def __enter__(self):
        self.saved = os.sched_getaffinity(0)
        if self.cpus:
            os.sched_setaffinity(0, self.cpus)
        return self

    def __exit__(self, *a):
        os.sched_setaffinity(0, self.saved)


def traffic_for(kernel_key):
    """DRAM bytes per launch of `kernel_key` from the committed ncu summary,
    valid only while the sources it names (the kernel, and the planner that
    shapes its launches) are unchanged (hash recorded)."""
    import hashlib

    path = os.path.join(ROOT, "profiles", "traffic.txt")
    if not os.path.exists(path):
        return None
    src = os.path.join(ROOT, "paper_2505_06021_gb300", "csrc")
    for line in open(path):
        f = dict(kv.split("=", 1) for kv in line.split() if "=" in kv)
        if f.get("kernel") != kernel_key:
            continue
        # source: one file, or several joined by '+' (hash of their concatenation)
        blob = b"".join(open(os.path.join(src, name), "rb").read() for name in f["source"].split("+"))
        h = hashlib.sha256(blob).hexdigest()[:16]
        if h != f.get("sha"):
            return None
        return float(f["bytes_per_launch_full"])
    return None


def run_reference(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    name = args.workload if args.workload in ("periodic2d", "slab") else "slab"
    p = workload(0, name)
    smp = OracleSampler(p, name)
    for i in range(args.warmup):
        smp.step(i)
    smp.chi_s, smp.tail_s = [], []
    step_s = [smp.step(args.warmup + i) for i in range(args.steps)]
    rec = smp.record()
    val = rec["value"]
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": "jobs/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * statistics.median(step_s),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded, shapes of the paper's periodic workloads)",
            "config": config_of(p, "fp64", 0, name),
            "cpu_baseline": rec,
            "e2e": {"value": val, "unit": "jobs/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def host_mem_available():
    """MemAvailable of this host in bytes (None if unknown)."""
    try:
        for line in open("/proc/meminfo"):
            if line.startswith("MemAvailable:"):
                return int(line.split()[1]) * 1024
    except OSError:
        pass
    return None


def served_latency(args, local, n_jobs):
    """p50/p99 job latency of a short Poisson stream of served jobs (the
    serving workload's 50/30/20 size mix, first n_jobs jobs) at 80 % of the
    capacity measured on the same stream in a closed loop."""
    a = argparse.Namespace(**vars(args))
    a.serve_jobs, a.serve_load = n_jobs, 0.8
    rec = serving_record(a, local)
    return {"p50_s": rec["latency_s"]["p50"], "p99_s": rec["latency_s"]["p99"], "mean_s": rec["latency_s"]["mean"],
            "jobs_s": rec["value"], "capacity_jobs_s": rec["config"]["capacity_jobs_s"],
            "queue_wait_p99_s": rec["queue_wait_s"]["p99"], "jobs": rec["steps"],
            "stream": "first %d jobs of the serving stream (50/30/20 Gamma-only N_aux 64 / 2-D periodic N_aux 512 / "
                      "uneven instances, n x n x 1 k-grids), arrivals at 80 %% of the closed-loop capacity, "
                      "rpa_submit/rpa_poll, mixed chi0" % n_jobs}


def fp64_roofline(achieved, dfma_kernel, **more):
    """Roofline record of an FP64 product step: the digit products on the tensor
    cores issue 36 BF16 flops per FP64 flop; their peak is the measured BF16 rate
    over that.  A rate above the FP64 pipe's can only be theirs."""
    if achieved <= FP64_PEAK_TFLOPS:
        return dict({"bound": "alu", "achieved": achieved, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
                     "frac": achieved / FP64_PEAK_TFLOPS, "traffic": None, "kernel": dfma_kernel,
                     "peak_source": "derived FP64 DFMA peak: 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz "
                                    "(microbenchmark measured 1.205 TFLOP/s)"}, **more)
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    bf16 = json.load(open(path)).get("bf16_tflops_sustained", 1700.0) if os.path.exists(path) else 1700.0
    return dict({"bound": "tensor", "achieved": achieved, "peak": bf16 / 36, "unit": "TFLOP/s",
                 "frac": 36 * achieved / bf16, "traffic": None,
                 "kernel": "g64_kernel (tcgen05, eight 7-bit digit planes, 36 digit pairs per product) with its slicing",
                 "peak_source": "MEASURED_PEAKS.json bf16_tflops_sustained / 36 (of measured)"}, **more)


def chi0_roofline(prec, prof, cnt, chi0_flops, steps, name, slices):
    """Roofline record of the dominant kernel (the chi0 contraction) from the
    library's CUDA-event profile: `chi0_flops` algorithmic FP64-equivalent
    flops over the profiled launches.  Returns (record, achieved TFLOP/s)."""
    chi_ms, chi_n = prof["chi0"]
    chi_launch_ms = chi_ms / max(chi_n, 1)
    flops_per_launch = chi0_flops / max(chi_n, 1)
    achieved = flops_per_launch / (chi_launch_ms / 1e3) / 1e12 if chi_ms > 0 else 0.0
    counting = ("achieved = the method's algorithmic FP64-equivalent chi0 flops (Hermitian lower triangle, "
                "4N(N+1)N_ov per (q, k, omega), complex; all n_w frequencies) per launch / the launch's mean "
                "CUDA-event time")
    if prec == "fp64":
        return fp64_roofline(achieved, "chi0_fp64_kernel", counting=counting), achieved
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    peak = peaks.get("bf16_tflops_sustained", 1700.0)
    ex_t = cnt["tensor_flops"] / (chi_ms / 1e3) / 1e12 if chi_ms > 0 else None
    return {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
            "traffic": traffic_for("chi0_mixed_" + name),
            "kernel": "chi0_tc_kernel<%d> (tcgen05, BF16 digit slices)" % (slices or 4),
            "peak_source": "MEASURED_PEAKS.json bf16_tflops_sustained (of measured; the kernel runs inside a "
                           "long step)", "counting": counting,
            "executed_tensor_tflops": ex_t, "executed_frac": ex_t / peak if ex_t else None,
            "executed_note": "tensor-core flops the launches issue (slice pairs x padded tiles x padded K x "
                             "the contractions run), counted by the library, per second of chi0 launch time",
            "launch_ms": chi_launch_ms, "launches_per_step": chi_n / max(steps, 1)}, achieved


def run_qshard(args):
    """One job split over the ranks by q-blocks (strong scaling): each rank
    materialises and computes only its own q-points through rpa_energy, the
    integrand table eps[q][w] is summed over ranks (one all-reduce of
    n_q x n_w doubles) and every rank forms E_c by the fixed-order
    quadrature.  A step is one whole job; time is host wall time between
    barriers with the device synchronised on both sides, max over ranks."""
    import torch

    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    import paper_2505_06021_gb300 as rpa
    from paper_2505_06021_gb300 import shard

    prec = args.prec
    if prec == "auto":
        prec = "mixed" if rpa_mixed_available() else "fp64"
    pc = rpa.PREC_MIXED if prec == "mixed" else rpa.PREC_FP64
    name = args.workload
    p = workload(args.n_q, name, args.tail_case)
    qs = list(shard.q_blocks(p.n_q, world)[rank])
    dev = "cuda:%d" % local
    t_gen = time.perf_counter()
    job = shard.block_job(p, rpa.upload_problem(p, dev, qs=qs), qs, pc) if qs else None
    torch.cuda.synchronize()
    t_gen = time.perf_counter() - t_gen
    log("inputs of q %s ready (%.1f s)" % (qs, t_gen))
    ctx = rpa.Context(local, n_slices=args.slices, hbm_cap_bytes=int(args.cap_gb * 1e9), chi0_freq=args.chi0_freq)

    def rows(_qs):
        return ctx.energy(job)["eps"]

    def step():
        return shard.energy_sharded(p.n_q, p.n_w, p.grid.w_q, p.zeta_w, rows, rank, world)

    for _ in range(args.warmup):
        step()
    clocks = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    clocks.start()
    ctx.profile(True)
    n0 = ctx.launches
    t0 = time.perf_counter()
    Ec = None
    for _ in range(args.steps):
        Ec, _table = step()
    torch.cuda.synchronize()
    t = time.perf_counter() - t0
    barrier(world)
    clk = clocks.stop()
    prof = ctx.profile_read()
    cnt = ctx.profile_counters()
    ctx.profile(False)
    launches = int(allreduce_sum(ctx.launches - n0, world))
    t_max = allreduce_max(t, world)
    flops_rank = p.chi0_flops() * len(qs) / p.n_q * args.steps
    roof, achieved = chi0_roofline(prec, prof, cnt, flops_rank, args.steps, name, args.slices)
    roof["note_qshard"] = "rank 0's chi0 launches (its own q-block)"
    if rank != 0:
        return
    cfg = dict(config_of(p, prec, args.n_q, name, args.tail_case),
               parallelism="one job q-sharded over %d ranks (strong scaling; one all-reduce of the n_q x n_w "
                           "integrand table per job)" % world)
    if prec == "mixed":
        cfg.update(chi0_slices=args.slices or 4,
                   chi0_freq=["auto", "per-frequency", "frequency-batched"][args.chi0_freq])
    line = {"metric": METRIC, "value": args.steps / t_max, "unit": "jobs/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * t_max / args.steps, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "f64" if prec == "fp64" else "bf16-slices->f64",
            "data": "synthetic (seeded, shapes of the paper's periodic workloads; no public data)", "config": cfg,
            "chi0_tflops": p.chi0_flops() * args.steps / t_max / 1e12, "chi0_tflops_kernel": achieved,
            "Ec": Ec, "gpu_launches": launches, "q_block_rank0": qs,
            "kernel_ms_per_step_rank0": {k: {"ms": v[0] / args.steps, "launches": v[1] // max(args.steps, 1)}
                                         for k, v in prof.items() if v[1]},
            "roofline": roof, "clocks": clk, "input_gen_s": t_gen,
            "e2e": {"skipped": "q-sharded mode: device-resident inputs only (the end-to-end leg is in the "
                               "default mode)"},
            "cpu_baseline": None}
    print(json.dumps(line), flush=True)


def run_ours(args):
    import numpy as np
    import torch

    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    import paper_2505_06021_gb300 as rpa

    prec = args.prec
    if prec == "auto":
        prec = "mixed" if rpa_mixed_available() else "fp64"
    pc = rpa.PREC_MIXED if prec == "mixed" else rpa.PREC_FP64
    name = args.workload
    p = workload(args.n_q, name, args.tail_case)
    dev = "cuda:%d" % local
    # end-to-end inputs: pinned host copies of the whole job (generated once;
    # the device-resident job is copied from them)
    want_e2e = not args.no_e2e and not args.n_q
    e2e_skip = None
    if want_e2e:
        avail = host_mem_available()
        need = 1.25 * p.c_bytes() * world + 16e9
        if avail is not None and avail < need:
            want_e2e, e2e_skip = False, "host memory: %.0f GB available, %.0f GB needed" % (avail / 1e9, need / 1e9)
    t_gen = time.perf_counter()
    th = None
    if want_e2e:
        with near_gpu(local) as ng:
            th = rpa.upload_problem(p, "cpu", pin=True)
        tens = {"C": [t.to(dev, non_blocking=True) for t in th["C"]], "V": [t.to(dev) for t in th["V"]],
                "eps_occ": th["eps_occ"].to(dev), "eps_virt": th["eps_virt"].to(dev)}
    else:
        tens = rpa.upload_problem(p, dev)
    torch.cuda.synchronize()
    t_gen = time.perf_counter() - t_gen
    log("inputs ready (%.1f s)" % t_gen)
    job = rpa.job_from_problem(p, tens, prec=pc)
    ctx = rpa.Context(local, n_slices=args.slices, hbm_cap_bytes=int(args.cap_gb * 1e9), chi0_freq=args.chi0_freq)
    for _ in range(args.warmup):
        ctx.energy(job)
    log("warm-up done")
    ext = torch.cuda.ExternalStream(ctx.stream_handle)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    clocks = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    clocks.start()
    ctx.profile(True)
    n0 = ctx.launches
    ev[0].record(ext)
    res = None
    for i in range(args.steps):
        res = ctx.energy(job)
        ev[i + 1].record(ext)
    torch.cuda.synchronize()
    barrier(world)
    clk = clocks.stop()
    prof = ctx.profile_read()
    cnt = ctx.profile_counters()
    ctx.profile(False)
    launches = ctx.launches - n0
    step_ms = [ev[i].elapsed_time(ev[i + 1]) for i in range(args.steps)]
    ms = ev[0].elapsed_time(ev[args.steps])
    ms_max = allreduce_max(ms, world)
    jobs_per_s = world * args.steps / (ms_max / 1e3)
    chi0_flops_job = p.chi0_flops()

    roof, achieved = chi0_roofline(prec, prof, cnt, chi0_flops_job * args.steps, args.steps, name, args.slices)
    kernel_ms = {k: {"ms": v[0] / args.steps, "launches": v[1] // max(args.steps, 1)} for k, v in prof.items()
                 if v[1]}
    line = {"metric": METRIC, "value": jobs_per_s, "unit": "jobs/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64" if prec == "fp64" else "bf16-slices->f64",
            "data": "synthetic (seeded, shapes of the paper's periodic workloads; no public data)",
            "config": dict(config_of(p, prec, args.n_q, name, args.tail_case),
                           **({"chi0_slices": args.slices or 4, "chi0_freq": ["auto", "per-frequency",
                                                                               "frequency-batched"][args.chi0_freq]}
                              if prec == "mixed" else {})),
            "chi0_tflops": chi0_flops_job * world * args.steps / (ms_max / 1e3) / 1e12,
            "chi0_tflops_kernel": achieved, "Ec": res["Ec"], "gpu_launches": launches,
            "chi0_freq_plan": plan_of(rpa, p, args.chi0_freq) if prec == "mixed" else None,
            "latency_s": {"p50": float(np.percentile(step_ms, 50)) / 1e3,
                          "p99": float(np.percentile(step_ms, 99)) / 1e3,
                          "what": "per-job latency of the timed jobs (one job at a time, device-resident inputs, "
                                  "CUDA events between jobs)"},
            "kernel_ms_per_step": kernel_ms, "roofline": roof, "clocks": clk, "input_gen_s": t_gen}

    log("timed steps done: %.1f ms/step" % (ms_max / args.steps))
    # end to end through the public API with HOST buffers (pinned), copies inside
    if want_e2e:
        jh = rpa.job_from_problem(p, th, prec=pc, mem=rpa.MEM_HOST)
        ctx.energy(jh)
        barrier(world)
        torch.cuda.synchronize()
        ctx.profile(True)
        t0 = time.perf_counter()
        step_s = []
        for _ in range(args.e2e_steps):
            t1 = time.perf_counter()
            rh = ctx.energy(jh)
            step_s.append(time.perf_counter() - t1)
        torch.cuda.synchronize()
        te = allreduce_max(time.perf_counter() - t0, world)
        hprof = ctx.profile_read()
        hcnt = ctx.profile_counters()
        ctx.profile(False)
        h2d = sum(t.numel() * t.element_size() for t in th["C"] + th["V"]) + 8 * (th["eps_occ"].numel() +
                                                                                    th["eps_virt"].numel())
        nqw = p.n_q * p.n_w
        cp_ms = hprof["h2d"][0]
        line["e2e"] = {"value": world * args.e2e_steps / te, "unit": "jobs/s", "h2d_bytes_per_step": h2d,
                       "d2h_bytes_per_step": 8 * (1 + 3 * nqw) + 4, "steps": args.e2e_steps,
                       "step_s": step_s,
                       "h2d_gbs_library": (hcnt["h2d_bytes"] / (cp_ms / 1e3) / 1e9) if cp_ms > 0 else None,
                       "h2d_gbs_note": "bytes rpa_energy copied host->device / the copies' own time (CUDA events "
                                       "around each q-batch's copies on the library's copy stream), over the "
                                       "e2e steps",
                       "h2d_bytes_library_per_step": hcnt["h2d_bytes"] / args.e2e_steps,
                       "h2d_copy_ms_per_step": cp_ms / args.e2e_steps,
                       "kernel_ms_per_step": {k: {"ms": v[0] / args.e2e_steps, "launches": v[1] / args.e2e_steps}
                                              for k, v in hprof.items() if v[1]},
                       "host_numa_node": ng.node, "pinned_near_gpu": bool(ng.cpus),
                       "abs_dEc_e2e_vs_device_Ha": abs(rh["Ec"] - res["Ec"]),
                       "dEc_note": "the host-staged job runs its chi0 in other q-batches and workspace rounds than "
                                   "the device-resident one, so the split-precision sums differ in the last bits"}
        del jh
    else:
        line["e2e"] = None if e2e_skip is None else {"skipped": e2e_skip}
    del th

    log("e2e done")
    # one step of the plain FP64 path on the same job, and the mixed path's error
    if prec == "mixed" and not args.no_fp64 and not args.n_q and world == 1:
        jf = job.with_prec(rpa.PREC_FP64)
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        f0.record(ext)
        rf = ctx.energy(jf)
        f1.record(ext)
        torch.cuda.synchronize()
        fms = f0.elapsed_time(f1)
        rel = np.abs(res["eps"] - rf["eps"]) / np.abs(rf["eps"])
        line["fp64"] = {"value": 1.0 / (fms / 1e3), "unit": "jobs/s", "ms_per_step": fms, "steps": 1,
                        "warmup": 0, "Ec": rf["Ec"], "abs_dEc_mixed_vs_fp64_Ha": abs(res["Ec"] - rf["Ec"]),
                        "max_rel_err_per_term": float(rel.max()), "median_rel_err_per_term": float(np.median(rel))}
        line["speedup_mixed_vs_fp64"] = jobs_per_s / line["fp64"]["value"]
        del jf
    ctx.close()
    del job, tens
    torch.cuda.empty_cache()

    log("fp64 step done")
    # p50/p99 of a short served stream (the metric's latency part)
    if args.lat_jobs > 0 and not args.n_q and world == 1:
        try:
            line["serving"] = served_latency(args, local, args.lat_jobs)
        except Exception as ex:  # recorded, the line still prints
            line["serving"] = {"error": repr(ex)[:300]}

    log("served stream done")
    if rank == 0 and not args.no_cpu_baseline and world == 1:
        smp = OracleSampler(p, name, n_vhalf=1)
        for i in range(3):
            smp.step(i)
        line["cpu_baseline"] = smp.record()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist

        dist.destroy_process_group()


def rpa_mixed_available():
    return True


def run_batch(args):
    """64 uneven Gamma-real / 2x2x1-complex instances per step through
    rpa_energy_batch (shared persistent tensor-core launches, replayed from a
    captured CUDA graph after the first, autotuned call)."""
    import numpy as np
    import torch

    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    import paper_2505_06021_gb300 as rpa
    from paper_2505_06021_gb300 import synth

    prec = "fp64" if args.prec == "fp64" else "mixed"
    pc = rpa.PREC_MIXED if prec == "mixed" else rpa.PREC_FP64
    probs = synth.config3_instances(n_inst=args.n_inst)
    t_gen = time.perf_counter()
    tens = [rpa.upload_problem(p, "cuda:%d" % local) for p in probs]
    torch.cuda.synchronize()
    t_gen = time.perf_counter() - t_gen
    jobs = [rpa.job_from_problem(p, t, prec=pc) for p, t in zip(probs, tens)]
    ctx = rpa.Context(local, n_slices=args.slices)
    t_first = time.perf_counter()
    E_first = ctx.energy_batch(jobs)  # eager + autotune + graph capture
    t_first = time.perf_counter() - t_first
    for _ in range(max(0, args.warmup - 1)):
        ctx.energy_batch(jobs)
    # one profiled (eager) step for the per-kernel split and the roofline
    ctx.profile(True)
    ctx.energy_batch(jobs)
    prof = ctx.profile_read()
    cnt = ctx.profile_counters()
    ctx.profile(False)
    ext = torch.cuda.ExternalStream(ctx.stream_handle)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    clocks.start()
    n0 = ctx.launches
    e0.record(ext)
    E = None
    for _ in range(args.steps):
        E = ctx.energy_batch(jobs)
    e1.record(ext)
    torch.cuda.synchronize()
    barrier(world)
    clk = clocks.stop()
    launches = ctx.launches - n0
    ms = allreduce_max(e0.elapsed_time(e1), world)
    n = len(jobs)
    val = world * n * args.steps / (ms / 1e3)
    alg = sum(p.chi0_flops() for p in probs)
    chi_ms, chi_n = prof["chi0"]
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    if prec == "mixed":
        peak = peaks.get("bf16_tflops_sustained", 1700.0)
        ach = alg / (chi_ms / 1e3) / 1e12
        ex_t = cnt["tensor_flops"] / (chi_ms / 1e3) / 1e12
        roof = {"bound": "tensor", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak,
                "traffic": None, "kernel": "chi0 tcgen05 sliced (persistent, all segments of a round)",
                "peak_source": "MEASURED_PEAKS.json bf16_tflops_sustained (of measured)",
                "counting": "achieved = the instances' algorithmic FP64-equivalent chi0 flops (Hermitian lower "
                            "triangle) per second of tensor-core launch time",
                "executed_tensor_tflops": ex_t, "executed_frac": ex_t / peak,
                "timing": "one profiled eager batch step: CUDA events around every tensor-core launch"}
    else:
        ach = alg / (chi_ms / 1e3) / 1e12
        roof = fp64_roofline(ach, "chi0_fp64_kernel")
    line = {"metric": METRIC, "value": val, "unit": "jobs/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64" if prec == "fp64" else "bf16-slices->f64",
            "data": "synthetic (seeded, shapes of the paper's workloads; no public data)",
            "config": {"workload": "batch-uneven: %d independent Gamma-real / 2x2x1-complex instances, N_aux ~ "
                                   "U[128,1024], N_occ ~ U[8,64], N_virt = 4-15 x N_occ, 16 frequencies each; "
                                   "one rpa_energy_batch call per step (CUDA graph replay)" % n,
                       "n_inst": n, "chi0_prec": prec, "chi0_slices": args.slices or 4,
                       "c_gb": sum(p.c_bytes() for p in probs) / 1e9,
                       "l2": "inputs larger than L2", "parallelism": "one batch per GPU (weak scaling)"},
            "chi0_tflops": alg * world * args.steps / (ms / 1e3) / 1e12, "gpu_launches": launches,
            "kernel_ms_per_step": {k: {"ms": v[0], "launches": v[1]} for k, v in prof.items() if v[1]},
            "roofline": roof, "clocks": clk, "input_gen_s": t_gen, "first_call_s": t_first,
            "first_call_matches_replay": bool(np.array_equal(E_first, E))}
    if prec == "mixed" and not args.no_fp64:
        jf = [j.with_prec(rpa.PREC_FP64) for j in jobs]
        Ef = ctx.energy_batch(jf)
        torch.cuda.synchronize()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(ext)
        Ef = ctx.energy_batch(jf)
        f1.record(ext)
        torch.cuda.synchronize()
        fms = f0.elapsed_time(f1)
        line["fp64"] = {"value": n / (fms / 1e3), "unit": "jobs/s", "ms_per_step": fms,
                        "max_abs_dEc_mixed_vs_fp64_Ha": float(np.max(np.abs(E - Ef)))}
        line["speedup_mixed_vs_fp64"] = val / line["fp64"]["value"]
    if not args.no_e2e:
        # host-resident inputs copied into the job's device buffers inside the timed region
        host = [{k: ([x.cpu().pin_memory() for x in v] if isinstance(v, list) else v.cpu().pin_memory())
                 for k, v in t.items()} for t in tens]
        h2d = 0
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with torch.cuda.stream(ext):
            for t, h in zip(tens, host):
                for k in ("C", "V"):
                    for d, x in zip(t[k], h[k]):
                        d.copy_(x, non_blocking=True)
                        h2d += x.numel() * x.element_size()
                for k in ("eps_occ", "eps_virt"):
                    t[k].copy_(h[k], non_blocking=True)
                    h2d += h[k].numel() * h[k].element_size()
        Ee = ctx.energy_batch(jobs)
        te = time.perf_counter() - t0
        line["e2e"] = {"value": n / te, "unit": "jobs/s", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": 8 * n,
                       "steps": 1, "Ec_matches_device": bool(np.array_equal(Ee, E))}
        del host
    else:
        line["e2e"] = None
    ctx.close()
    if rank == 0:
        print(json.dumps(line), flush=True)


_V_CACHE = {}  # V(q) depends only on the shape here: shared by jobs of one shape


def plan_of(rpa, p, mode):
    """The frequency-batched chi0 plan of a problem (rpa_chi0_plan on a host
    descriptor with placeholder C/V pointers: the plan reads only the shapes,
    pairs, frequencies and band energies)."""
    import numpy as np
    import torch

    ph = torch.empty(1)
    t = {"C": [ph] * (p.n_q * p.n_k), "V": [ph] * p.n_q,
         "eps_occ": torch.from_numpy(np.ascontiguousarray(p.eps_occ, np.float64)),
         "eps_virt": torch.from_numpy(np.ascontiguousarray(p.eps_virt, np.float64))}
    pl = rpa.job_from_problem(p, t, prec=rpa.PREC_MIXED, mem=rpa.MEM_HOST).chi0_plan(2 if mode == 2 else 0)
    if mode == 1 or pl["n_bins"] == 0:
        return {"used": False}
    return {"used": True, "n_bins": pl["n_bins"], "rank": [int(x) for x in pl["rank"]],
            "max_residual": float(pl["err"].max()), "work_ratio": pl["work_ratio"]}


def footprint_of(rpa, p, prec):
    """rpa_job_footprint of a problem's job (placeholder pointers: the
    footprint reads only the shape fields)."""
    import torch

    ph = torch.empty(1)
    t = {"C": [ph] * (p.n_q * p.n_k), "V": [ph] * p.n_q, "eps_occ": torch.empty((p.eps_occ.shape[0], 1)),
         "eps_virt": ph}
    return rpa.job_from_problem(p, t, prec=prec).footprint()


def device_inputs(p, device, seed):
    """Seeded synthetic inputs generated on the device (serving workload: jobs
    are materialised as they arrive).  Same laws as the host generator: C
    Gaussian with variance 1/N_ov, V = Q diag(lam) Q^H with Q Haar-random and
    the problem's eigenvalue law, bands from the problem."""
    import numpy as np
    import torch

    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    rdt = torch.float64
    C = []
    for _ in range(p.n_q * p.n_k):
        if p.is_complex:
            x = torch.randn((p.n_aux, p.n_ov, 2), dtype=rdt, device=device, generator=g) * math.sqrt(0.5 / p.n_ov)
            C.append(torch.view_as_complex(x))
        else:
            C.append(torch.randn((p.n_aux, p.n_ov), dtype=rdt, device=device, generator=g) / math.sqrt(p.n_ov))
    V = []
    for q in range(p.n_q):
        key = (p.is_complex, p.n_aux, p.n_q, q)
        if key in _V_CACHE:
            V.append(_V_CACHE[key])
            continue
        rng = np.random.default_rng([int(seed), q])
        if p.is_complex:
            z = torch.view_as_complex(torch.randn((p.n_aux, p.n_aux, 2), dtype=rdt, device=device, generator=g))
        else:
            z = torch.randn((p.n_aux, p.n_aux), dtype=rdt, device=device, generator=g)
        Q, R = torch.linalg.qr(z)
        d = torch.diagonal(R)
        Q = Q * (d / d.abs())[None, :]
        lam = np.exp(rng.uniform(math.log(p.lam_lo), math.log(p.lam_hi), p.n_aux))
        if p.scale_lead and p.n_q > 1:
            qn = float(np.linalg.norm(p.grid.qpts[q]))
            if qn > 1e-12:
                lam[int(np.argmax(lam))] *= (p.grid.q_min / qn) ** 2
        lt = torch.from_numpy(lam).to(device=device, dtype=rdt).to(Q.dtype)
        Vq = (Q * lt[None, :]) @ Q.conj().T
        Vq = (0.5 * (Vq + Vq.conj().T)).contiguous()
        _V_CACHE[key] = Vq
        V.append(Vq)
    eo = torch.from_numpy(p.eps_occ.astype(np.float64)).to(device)
    ev = torch.from_numpy(p.eps_virt.astype(np.float64)).to(device)
    return {"C": C, "V": V, "eps_occ": eo, "eps_virt": ev}


def run_serving(args):
    world, rank, local = dist_setup()
    line = serving_record(args, local)
    line["n_gpus"] = world
    if rank == 0:
        print(json.dumps(line), flush=True)


def serving_record(args, local):
    """Poisson stream of RPA energy jobs through rpa_submit / rpa_wait: sizes
    drawn 50/30/20 from Gamma-only (N_aux=64), 2-D periodic (N_aux=512) and
    uneven-instance shapes with n x n x 1 k-grids, n ~ U{1..4}; inputs made
    on the device as each job arrives; mixed-precision chi0; admission by HBM
    footprint under the cap.  The arrival rate is a fraction of the capacity
    measured first by running the whole stream in a closed loop."""
    os.environ.setdefault("PYTORCH_ALLOC_CONF", "expandable_segments:True")
    import torch

    world = int(os.environ.get("WORLD_SIZE", "1"))
    torch.cuda.set_device(local)
    import paper_2505_06021_gb300 as rpa
    from paper_2505_06021_gb300 import synth

    dev = "cuda:%d" % local
    pc = rpa.PREC_FP64 if args.prec == "fp64" else rpa.PREC_MIXED
    cap = int(args.serve_cap_gb * (1 << 30))
    stream = synth.serving_stream(n_jobs=args.serve_jobs, rate_per_s=1.0)
    gen_stream = torch.cuda.Stream()

    def make(i, p):
        with torch.cuda.stream(gen_stream):
            t = device_inputs(p, dev, 1000 + i)
        gen_stream.synchronize()
        return t, rpa.job_from_problem(p, t, prec=pc)

    ctx = rpa.Context(local, hbm_cap_bytes=cap, n_slices=args.slices)
    fits = [footprint_of(rpa, p, pc) <= cap for _, p in stream]
    # capacity: the whole stream in a closed loop (the job-size mix is heavy
    # tailed, so samples mislead), at most 8 jobs in flight, each job's inputs
    # made on the device while earlier jobs run; also the warm-up
    adm = [i for i in range(len(stream)) if fits[i]]
    t0 = time.perf_counter()
    window = []
    for i in adm:
        # at most 8 jobs and ~100 GB of their inputs outstanding
        while window and (len(window) >= 8 or sum(stream[k][1].c_bytes() for k, *_ in window) +
                          stream[i][1].c_bytes() > 100e9):
            ctx.wait(window.pop(0)[1], 600.0)
        tens_i, job_i = make(i, stream[i][1])
        window.append((i, ctx.submit(job_i), tens_i, job_i))
    for _, t, _, _ in window:
        ctx.wait(t, 600.0)
    cap_jobs_s = len(adm) / (time.perf_counter() - t0)
    del window
    ctx.close()
    torch.cuda.empty_cache()
    rate = args.serve_load * cap_jobs_s
    # open loop: arrivals at `rate`, inputs made on the device as each job arrives
    import threading

    ctx2 = rpa.Context(local, hbm_cap_bytes=cap, n_slices=args.slices)
    lock = threading.Lock()
    live = {}
    done_t = {}
    rejected = []
    clocks = ClockSampler(local)
    clocks.start()
    t_start = time.perf_counter()

    failed = []

    def producer():
        for i, (ta, p) in enumerate(stream):
            if not fits[i]:
                rejected.append(i)
                continue
            t_arr = t_start + ta / rate
            dt = t_arr - time.perf_counter()
            if dt > 0:
                time.sleep(dt)
            # the harness's own memory: wait while ~130 GB of inputs are out
            while True:
                with lock:
                    held = sum(stream[k][1].c_bytes() for k, _, _ in live.values())
                if held + p.c_bytes() <= 130e9 or not live:
                    break
                time.sleep(0.001)
            try:
                tens, job = make(i, p)
                with lock:
                    live[ctx2.submit(job)] = (i, tens, job)
            except Exception as ex:  # recorded in the JSON line, the stream goes on
                failed.append((i, repr(ex)[:200]))

    th = threading.Thread(target=producer)
    th.start()
    results = {}
    while th.is_alive() or live:
        with lock:
            items = list(live.items())
        progressed = False
        for t, (i, tens, job) in items:
            r = ctx2.poll(t)
            if r is not None:
                results[i] = r[0]
                done_t[i] = time.perf_counter()
                with lock:
                    del live[t]
                progressed = True
        if not progressed:
            time.sleep(0.0005)
    th.join()
    makespan = time.perf_counter() - t_start
    clk = clocks.stop()
    st = ctx2.serving_stats()
    peak = ctx2.serving_peak()
    launches = ctx2.launches
    ctx2.close()
    n_done = len(results)
    line = {"metric": METRIC, "value": n_done / makespan, "unit": "jobs/s", "n_gpus": world, "steps": n_done,
            "warmup": len(adm), "ms_per_step": 1e3 * makespan / max(n_done, 1), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64" if pc == rpa.PREC_FP64 else "bf16-slices->f64",
            "data": "synthetic (seeded; inputs generated on the device at arrival)",
            "config": {"workload": "serving: Poisson stream of %d RPA energy jobs, 50/30/20 Gamma-only (N_aux=64) / "
                                   "2-D periodic (N_aux=512) / uneven-instance shapes, k-grids n x n x 1 with "
                                   "n ~ U{1..4}; arrival rate %.2f x measured capacity; admission by HBM "
                                   "footprint under a %.0f GB cap" % (len(stream), args.serve_load,
                                                                       args.serve_cap_gb),
                       "chi0_slices": args.slices or 4,
                       "arrival_rate_jobs_s": rate, "capacity_jobs_s": cap_jobs_s,
                       "capacity_sample": "closed loop over the %d admissible jobs of the stream, at most 8 in "
                                          "flight, inputs made on the device meanwhile" % len(adm),
                       "rejected_over_cap": len(rejected),
                       "failed_to_submit": len(failed), "failures": failed[:3],
                       "l2": "inputs larger than L2", "parallelism": "one serving context per GPU"},
            "latency_s": {"p50": st["lat_p50_s"], "p99": st["lat_p99_s"], "mean": st["lat_mean_s"]},
            "queue_wait_s": {"p50": st["wait_p50_s"], "p99": st["wait_p99_s"]},
            "peak_running_jobs": peak["max_running"], "peak_admitted_gb": peak["max_bytes"] / 1e9,
            "largest_micro_batch": peak["max_batch"],
            "gpu_launches": launches, "clocks": clk, "roofline": None, "e2e": None}
    return line


def ao_flops(p):
    """Algorithmic FP64 flops of the AO -> MO transform of a whole AO-form job
    (8 per complex multiply-add, 2 per real one): the half-transforms
    n_bas * S * n_occ per k-point used as k and n_bas * S * n_virt per k-point
    used as k+q (plus, lattice form, the lattice sums), then
    2 * sum_A nb_A nf_A * N_ov per (q, k) pair."""
    f = 8.0 if p.is_complex else 2.0
    ko = len(set(p.grid.pair_k.reshape(-1).tolist()))
    kv = len(set(p.grid.pair_kq.reshape(-1).tolist()))
    half = f * p.n_bas * p.n_pf * (ko * p.n_occ + kv * p.n_virt)
    if getattr(p, "lattice", None) is not None:  # lattice sums: a real-times-phase multiply-add per vector
        kk = len(set(p.grid.pair_k.reshape(-1).tolist()) | set(p.grid.pair_kq.reshape(-1).tolist()))
        half += (4.0 if p.is_complex else 2.0) * len(p.lattice) * p.n_bas * p.n_pf * kk
    asm = f * 2.0 * p.n_pf * p.n_ov * p.n_q * p.n_k
    return half, asm


def run_ao(args):
    """The 2-D periodic job given in AO form (two atoms, PADF and MO
    coefficients per k-point): the library forms each q's MO-basis fit
    coefficients on the device just before its chi0 (rpa_energy)."""
    import numpy as np
    import torch

    import paper_2505_06021_gb300 as rpa
    from paper_2505_06021_gb300 import synth

    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    prec = "mixed" if args.prec in ("auto", "mixed") else "fp64"
    pc = rpa.PREC_MIXED if prec == "mixed" else rpa.PREC_FP64
    sc = max(1, args.ao_scale)
    p = synth.config1_ao(n_bas_atom=(128 // sc,) * 2, n_fit_atom=(256 // sc,) * 2, n_occ=32 // sc, n_virt=224 // sc,
                         lattice_radius=args.ao_lattice or None)
    if args.ao_projector > 0.0:
        p.eps_d = args.ao_projector
    if args.n_q:
        g = p.grid
        g.pair_k, g.pair_kq, g.w_q, g.qpts = g.pair_k[:args.n_q], g.pair_kq[:args.n_q], g.w_q[:args.n_q], \
            g.qpts[:args.n_q]
    t_gen = time.perf_counter()
    tens = rpa.upload_ao_problem(p, "cuda:%d" % local)
    torch.cuda.synchronize()
    t_gen = time.perf_counter() - t_gen
    job = rpa.job_from_ao_problem(p, tens, prec=pc)
    ctx = rpa.Context(local, n_slices=args.slices)
    for _ in range(args.warmup):
        ctx.energy(job)
    ext = torch.cuda.ExternalStream(ctx.stream_handle)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    clocks.start()
    ctx.profile(True)
    n0 = ctx.launches
    e0.record(ext)
    res = None
    for _ in range(args.steps):
        res = ctx.energy(job)
    e1.record(ext)
    torch.cuda.synchronize()
    barrier(world)
    clk = clocks.stop()
    prof = ctx.profile_read()
    ctx.profile(False)
    launches = ctx.launches - n0
    ms_max = allreduce_max(e0.elapsed_time(e1), world)
    jobs_per_s = world * args.steps / (ms_max / 1e3)
    half, asm = ao_flops(p)
    ao_ms, ao_n = prof["ao2mo"]
    ach = (half + asm) * args.steps / (ao_ms / 1e3) / 1e12
    roof = fp64_roofline(ach, "ao_half_kernel + ao_assemble_kernel (AO -> MO transform, FP64)",
                         algorithmic_tflop_per_job=(half + asm) / 1e12, launches_per_job=ao_n // max(args.steps, 1))
    kernel_ms = {k: {"ms": v[0] / args.steps, "launches": v[1] // max(args.steps, 1)} for k, v in prof.items()
                 if v[1]}
    line = {"metric": METRIC, "value": jobs_per_s, "unit": "jobs/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64" if prec == "fp64" else "bf16-slices->f64",
            "data": "synthetic (seeded PADF and MO coefficients with the shapes of the 2-D periodic workload)",
            "config": {"workload": "periodic2d-ao: the 2-D periodic job (16 q x 16 k, N_aux=%d, N_occ=%d, "
                                   "N_virt=%d, 20 frequencies) in AO form: 2 atoms x (%d basis, %d fit "
                                   "functions), N_bas=%d, PADF %.1f GB %s + MO coefficients per k-point; "
                                   "MO-basis coefficients formed per q on the device%s"
                                   % (p.n_aux, p.n_occ, p.n_virt, p.n_bas_atom[0], p.n_fit_atom[0], p.n_bas,
                                      p.padf_bytes() / 1e9,
                                      "per k-point" if p.lattice is None else
                                      "(real, per lattice vector of %d; k-point arrays formed as lattice sums)"
                                      % len(p.lattice),
                                      "" if sc == 1 and not args.n_q else " [reduced: profiling case]"),
                       "n_q": p.n_q, "n_k": p.n_k, "n_aux": p.n_aux, "n_occ": p.n_occ, "n_virt": p.n_virt,
                       "n_w": p.n_w, "n_bas": p.n_bas, "n_atoms": p.n_atoms, "chi0_prec": prec,
                       "projector_eps_d": p.eps_d,
                       "l2": "inputs larger than L2 (PADF %.1f GB)" % (p.padf_bytes() / 1e9),
                       "parallelism": "one job per GPU (weak scaling)"},
            "chi0_tflops": p.chi0_flops() * world * args.steps / (ms_max / 1e3) / 1e12, "Ec": res["Ec"],
            "gpu_launches": launches, "kernel_ms_per_step": kernel_ms, "roofline": roof, "clocks": clk,
            "input_gen_s": t_gen}
    if prec == "mixed" and not args.no_fp64 and not args.n_q:
        jf = job.with_prec(rpa.PREC_FP64)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rf = ctx.energy(jf)
        tf = time.perf_counter() - t0
        rel = np.abs(res["eps"] - rf["eps"]) / np.abs(rf["eps"])
        line["fp64"] = {"value": 1.0 / tf, "unit": "jobs/s", "Ec": rf["Ec"],
                        "abs_dEc_mixed_vs_fp64_Ha": abs(res["Ec"] - rf["Ec"]),
                        "max_rel_err_per_term": float(rel.max())}
    if not args.no_e2e and not args.n_q:
        # host-resident AO inputs (pinned) copied to the device inside the timed region
        pin_src = tens["padf"] if tens["padf"] is not None else tens["padf_R"]
        with near_gpu(local):
            hp = [t.cpu().pin_memory() for t in pin_src]
            hm = [t.cpu().pin_memory() for t in tens["mo"]]
            hv = [t.cpu().pin_memory() for t in tens["V"]]
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(args.e2e_steps):
            for d, h in zip(pin_src + tens["mo"] + tens["V"], hp + hm + hv):
                d.copy_(h, non_blocking=True)
            torch.cuda.synchronize()
            rh = ctx.energy(job)
        te = allreduce_max(time.perf_counter() - t0, world)
        h2d = sum(t.numel() * t.element_size() for t in hp + hm + hv)
        line["e2e"] = {"value": world * args.e2e_steps / te, "unit": "jobs/s", "h2d_bytes_per_step": h2d,
                       "d2h_bytes_per_step": 8 * (1 + 3 * p.n_q * p.n_w) + 4, "steps": args.e2e_steps,
                       "Ec_matches_device": bool(rh["Ec"] == res["Ec"])}
    else:
        line["e2e"] = None
    if rank == 0 and not args.no_cpu_baseline and world == 1:
        import oracle

        rng = np.random.default_rng(3)
        ent = np.stack([rng.integers(0, p.n_aux, 4000), rng.integers(0, p.n_ov, 4000)], axis=1)
        t0 = time.perf_counter()
        oracle.ao2mo_block(p, 0, 0, entries=ent)
        t_ent = (time.perf_counter() - t0) / len(ent)
        s = cpu_oracle_sample_ao(p)
        job_s = p.n_q * p.n_k * p.n_aux * p.n_ov * t_ent + p.n_q * s["vhalf_s"] + p.n_q * p.n_w * s["term_s"]
        line["cpu_baseline"] = {"value": 1.0 / job_s, "unit": "jobs/s", "cores": s["threads"], "kind": "oracle",
                                "sample": "4000 entries of one (q, k) block of the AO -> MO transform (double "
                                          "sum over mu, nu), one (q=0, w=0) term and one V(q)^1/2; job time "
                                          "extrapolated", "extrapolated_job_s": job_s}
    ctx.close()
    if rank == 0:
        print(json.dumps(line), flush=True)


def cpu_oracle_sample_ao(p):
    """Oracle timing sample for an AO-form problem: the term's coefficient blocks
    are random stand-ins of the right shape (the term's cost does not depend
    on their values; the transform is timed separately)."""
    import numpy as np

    import oracle

    nthr = oracle.max_threads()
    t0 = time.perf_counter()
    Vh = oracle.vhalf(p.V(0))
    t1 = time.perf_counter()
    rng = np.random.default_rng(0)
    C = [(rng.standard_normal((p.n_aux, p.n_ov)) + 1j * rng.standard_normal((p.n_aux, p.n_ov))) /
         math.sqrt(2 * p.n_ov) for _ in range(p.n_k)]
    t2 = time.perf_counter()
    oracle.term(p, 0, 0, Vh=Vh, C_blocks=C)
    t3 = time.perf_counter()
    return {"vhalf_s": t1 - t0, "term_s": t3 - t2, "threads": nthr}


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batch":
        run_batch(args)
    elif args.workload == "serving":
        run_serving(args)
    elif args.workload == "periodic2d-ao":
        run_ao(args)
    elif args.q_shard:
        run_qshard(args)
    else:
        run_ours(args)  # slab (default) or periodic2d


if __name__ == "__main__":
    main()
