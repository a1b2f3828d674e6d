"""Throughput of batched Boys-function evaluation on GB300 (one JSON line).

Workload (one step): FP64 stored mode at kmax = 32 over N = 2^26 arguments
drawn from the ERI-shaped mixture (40% log-uniform [1e-12, 1e2], 40% uniform
[0, 60], 20% uniform [60, 1e4]); output F_0..F_32 order-major [33][N]
(17.7 GB).  Metric: F_k values per second = N * 33 / step time.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--modes fused,fp32,grad,pairwise,ragged | none]

* ``value``     device-resident inputs, CUDA-event timing of K steps on the
                launching stream, barrier + synchronize on both sides, max
                over ranks; rank r evaluates elements [r 2^26, (r+1) 2^26) of
                one argument stream (weak scaling, no data-path collective).
* ``e2e``       the same metric through the public API with host buffers
                (boys_eval_host): every step reads x from pinned host memory
                and writes all of F to pinned host memory over the host link,
                inside the timed region.
* ``modes``     the other kernels on their own workloads: fused consumer,
                FP32 tier, gradient, the paper's Algorithm 2 at N = 2^19,
                ragged batch (CUDA events, one line each).
* ``roofline``  the dominant kernel (the FP64 evaluation kernel) against the
                HBM roof: algorithmic bytes (8 + 8*33 per argument) over the
                measured copy bandwidth; beside it the paper's algorithmic
                FP64 flops (FMA = 2, each divide / exp / rsqrt = 1) over the
                nominal FP64 peak, which the kernel can exceed because much
                of that work runs on its integer pipes.
* ``cpu_baseline`` the binary128 oracle on the host cores, on a bounded
                sample of the same workload.
``--impl reference`` times that oracle alone (rank 0 only) and prints its line.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "F_k values/s at kmax=32: FP64 (≤5e-14) vs FP32 tier (≤1e-6); % of roofline"
UNIT = "F_k values/s"
KMAX = 32
N_PER_GPU = 1 << 26
WORKLOAD = "boys_fp64_stored_kmax32_n2^26_eri_mixture"

# FP64 peak: the nominal rate at the SM clock seen during the timed region,
# SMs (from the device) x 2 DFMA per clock per SM (GB300's FP64 unit) x 2 flop;
# at 152 SMs and 2.07 GHz that is 1.259 TFLOP/s (an in-house DFMA loop reached
# 95% of it).  Burst HBM copy bandwidth comes from MEASURED_PEAKS.json; the
# fallback is the pool's stated 6.8 TB/s.
DFMA_PER_SM_PER_CLOCK = 2
HBM_FALLBACK_GBS = 6800.0
# DRAM bytes per argument of the timed kernel from one ncu capture at N = 2^22
# (profiles/k_eval_f64_kmax32_eri_mixture.md), scaled to the launch by the
# arguments it processes.  Valid only for the kernel sources it was taken on:
# the bench reports traffic null whenever their SHA-256 differs.
TRAFFIC_CAPTURE = {"bytes_per_x": 257.14, "sources_sha256": "1779eaf727ff8e40a21593be5f53cdd0a051edd8f2cb5f2fbaf0e1d8da99a13d"}
KERNEL_SOURCES = ("boys_fp64.cu", "boys_region.cuh", "gen_local.py", "gen_coeffs_fixed.py", "boys_coeffs_fp64.h",
                  "boys_xf.cuh", "boys_xf_consts.h", "boys_internal.h", "boys_abi.cu")


def kernel_sources_sha256():
    import hashlib
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_2512_10059_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def fp64_peak_tflops(sm_count, sm_mhz):
    """Nominal FP64 FMA rate of the device at the given SM clock."""
    return sm_count * DFMA_PER_SM_PER_CLOCK * 2 * sm_mhz * 1e6 / 1e12


def sm_clock_mhz(clocks):
    """SM clock for the FP64 peak: the median sampled under load, else the
    device's maximum (nvidia-smi, else MEASURED_PEAKS.json)."""
    for key in ("sm_mhz", "sm_max_mhz"):
        v = clocks.get(key) if clocks else None
        if v:
            return float(v), f"{key} sampled by nvidia-smi"
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["sm_max_mhz"]), "sm_max_mhz of MEASURED_PEAKS.json"
    except Exception:
        return 2070.0, "GB300 maximum SM clock as stated for the pool (no clock reading available)"


ALL_MODES = ("fused", "fp32", "grad", "pairwise", "ragged")


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return HBM_FALLBACK_GBS, "fallback"


def flops_per_x(x, kmax):
    """Algorithmic FP64 flops per argument, by region (FMA = 2; divide, exp,
    rsqrt = 1 each), summed over the actual region membership of x."""
    from paper_2512_10059_gb300 import workloads as W
    na, ma = RA_DEGREES[kmax]
    a = 2 * (na + ma) + 2 + 3 * kmax           # Horner P,Q + divide + exp + kmax (FMA + MUL)
    b = 2 * (5 + 6) + 4 + 3 * kmax             # Horner r_B + divide + exp + 2x + 1/(2x) + steps
    c = 2 + 2 * kmax                           # rsqrt + 1/x + kmax * 2 MUL
    inA = x < W.X0_PRINTED
    inC = x >= W.X1_PRINTED
    nA = int(np.count_nonzero(inA))
    nC = int(np.count_nonzero(inC))
    nB = x.size - nA - nC
    return (a * nA + b * nB + c * nC) / x.size, (nA / x.size, nB / x.size, nC / x.size)


# (n, m) of r_{A,k}, Appendix D
RA_DEGREES = [(6, 9), (6, 10), (6, 10), (4, 12), (8, 9), (4, 13), (8, 9), (4, 13), (8, 9), (8, 9),
              (8, 9), (8, 9), (8, 9), (8, 9), (8, 9), (8, 9), (8, 9), (8, 9), (8, 8), (8, 8), (7, 9),
              (8, 8), (8, 8), (8, 8), (8, 8), (8, 8), (7, 8), (7, 8), (7, 8), (7, 8), (7, 8), (7, 8),
              (7, 8)]


class ClockSampler:
    """nvidia-smi sampling of SM clock and throttle reasons during a region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id):
        self.gpu = gpu_id
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        rows = []
        try:
            for ln in open(self.path):
                parts = [p.strip() for p in ln.split(",")]
                if len(parts) >= 9 and parts[1].replace(".", "").isdigit():
                    rows.append(parts)
        finally:
            try:
                os.unlink(self.path)
            except OSError:
                pass
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        sm = [float(r[1]) for r in rows]
        pw = [float(r[3]) for r in rows if r[3].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[j] for r in rows for j in range(4) if r[5 + j].lower() == "active"})
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": float(rows[0][2]), "reasons": reasons,
                "samples": len(rows), "power_w_max": max(pw) if pw else None}


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def rank_arguments(n, rank):
    """Rank r's shard of the headline workload: elements [r n, (r+1) n) of one
    global argument stream (weak scaling: every rank evaluates n arguments, no
    data-path collective)."""
    from paper_2512_10059_gb300 import workloads as W
    return W.mixture_c2(n, seed=1, start=rank * n)


def max_over_ranks(value, dist, device):
    """The largest of the ranks' values (all ranks receive it)."""
    if dist is None:
        return float(value)
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(world_size, n, kmax, steps, total_ms):
    """Whole-job F_k values/s: every rank's arguments over the slowest rank's time."""
    return world_size * n * (kmax + 1) * steps / (total_ms / 1e3)


def oracle_sample_rate(kmax, seconds=12.0, threads=0, start=0):
    """The binary128 oracle on host cores over consecutive chunks of the same
    workload until ~`seconds` of wall time; returns (values/s, x evaluated)."""
    import oracle
    from paper_2512_10059_gb300 import workloads as W
    chunk = 2048
    done = 0
    t0 = time.perf_counter()
    pool = W.mixture_c2(1 << 21, seed=1)
    while time.perf_counter() - t0 < seconds and done + chunk <= pool.size:
        oracle.boys(pool[done:done + chunk], kmax, nthreads=threads)
        done += chunk
    dt = time.perf_counter() - t0
    return done * (kmax + 1) / dt, done, dt


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    threads = oracle.max_threads()
    for _ in range(args.warmup):
        oracle_sample_rate(KMAX, seconds=0.5)
    step_s = args.ref_step_seconds or min(5.0, 150.0 / max(1, args.steps))
    rates, xs, secs = [], 0, 0.0
    for _ in range(args.steps):
        r, n, dt = oracle_sample_rate(KMAX, seconds=step_s)
        rates.append(r)
        xs += n
        secs += dt
    value = xs * (KMAX + 1) / secs
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * secs / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f128",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "kmax": KMAX, "n": N_PER_GPU,
                   "reference": "binary128 CPU oracle (oracle/boys_oracle.c), bounded samples of the workload"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
                         "sample": f"{xs} arguments of the same mixture in 2048-argument chunks, "
                                   f"~{step_s:.1f} s per step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


def run_ours(args):
    import torch
    modes = args.modes
    ws, rank, local = dist_env()
    dist = None
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    import paper_2512_10059_gb300 as pb
    from paper_2512_10059_gb300 import _lib
    from paper_2512_10059_gb300 import workloads as W

    n = 1 << args.n_log2
    x_host = rank_arguments(n, rank)
    fpx, fracs = flops_per_x(x_host, KMAX)
    x = torch.from_numpy(x_host).to(dev)
    out = torch.empty((KMAX + 1, n), dtype=torch.float64, device=dev)
    stream = torch.cuda.current_stream(dev)
    L = _lib.lib()
    hs = int(stream.cuda_stream)

    def step():
        st = L.boys_eval(x.data_ptr(), n, KMAX, out.data_ptr(), n, hs)
        if st != 0:
            _lib.check("boys_eval", st)

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize(dev)

    for _ in range(args.warmup):
        step()
    barrier()

    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    props = torch.cuda.get_device_properties(dev)
    smi_id = f"GPU-{props.uuid}" if getattr(props, "uuid", None) else str(local)
    with ClockSampler(smi_id) as clk:
        barrier()
        t_start.record(stream)
        for e0, e1 in evs:
            e0.record(stream)
            step()
            e1.record(stream)
        t_end.record(stream)
        torch.cuda.synchronize(dev)
        barrier()
    clocks = clk.summary()
    total_ms = t_start.elapsed_time(t_end)
    launch_ms = [a.elapsed_time(b) for a, b in evs]
    total_ms = max_over_ranks(total_ms, dist, dev)
    ms_per_step = total_ms / args.steps
    value = job_value(ws, n, KMAX, args.steps, total_ms)

    # roofline of the evaluation kernel
    hbm_gbs, hbm_src = peaks()
    sm_mhz, clk_src = sm_clock_mhz(clocks)
    FP64_PEAK_TFLOPS = fp64_peak_tflops(props.multi_processor_count, sm_mhz)
    fp64_peak_source = (f"FP64 nominal: {props.multi_processor_count} SMs x {DFMA_PER_SM_PER_CLOCK} DFMA/clk x 2 flop "
                        f"x {sm_mhz:.0f} MHz ({clk_src})")
    avg_launch_s = statistics.mean(launch_ms) / 1e3
    bytes_per_launch = n * 8 * (KMAX + 2)
    flops_per_launch = n * fpx
    # Primary roof: HBM, the hard floor of stored mode (8 + 8*33 bytes per
    # argument must move).  The paper's algorithmic FP64 work per argument is
    # reported beside it: the kernel runs most of it on the integer pipes (and
    # takes the anchors from tables), so that fraction can exceed 1 and does not
    # bound the kernel.
    roof = {"bound": "hbm", "achieved": bytes_per_launch / avg_launch_s / 1e9, "peak": hbm_gbs,
            "unit": "GB/s", "peak_source": f"{hbm_src} copy bandwidth (MEASURED_PEAKS.json hbm_gbs)"}
    roof["frac"] = roof["achieved"] / roof["peak"]
    same_kernel = TRAFFIC_CAPTURE["sources_sha256"] == kernel_sources_sha256()
    roof["traffic"] = TRAFFIC_CAPTURE["bytes_per_x"] * n if same_kernel else None
    roof["kernel"] = "k_eval_f64<32>"
    roof["algorithmic_bytes_per_x"] = 8 * (KMAX + 2)
    roof["fp64_algorithmic"] = {"flops_per_x": fpx, "achieved": flops_per_launch / avg_launch_s / 1e12,
                                "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s", "peak_source": fp64_peak_source,
                                "frac": flops_per_launch / avg_launch_s / 1e12 / FP64_PEAK_TFLOPS}

    def time_launches(fn, reps):
        """Mean device time of one launch of fn on the stream, after warm-up."""
        for _ in range(args.warmup):
            fn()
        torch.cuda.synchronize(dev)
        a0 = torch.cuda.Event(enable_timing=True)
        a1 = torch.cuda.Event(enable_timing=True)
        a0.record(stream)
        for _ in range(reps):
            fn()
        a1.record(stream)
        torch.cuda.synchronize(dev)
        return a0.elapsed_time(a1) / reps

    # fused consumer on the same arguments (one extra input rho, one output per x)
    fused = None
    if "fused" in modes:
        rho = torch.from_numpy(W.rho_c2(n, seed=2)).to(dev)
        fout = torch.empty(n, dtype=torch.float64, device=dev)
        for _ in range(args.warmup):
            pb.boys_eval_fused(x, rho, KMAX, out=fout)
        barrier()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        for _ in range(args.steps):
            pb.boys_eval_fused(x, rho, KMAX, out=fout)
        f1.record(stream)
        torch.cuda.synchronize(dev)
        fms = f0.elapsed_time(f1) / args.steps
        ffl = n * (fpx + 2 * KMAX + 1)
        fused = {"value": n * (KMAX + 1) / (fms / 1e3), "unit": UNIT, "ms_per_step": fms,
                 "fp64_tflops": ffl / (fms / 1e3) / 1e12,
                 "fp64_frac": ffl / (fms / 1e3) / 1e12 / FP64_PEAK_TFLOPS,
                 "hbm_gbs": n * 24 / (fms / 1e3) / 1e9}
        del rho, fout

    # FP32 tier on the same arguments (rounded to float) and on the FP32-tier
    # workload (parity mixture, N = 2^26) at kmax 4 / 12 / 24 next to FP64
    fp32 = None
    if "fp32" in modes:
        reps = max(5, min(args.steps, 20))
        xf = x.float()
        of = torch.empty((KMAX + 1, n), dtype=torch.float32, device=dev)
        ms32 = time_launches(lambda: pb.boys_eval_f32(xf, KMAX, out=of), reps)
        fp32 = {"kmax32_same_args": {"value": n * (KMAX + 1) / (ms32 / 1e3), "unit": UNIT, "ms": ms32,
                                     "vs_fp64": ms_per_step / ms32,
                                     "hbm_gbs": n * 4 * (KMAX + 2) / (ms32 / 1e3) / 1e9,
                                     "hbm_frac": n * 4 * (KMAX + 2) / (ms32 / 1e3) / 1e9 / hbm_gbs}}
        del xf, of
        x4 = W.mixture_c1(n, seed=4)
        x4d = torch.from_numpy(x4).to(dev)
        x4f = x4d.float()
        for km in (4, 12, 24):
            o32 = torch.empty((km + 1, n), dtype=torch.float32, device=dev)
            o64 = torch.empty((km + 1, n), dtype=torch.float64, device=dev)
            t32 = time_launches(lambda: pb.boys_eval_f32(x4f, km, out=o32), reps)
            t64 = time_launches(lambda: pb.boys_eval(x4d, km, out=o64), reps)
            fp32[f"parity_mix_kmax{km}"] = {
                "fp32_value": n * (km + 1) / (t32 / 1e3), "fp64_value": n * (km + 1) / (t64 / 1e3),
                "unit": UNIT, "fp32_ms": t32, "fp64_ms": t64, "speedup": t64 / t32,
                "fp32_hbm_frac": n * 4 * (km + 2) / (t32 / 1e3) / 1e9 / hbm_gbs}
            del o32, o64
        del x4d, x4f

    # backward: N = 2^24 (2^(n_log2 - 2) when profiling), kmax = 16, x log-uniform
    # [1e-10, 1e3], upstream gradients N(0,1) drawn on the device (seeded)
    grad = None
    if "grad" in modes:
        ng = n >> 2
        kg = 16
        xg_host = W.log_uniform(W.uniform01(W.stream_key(5, 1), ng), 1e-10, 1e3)
        xg = torch.from_numpy(xg_host).to(dev)
        gen = torch.Generator(device=dev)
        gen.manual_seed(6)
        gg = torch.randn((kg + 1, ng), dtype=torch.float64, device=dev, generator=gen)
        dxg = torch.empty(ng, dtype=torch.float64, device=dev)
        gms = time_launches(lambda: pb.boys_grad(xg, gg, kg, out=dxg), max(5, min(args.steps, 20)))
        # algorithmic work: the forward at order kmax + 1 plus kmax + 1 FMAs
        gfl = ng * (flops_per_x(xg_host, kg + 1)[0] + 2 * (kg + 1))
        grad = {"value": ng * (kg + 1) / (gms / 1e3), "unit": "dL/dF_k terms/s", "ms": gms, "n": ng, "kmax": kg,
                "hbm_gbs": ng * 8 * (kg + 3) / (gms / 1e3) / 1e9,
                "fp64_frac": gfl / (gms / 1e3) / 1e12 / FP64_PEAK_TFLOPS}
        del xg, gg, dxg

    # the paper's benchmark workload (Section III, Algorithm 2): k = 12,
    # x uniform on [0, 30]; N = 2^17 here (2^34 pairs), extrapolated to the
    # paper's N = 2^19 by the n^2 law.  The paper's own figure (72 s on an
    # NVIDIA A100) is context, not a target.
    pair = None
    if "pairwise" in modes:
        # N = 2^17 sorted and unsorted (the effect of sorting), then the paper's
        # own size N = 2^19, sorted, one launch (2^(n_log2 - 9) and 2^(n_log2 - 7)
        # when profiling)
        npw = 1 << max(10, args.n_log2 - 9)
        xs, ys, cs = W.pairwise_alg2(npw, 12, seed=8, sort=True)
        xpt, ypt, cpt = (torch.from_numpy(a).to(dev) for a in (xs, ys, cs))
        zpt = torch.empty(npw, dtype=torch.float64, device=dev)
        pms = time_launches(lambda: pb.boys_pairwise(xpt, ypt, cpt, out=zpt), 2)
        xu, yu, _ = W.pairwise_alg2(npw, 12, seed=8, sort=False)
        xut, yut = torch.from_numpy(xu).to(dev), torch.from_numpy(yu).to(dev)
        ums = time_launches(lambda: pb.boys_pairwise(xut, yut, cpt, out=zpt), 1)
        del xpt, ypt, zpt, xut, yut
        nbig = 1 << max(10, args.n_log2 - 7)
        xb, yb, _ = W.pairwise_alg2(nbig, 12, seed=8, sort=True)
        xbt, ybt = torch.from_numpy(xb).to(dev), torch.from_numpy(yb).to(dev)
        zbt = torch.empty(nbig, dtype=torch.float64, device=dev)
        b0 = torch.cuda.Event(enable_timing=True)
        b1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        b0.record(stream)
        pb.boys_pairwise(xbt, ybt, cpt, out=zbt)
        b1.record(stream)
        torch.cuda.synchronize(dev)
        bms = b0.elapsed_time(b1)
        pairs = float(nbig) * nbig
        # algorithmic FP64 work per pair: Algorithm 1 at k = 12 for the region
        # of x_i + x_j (mix from 2^20 random pairs), w = sum_l c_l F_l (13 FMA)
        # and z_i += y_j w (1 FMA)
        rng = np.random.default_rng(0)
        xsum = xb[rng.integers(0, nbig, 1 << 20)] + xb[rng.integers(0, nbig, 1 << 20)]
        pfl, pfr = flops_per_x(xsum, 12)
        pfl += 2 * 13 + 2
        ptf = pairs * pfl / (bms / 1e3) / 1e12
        pair = {"n": nbig, "k": 12, "seconds": bms / 1e3, "pairs_per_s": pairs / (bms / 1e3),
                "value": pairs * 13 / (bms / 1e3), "unit": UNIT, "paper_a100_s_n2^19": 72.0,
                "n_small": npw, "small_sorted_ms": pms, "small_unsorted_ms": ums,
                "roofline": {"bound": "fp64", "algorithmic_flops_per_pair": pfl,
                             "region_fractions_ABC": [round(f, 4) for f in pfr], "achieved": ptf,
                             "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s", "frac": ptf / FP64_PEAK_TFLOPS,
                             "note": "the paper's FP64 work per pair against the nominal FP64 peak; nominal, as the "
                                     "values are: a pair evaluates an expansion of sum_l c_l F_l that its block "
                                     "forms, on the integer pipes (ncu: multiply pipe 60% busy), and no F_l",
                             "hbm": "negligible: x, y are re-read from L2/shared memory, 24 B per i"}}
        del xbt, ybt, zbt, cpt

    ragged = None
    if "ragged" in modes:
        x3, off3, km3 = W.ragged_c3()
        xt3 = torch.from_numpy(x3).to(dev)
        ot3 = torch.from_numpy(off3).to(dev)
        kt3 = torch.from_numpy(km3).to(dev)
        plan = pb.RaggedPlan(xt3, ot3, kt3, autotune=True)
        for _ in range(args.warmup):
            plan.launch()
        barrier()
        r0 = torch.cuda.Event(enable_timing=True)
        r1 = torch.cuda.Event(enable_timing=True)
        r0.record(stream)
        for _ in range(args.steps):
            plan.launch()
        r1.record(stream)
        torch.cuda.synchronize(dev)
        rms = r0.elapsed_time(r1) / args.steps
        # the same batch without a plan: boys_eval_ragged with a grouped-size
        # workspace (device-built tile table, one launch over it)
        wsb = _lib.lib().boys_ragged_workspace_size_grouped(int(km3.size), int(x3.size))
        ws3 = torch.empty(wsb, dtype=torch.uint8, device=dev)
        o3 = torch.empty_like(plan.out)
        pl_ms = time_launches(lambda: pb.boys_eval_ragged(xt3, ot3, kt3, out=o3, out_off=plan.out_off, workspace=ws3),
                              max(5, min(args.steps, 20)))
        # and with a 256-byte workspace: the persistent kernel (the shape
        # boys_eval_ragged_noalloc uses)
        ws_small = torch.empty(256, dtype=torch.uint8, device=dev)
        ps_ms = time_launches(lambda: pb.boys_eval_ragged(xt3, ot3, kt3, out=o3, out_off=plan.out_off,
                                                          workspace=ws_small), max(5, min(args.steps, 20)))
        del ws3, o3, ws_small
        lens = np.diff(off3)
        nval = int(np.sum((km3.astype(np.int64) + 1) * lens))
        rbytes = 8 * x3.size + 8 * nval + 20 * km3.size
        rfl = sum(flops_per_x(x3[off3[j]:off3[j + 1]], int(km3[j]))[0] * int(lens[j]) for j in range(km3.size))
        ragged = {"value": nval / (rms / 1e3), "unit": UNIT, "ms_per_step": rms, "arguments": int(x3.size),
                  "segments": int(km3.size), "mean_kmax_weighted": float(np.sum(km3 * lens) / lens.sum()),
                  "hbm_gbs": rbytes / (rms / 1e3) / 1e9,
                  "fp64_frac": rfl / (rms / 1e3) / 1e12 / FP64_PEAK_TFLOPS, "config": plan.config(),
                  "planless_ms": pl_ms, "planless_vs_plan": pl_ms / rms, "persistent_ms": ps_ms,
                  "launch": "one cudaGraphLaunch: " +
                            ("one kernel over a table of tiles sorted by kmax" if plan.config()["waves"] == 0
                             else "workspace memset + persistent kernel")}
        plan.close()
        del xt3, ot3, kt3, plan

    # end to end through the public API with pinned host buffers: the kernel
    # reads x from host memory and writes F to host memory over the host link
    e2e = None
    if not args.skip_e2e:
        xh = torch.from_numpy(x_host).pin_memory()
        oh = torch.empty((KMAX + 1, n), dtype=torch.float64, pin_memory=True)

        def copy_ms(dst, src, reps=3):
            # best of `reps` timed copies after one untimed one: the floor the
            # link allows (a single copy can be slowed by other host traffic)
            dst.copy_(src, non_blocking=True)
            best = float("inf")
            for _ in range(reps):
                c0 = torch.cuda.Event(enable_timing=True)
                c1 = torch.cuda.Event(enable_timing=True)
                c0.record(stream)
                dst.copy_(src, non_blocking=True)
                c1.record(stream)
                torch.cuda.synchronize(dev)
                best = min(best, c0.elapsed_time(c1))
            return best

        # the host link's own floor for this step, measured here with copy
        # engines: x in and all of F out (the link is full duplex)
        d2h_ms = copy_ms(oh, out)
        h2d_ms = copy_ms(x, xh)
        del out
        torch.cuda.empty_cache()

        def e2e_step():
            pb.boys_eval_host(xh, KMAX, out=oh, stream=stream, device=dev)

        for _ in range(2):
            e2e_step()
        barrier()
        k_e2e = max(2, min(args.steps, 5))
        g0 = torch.cuda.Event(enable_timing=True)
        g1 = torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        for _ in range(k_e2e):
            e2e_step()
        g1.record(stream)
        torch.cuda.synchronize(dev)
        barrier()
        ems = torch.tensor([g0.elapsed_time(g1)], dtype=torch.float64, device=dev)
        if dist is not None:
            dist.all_reduce(ems, op=dist.ReduceOp.MAX)
        ems = float(ems.item())
        d2h_bytes = 8 * (KMAX + 1) * n
        e2e = {"value": ws * n * (KMAX + 1) * k_e2e / (ems / 1e3), "unit": UNIT,
               "h2d_bytes_per_step": 8 * n, "d2h_bytes_per_step": d2h_bytes,
               "ms_per_step": ems / k_e2e, "steps": k_e2e,
               "api": "boys_eval_host: pinned host x and F; the kernel moves them over NVLink-C2C",
               "link_bound_ms": max(d2h_ms, h2d_ms),
               "link_measured": {"d2h_ms": d2h_ms, "d2h_gbs": d2h_bytes / (d2h_ms / 1e3) / 1e9,
                                 "h2d_ms": h2d_ms, "h2d_gbs": 8 * n / (h2d_ms / 1e3) / 1e9,
                                 "how": "cudaMemcpyAsync of the same bytes, pinned host <-> device, CUDA events, best of 3"}}
        del xh, oh

    cpu = None
    if rank == 0 and not args.skip_cpu:
        import oracle
        r, xs, dt = oracle_sample_rate(KMAX, seconds=args.cpu_seconds)
        cpu = {"value": r, "unit": UNIT, "cores": oracle.max_threads(), "kind": "oracle",
               "sample": f"{xs} arguments of the same mixture (binary128, {dt:.1f} s wall)"}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD if args.n_log2 == 26 else f"{WORKLOAD}_profiling_n2^{args.n_log2}",
                       "kmax": KMAX, "n_per_gpu": n, "output": "order-major [33][N] FP64",
                       "region_fractions_ABC": [round(f, 4) for f in fracs],
                       "l2": "inputs larger than L2 (x 0.54 GB read, 17.7 GB written per step); no flush",
                       "parallelism": f"replicas x{ws}, no data-path collective"},
            "roofline": roof, "cpu_baseline": cpu, "e2e": e2e,
            "gpu_launches": args.steps,
            "clocks": clocks, "modes": {"fused_kmax32": fused, "ragged_4096seg": ragged, "fp32_tier": fp32, "grad_kmax16": grad,
                      "pairwise_alg2_k12": pair},
        }
        print(json.dumps(line))
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser(description=__doc__.splitlines()[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--ref-step-seconds", type=float, default=None)
    ap.add_argument("--n-log2", type=int, default=26,
                    help="arguments per GPU = 2^n (26 is the benchmarked workload; smaller only for profiling)")
    ap.add_argument("--skip-e2e", action="store_true")
    ap.add_argument("--skip-cpu", action="store_true")
    ap.add_argument("--modes", default=",".join(ALL_MODES),
                    help="comma list of the secondary modes to time (" + ",".join(ALL_MODES) + "), or none")
    ap.add_argument("--skip-modes", action="store_true", help="same as --modes none")
    args = ap.parse_args()
    args.modes = set() if args.skip_modes or args.modes == "none" else set(args.modes.split(","))
    if args.modes - set(ALL_MODES):
        ap.error(f"unknown modes {sorted(args.modes - set(ALL_MODES))}")
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
