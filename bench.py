#!/usr/bin/env python
"""Benchmark of the block-scaled e4m3 fast-matmul hot path on B200.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
                    [--n 8192] [--levels 1] [--realization phi_optimal]
                    [--scale-mode fp32|ue8m0] [--block-k 32|128] [--no-variants]

One "step" is one pass of the whole hot path (fmm_matmul: pre-addition + quantization of both
operands, the 7^levels block-scaled fp8 products on the tensor cores, fused post-addition) over one
pair of synthetic N(0,1) fp32 operands.  The metric is effective TFLOP/s = 2*M*N*K / time.

The path does not shard (one GPU per matmul, no exchange step): with --gpus N every rank runs an
independent replica of the same problem and the value is the sum over ranks ("replicas only").

--impl reference times the CPU oracle (oracle/, test infrastructure) on a bounded sample instead.
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
sys.path.insert(0, ROOT)

METRIC = "effective fp8 TFLOP/s (2*M*N*K/t), one-level rank-7 block-scaled e4m3 matmul, n=8192"
UNIT = "TFLOP/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=8192)
    ap.add_argument("--shape", default="", help="M,K,N of a rectangular problem (profiling captures); overrides --n")
    ap.add_argument("--levels", type=int, default=1)
    ap.add_argument("--realization", default="phi_optimal")
    ap.add_argument("--scale-mode", default="fp32", choices=["fp32", "ue8m0"])
    ap.add_argument("--block-k", type=int, default=32, choices=[32, 128])
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--ref-n", type=int, default=0, help="reference arm: size of one oracle step (0 = --n / 2, --n / 4 with few host threads)")
    ap.add_argument("--cpu-baseline-n", type=int, default=0, help="size of the oracle pass of the cpu_baseline leg (0 = --n)")
    return ap.parse_args()


# ------------------------------------------------------------------------------------------------
def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return {"hbm_gbs": float(d["hbm_gbs"]), "bf16_tflops": float(d["bf16_tflops"]),
                "bf16_tflops_sustained": float(d.get("bf16_tflops_sustained", d["bf16_tflops"])), "source": "measured"}
    return {"hbm_gbs": 6650.0, "bf16_tflops": 1590.0, "bf16_tflops_sustained": 1400.0, "source": "fallback"}


class ClockSampler:
    """Samples SM clock and throttle reasons with nvidia-smi while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.proc, self.lines = index, None, []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "25"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=2)
        except Exception:
            pass
        sm, smax, power, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1])); smax.append(float(f[2])); power.append(float(f[3]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        busy = sorted(sm)[len(sm) // 2:]          # the loaded half of the samples
        return {"sm_mhz": statistics.median(busy), "sm_max_mhz": max(smax), "power_w_max": max(power),
                "samples": len(sm), "reasons": sorted(reasons)}


def reduce_max_ms(ms, dist=None, device="cpu"):
    """Time of the slowest rank (replicas run independently; the job is as slow as its slowest replica)."""
    if dist is None:
        return ms
    import torch
    t = torch.tensor([ms], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(flop_per_replica, world, ms_slowest):
    """Whole-job value for `world` independent replicas timed by the slowest one, in TFLOP/s."""
    return world * flop_per_replica / (ms_slowest * 1e-3) / 1e12


def algorithmic_work(M, N, K, levels, rank, scale_bytes, blk):
    """Flops of the products and HBM bytes the method itself must move (fused post-addition):
    read A and B once, write then read the quantized operands and their scales once, write C once."""
    f = (rank / 8.0) ** levels if levels > 0 else 1.0
    r = (rank / 4.0) ** levels if levels > 0 else 1.0
    flops = 2.0 * M * N * K * f
    qbytes = r * (M * K + K * N) * (1.0 + scale_bytes / blk)
    enc_bytes = 4.0 * (M * K + K * N) + qbytes
    gemm_bytes = qbytes + 4.0 * M * N
    return flops, enc_bytes, gemm_bytes


ARM_PAUSE_S = 0.5          # idle time before each variant / rectangular arm (see the note where it is used)
SPEC_FP8_TFLOPS, SPEC_HBM_GBS = 4500.0, 8000.0      # B200 nominal dense fp8 and HBM3e figures


def combined_roofline_ms(M, N, K, levels, rank, mode, blk, fp8_peak_tflops, hbm_gbs):
    """Combined roofline time of one pass: the product phase at the fp8 tensor peak plus the algorithmic HBM bytes
    (pre-addition + quantization, operand reads of the products, one write of C) at the copy bandwidth, phases
    serialized.  The same formula for every scale mode."""
    scale_bytes = 1 if mode.startswith("ue8m0") else 4
    flops, enc_bytes, gemm_bytes = algorithmic_work(M, N, K, levels, rank, scale_bytes, blk)
    return (flops / (fp8_peak_tflops * 1e12) + (enc_bytes + gemm_bytes) / (hbm_gbs * 1e9)) * 1e3


def overlap_bound_ms(M, N, K, levels, rank, mode, blk, fp8_peak_tflops, hbm_gbs):
    """The same two terms with the phases fully overlapped: max(tensor time, HBM time).  No schedule of this path
    can reach it (the products need the encoded operands), it brackets the serialized roofline from below."""
    scale_bytes = 1 if mode.startswith("ue8m0") else 4
    flops, enc_bytes, gemm_bytes = algorithmic_work(M, N, K, levels, rank, scale_bytes, blk)
    return max(flops / (fp8_peak_tflops * 1e12), (enc_bytes + gemm_bytes) / (hbm_gbs * 1e9)) * 1e3


def alu_floor_ms(M, N, K, levels, rank, mode, blk):
    """fp32 scales only: CUDA-core time of the per-block promotion acc += P * (sA * sB) that the chosen algorithm
    needs (the tensor core cannot apply a per-row x per-column fp32 factor per K block): M*N*(K/blk) elements,
    1 mul + 1 fma each (1 fma with 128 x 128 weight tiles), on 148 SMs x 128 fp32 lanes at the 1.965 GHz maximum
    clock.  A floor of this implementation's design, reported beside the roofline and not part of it."""
    if mode.startswith("ue8m0"):
        return 0.0
    f = (rank / 8.0) ** levels if levels > 0 else 1.0
    ops = 1.0 if "tile" in mode else 2.0
    return ops * M * N * (K / blk) * f / (148 * 128 * 1.965e9) * 1e3


def roofline_fractions(M, N, K, levels, rank, mode, blk, ms, pk):
    """Fractions of the combined roofline against the measured and the nominal peaks, plus the ALU floor."""
    meas = combined_roofline_ms(M, N, K, levels, rank, mode, blk, 2.0 * pk["bf16_tflops"], pk["hbm_gbs"])
    spec = combined_roofline_ms(M, N, K, levels, rank, mode, blk, SPEC_FP8_TFLOPS, SPEC_HBM_GBS)
    return {"combined_roofline_ms": meas, "combined_frac": meas / ms,
            "combined_roofline_spec_ms": spec, "combined_frac_spec": spec / ms,
            "overlap_bound_ms": overlap_bound_ms(M, N, K, levels, rank, mode, blk, 2.0 * pk["bf16_tflops"], pk["hbm_gbs"]),
            "overlap_bound_spec_ms": overlap_bound_ms(M, N, K, levels, rank, mode, blk, SPEC_FP8_TFLOPS, SPEC_HBM_GBS),
            "alu_floor_ms": alu_floor_ms(M, N, K, levels, rank, mode, blk)}


def run_ours(args):
    import numpy as np
    import torch
    from paper_2609_26077_b200 import fmm, realizations as P

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank_id = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if not torch.cuda.is_available():
        raise SystemExit("bench.py: no CUDA device (the hot path has no CPU fallback)")
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    n, K_steps, W_steps = args.n, args.steps, max(args.warmup, 3)
    M = N = K = n
    if args.shape:
        M, K, N = (int(x) for x in args.shape.split(","))
    pk = peaks()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1234 + rank_id)
    A = torch.randn(M, K, device="cuda", generator=gen)
    B = torch.randn(K, N, device="cuda", generator=gen)
    C = torch.empty(M, N, device="cuda")

    def make_plan(name, levels, blk, mode):
        # mode "fp32+tile128": fp32 scales with one weight-side scale per 128 x 128 tile (App. E.5)
        kw = dict(block_k=blk, scale_mode=mode.split("+")[0], b_tile_n=128 if mode.endswith("+tile128") else 0)
        if name == "cubic" or levels == 0:
            return fmm.Plan(levels=0, **kw)
        return fmm.Plan(*P.get(name), levels=levels, **kw)

    def barrier():
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    def time_steps(fn, steps, warm):
        for _ in range(warm):
            fn()
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            fn()
        e1.record()
        barrier()
        return reduce_max_ms(e0.elapsed_time(e1), dist, "cuda") / steps

    plan = make_plan(args.realization, args.levels, args.block_k, args.scale_mode)
    ws = plan.workspace(M, N, K)
    sampler = ClockSampler(local)

    # ---- timed region 1: K steps of the public call, inputs resident in HBM
    sampler.start()
    ms_step = time_steps(lambda: plan.matmul(A, B, out=C, workspace=ws), K_steps, W_steps)
    launches_per_step = plan.last_launch_count()

    # ---- timed region 2: the same K steps with the two phases bracketed by events (roofline of the dominant kernel)
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(K_steps)]
    barrier()
    for i in range(K_steps):
        ev[i][0].record()
        plan.encode_only(A, B, workspace=ws)
        ev[i][1].record()
        plan.multiply_only(M, N, K, C, workspace=ws)
        ev[i][2].record()
    barrier()
    enc_ms = statistics.mean(e[0].elapsed_time(e[1]) for e in ev)
    mul_ms = statistics.mean(e[1].elapsed_time(e[2]) for e in ev)
    clocks = sampler.stop()
    status = plan.device_status()

    # ---- end to end: the library's host-operand call, host buffers in pinned memory, copies inside the timed region.
    # Two streams, each with its own device workspace and its own result buffer, take alternate steps, so that one
    # step's upload overlaps the previous step's product and download (every step still moves all of its inputs
    # and its result across the host link inside the timed region).
    Ah = torch.empty(M, K, dtype=torch.float32, pin_memory=True)
    Bh = torch.empty(K, N, dtype=torch.float32, pin_memory=True)
    Ah.copy_(A); Bh.copy_(B)
    lanes = 2
    e2e_streams = [torch.cuda.Stream() for _ in range(lanes)]
    e2e_ws = [plan.host_workspace(M, N, K) for _ in range(lanes)]
    Ch = [torch.empty(M, N, dtype=torch.float32, pin_memory=True) for _ in range(lanes)]
    e2e_count = [0]

    def e2e_step():
        i = e2e_count[0] % lanes
        e2e_count[0] += 1
        plan.matmul_host(Ah, Bh, Ch[i], e2e_ws[i], stream=e2e_streams[i])

    def time_e2e(steps, warm):
        cur = torch.cuda.current_stream()
        for _ in range(warm):
            e2e_step()
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for st in e2e_streams:
            st.wait_stream(cur)
        e0.record(cur)
        for st in e2e_streams:
            st.wait_event(e0)
        for _ in range(steps):
            e2e_step()
        for st in e2e_streams:
            cur.wait_stream(st)
        e1.record(cur)
        barrier()
        return reduce_max_ms(e0.elapsed_time(e1), dist, "cuda") / steps

    e2e_steps = max(4, min(K_steps, 10))
    ms_e2e = time_e2e(e2e_steps, 4)
    e2e_ok = bool(torch.equal(Ch[0], Ch[1]) and torch.equal(Ch[0], C.cpu()))

    flop_eff = 2.0 * M * N * K
    value = replica_throughput(flop_eff, world, ms_step)
    scale_bytes = 4 if args.scale_mode == "fp32" else 1
    rank_r = plan.rank if args.levels > 0 else 8
    flops_alg, enc_bytes, gemm_bytes = algorithmic_work(M, N, K, args.levels, rank_r, scale_bytes, args.block_k)
    fp8_peak = 2.0 * pk["bf16_tflops"]           # nominal fp8 : bf16 ratio applied to the measured bf16 burst
    hbm = pk["hbm_gbs"]

    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K_steps, "warmup": W_steps,
        "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "fp8_e4m3", "data": "synthetic",
        "config": {"workload": (f"n={n} square" if not args.shape else f"M,K,N={M},{K},{N}") +
                               f", {args.levels} level(s), {args.realization}, A,B iid N(0,1) fp32",
                   "scale_mode": args.scale_mode, "block_k": args.block_k, "M": M, "N": N, "K": K,
                   "l2": f"inputs larger than L2 ({4 * M * K / 1e6:.0f} + {4 * K * N / 1e6:.0f} MB fp32 operands, {4 * M * N / 1e6:.0f} MB output)",
                   "multi_gpu": "replicas only"},
        "clocks": clocks,
        "gpu_launches": launches_per_step * K_steps,
        "e2e": {"value": replica_throughput(flop_eff, world, ms_e2e), "unit": UNIT, "ms_per_step": ms_e2e,
                "h2d_bytes_per_step": 4 * (M * K + K * N), "d2h_bytes_per_step": 4 * M * N, "steps": e2e_steps,
                "call": "fmm_matmul_host, 2 streams x own workspace (uploads overlap the other stream's product and download)",
                "result_matches_device_path": e2e_ok},
        "phases": {"encode_ms": enc_ms, "multiply_ms": mul_ms,
                   "encode_hbm_frac": enc_bytes / (enc_ms * 1e-3) / 1e9 / hbm,
                   "encode_gbs": enc_bytes / (enc_ms * 1e-3) / 1e9,
                   "multiply_tflops": flops_alg / (mul_ms * 1e-3) / 1e12},
        "device_status": status[1],
    }
    # dominant kernel = the tcgen05 product kernel, timed live above (events around fmm_multiply_only).
    # DRAM traffic per launch comes from one-pass ncu captures (two counters, mean of two launches) of the same product at
    # the same size; the live C tiles and the operand streams compete for L2, so traffic does not scale with M*N and only captured sizes are reported.
    measured = {("fp32", 32, 8192): 1569.6e6, ("ue8m0", 32, 8192): 1276.9e6, ("fp32", 128, 8192): 1391.1e6,
                ("ue8m0", 32, 4096): 102.5e6}
    traffic = None
    if args.levels == 1 and M == N == K and args.realization == "phi_optimal":
        traffic = measured.get((args.scale_mode, args.block_k, M))
    mode_name = args.scale_mode
    out["roofline"] = {"kernel": "fmm_gemm_kernel", "bound": "tensor",
                       "achieved": flops_alg / (mul_ms * 1e-3) / 1e12, "peak": fp8_peak, "unit": "TFLOP/s",
                       "frac": flops_alg / (mul_ms * 1e-3) / 1e12 / fp8_peak,
                       "frac_spec": flops_alg / (mul_ms * 1e-3) / 1e12 / SPEC_FP8_TFLOPS,
                       "traffic": traffic,
                       "traffic_source": ("ncu dram__bytes_read.sum + dram__bytes_write.sum, one-pass capture of the "
                                          "same product at this size" if traffic else None),
                       "algorithmic_bytes": gemm_bytes,
                       "peak_source": f"2 x {pk['source']} bf16 burst ({pk['bf16_tflops']} TF/s); spec {SPEC_FP8_TFLOPS} TF/s, {SPEC_HBM_GBS} GB/s",
                       "hbm_peak_gbs": hbm}
    out["roofline"].update(roofline_fractions(M, N, K, args.levels, rank_r, mode_name, args.block_k, ms_step, pk))

    if rank_id == 0 and world == 1 and not args.no_variants:
        variants = []
        todo = [("cubic", 0, args.block_k, args.scale_mode), ("strassen", 1, args.block_k, args.scale_mode),
                ("phi_optimal", 1, 32, "ue8m0"), ("cubic", 0, 32, "ue8m0"),
                ("phi_optimal", 1, 128, "fp32"), ("cubic", 0, 128, "fp32"), ("phi_optimal", 1, 32, "fp32"),
                ("phi_optimal", 1, 128, "fp32+tile128"), ("cubic", 0, 128, "fp32+tile128"),
                ("phi_optimal", 2, 32, "ue8m0")]
        seen = {(args.realization, args.levels, args.block_k, args.scale_mode)}
        for name, lv, blk, mode in todo:
            if (name, lv, blk, mode) in seen:
                continue
            seen.add((name, lv, blk, mode))
            p2 = make_plan(name, lv, blk, mode)
            w2 = p2.workspace(M, N, K)
            # Every arm starts from an idle GPU: after about 60 ms of back-to-back tensor-heavy steps this part lowers
            # its SM clock to about 1.7 GHz (reason: software power cap) and an arm timed right behind another one
            # came out up to 11 % slower than the same arm timed alone.
            time.sleep(ARM_PAUSE_S)
            ms = time_steps(lambda: p2.matmul(A, B, out=C, workspace=w2), 10, 5)
            v = {"realization": name, "levels": lv, "block_k": blk, "scale_mode": mode,
                 "ms_per_step": ms, "value": flop_eff / (ms * 1e-3) / 1e12}
            v.update(roofline_fractions(M, N, K, lv, p2.rank if lv > 0 else 8, mode, blk, ms, pk))
            if lv >= 2:
                # outside the algorithmic bytes: the outer decoder reads the 7 partially decoded products of every
                # parent and writes its four blocks (its own kernel, one extra HBM round trip per outer level)
                v["decode_round_trip_bytes"] = sum(4.0 * M * N * ((7.0 / 4.0) ** l + (7.0 / 4.0) ** (l - 1)) for l in range(1, lv))
            variants.append(v)
            p2.close()
        out["variants"] = variants
        out["variants_protocol"] = (f"each arm: {ARM_PAUSE_S} s idle, 5 warm-up + 10 timed back-to-back steps (a burst of about "
                                    "10 - 30 ms at the maximum SM clock; sustained back-to-back load of the tensor-heavy "
                                    "modes runs power-capped at about 1.7 GHz and 10 % slower)")
        # rectangular LLM-shaped case: M, K, N = 16384, 8192, 8192, A = N(0,1) rows with per-column lognormal(0, 1.5)
        # outlier channels, B ~ N(0, 0.02^2); rank-7 at one level next to the cubic product in the same kernels
        if M == N == K == 8192 and args.levels == 1:
            Mr, Kr, Nr = 16384, 8192, 8192
            Ar = torch.randn(Mr, Kr, device="cuda", generator=gen) * torch.exp(1.5 * torch.randn(Kr, device="cuda", generator=gen))
            Br = 0.02 * torch.randn(Kr, Nr, device="cuda", generator=gen)
            Cr = torch.empty(Mr, Nr, device="cuda")
            rect = []
            for name, lv, blk, mode in [("phi_optimal", 1, args.block_k, args.scale_mode), ("strassen", 1, args.block_k, args.scale_mode),
                                        ("cubic", 0, args.block_k, args.scale_mode),
                                        ("phi_optimal", 1, 128, "fp32"), ("cubic", 0, 128, "fp32"),
                                        ("phi_optimal", 1, 32, "ue8m0"), ("strassen", 1, 32, "ue8m0"), ("cubic", 0, 32, "ue8m0")]:
                p2 = make_plan(name, lv, blk, mode)
                w2 = p2.workspace(Mr, Nr, Kr)
                time.sleep(ARM_PAUSE_S)
                ms = time_steps(lambda: p2.matmul(Ar, Br, out=Cr, workspace=w2), 10, 5)
                v = {"realization": name, "levels": lv, "block_k": blk, "scale_mode": mode, "ms_per_step": ms,
                     "value": 2.0 * Mr * Nr * Kr / (ms * 1e-3) / 1e12}
                v.update(roofline_fractions(Mr, Nr, Kr, lv, p2.rank if lv > 0 else 8, mode, blk, ms, pk))
                rect.append(v)
                p2.close()
                del w2
            out["rectangular"] = {"workload": f"M,K,N={Mr},{Kr},{Nr}, A rows N(0,1) x per-column lognormal(0,1.5) factors, B iid N(0,0.02)",
                                  "arms": rect}
            del Ar, Br, Cr
            torch.cuda.empty_cache()
        # the paper's timing protocol (App. E.7): interleaved repetitions across realizations, median and a
        # bootstrap 95 % interval of the median, so that clock drift hits every arm alike
        arms = [("cubic", 0), ("strassen", 1), ("phi_optimal", 1)]
        plans = [(nm, make_plan(nm, lv, args.block_k, args.scale_mode)) for nm, lv in arms]
        wss = [pl.workspace(M, N, K) for _, pl in plans]
        for (_, pl), w2 in zip(plans, wss):
            for _ in range(5):
                pl.matmul(A, B, out=C, workspace=w2)
        torch.cuda.synchronize()
        samples = {nm: [] for nm, _ in arms}
        for _ in range(25):
            for (nm, pl), w2 in zip(plans, wss):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                pl.matmul(A, B, out=C, workspace=w2)
                e1.record()
                e1.synchronize()
                samples[nm].append(e0.elapsed_time(e1))
        import numpy as _np
        rng = _np.random.default_rng(0)
        inter = {}
        for nm, xs in samples.items():
            xs = _np.array(xs)
            boot = _np.median(rng.choice(xs, size=(2000, xs.size), replace=True), axis=1)
            inter[nm] = {"median_ms": float(_np.median(xs)), "ci95_ms": [float(_np.percentile(boot, 2.5)), float(_np.percentile(boot, 97.5))],
                         "value": flop_eff / (float(_np.median(xs)) * 1e-3) / 1e12}
        out["interleaved"] = {"repetitions": 25, "scale_mode": args.scale_mode, "block_k": args.block_k, "arms": inter}
        for _, pl in plans:
            pl.close()
        # RMS relative error vs the fp64 product, and ratios vs cubic fp8 in the same quantizer
        ref = fmm.fmm_ref_gemm_fp64(A, B)
        errs = {}
        for name, lv in [("cubic", 0), ("strassen", 1), ("winograd", 1), ("phi_optimal", 1)]:
            p2 = make_plan(name, lv, args.block_k, args.scale_mode)
            errs[name] = fmm.rel_frobenius(p2.matmul(A, B, out=C, workspace=p2.workspace(M, N, K)), ref)
            p2.close()
        out["error"] = {"rel_frobenius": errs, "ratio_vs_cubic": {k: v / errs["cubic"] for k, v in errs.items()},
                        "predicted_sqrt_phi_over_8": {"strassen": 2.0, "winograd": 7 ** 0.5, "phi_optimal": 5 / 3}}
        # the measurement step itself: the error statistics read 12 bytes per element (C fp32 + C_ref fp64), HBM-bound;
        # the fp64 reference product is off the timed path and is reported for the record
        out3 = torch.empty(3, dtype=torch.float64, device="cuda")
        ms_stats = time_steps(lambda: fmm.fmm_error_stats(C, ref, out3=out3), 10, 3)
        ms_ref = time_steps(lambda: fmm.fmm_ref_gemm_fp64(A, B, out=ref), 2, 1)
        out["measurement_kernels"] = {
            "error_stats": {"ms": ms_stats, "gbs": 12.0 * M * N / (ms_stats * 1e-3) / 1e9,
                            "hbm_frac": 12.0 * M * N / (ms_stats * 1e-3) / 1e9 / hbm, "bytes": 12.0 * M * N},
            "ref_gemm_fp64": {"ms": ms_ref, "tflops_fp64": 2.0 * M * N * K / (ms_ref * 1e-3) / 1e12}}
        out["cpu_baseline"] = cpu_baseline(args)
    elif rank_id == 0:
        out["cpu_baseline"] = None

    if rank_id == 0:
        print(json.dumps(out), flush=True)
    plan.close()
    if dist is not None:
        dist.destroy_process_group()


# ------------------------------------------------------------------------------------------------
def _oracle_step(n, levels, realization, blk, mode, seed=0):
    """One oracle pass over an n x n x n problem of the benchmarked kind; returns the seconds it took."""
    import numpy as np
    from oracle import oracle as O, realizations as R
    from paper_2609_26077_b200 import workloads as Wl
    A, B = Wl.gaussian(n, n, n, seed)
    key = {"phi_optimal": "phi_optimal", "strassen": "strassen", "winograd": "winograd", "cubic": "cubic"}[realization]
    U, V, W = [np.array(R.to_float(x), dtype=np.float32) for x in R.NAMED[key]()]
    t0 = time.perf_counter()
    O.fused_fmm(A, B, U, V, W, levels=levels, blk=blk, mode=O.SCALE_FP32 if mode == "fp32" else O.SCALE_UE8M0)
    return time.perf_counter() - t0


def cpu_baseline(args):
    """The oracle as it stands, timed once on the benchmarked configuration itself (n = 8192: about half a minute on
    16 cores); with fewer than 8 host threads one pass at half the size is timed instead and the sample says so."""
    from oracle import oracle as O
    n = args.cpu_baseline_n or (args.n if O.num_threads() >= 8 else args.n // 2)
    t = _oracle_step(n, args.levels, args.realization, args.block_k, args.scale_mode)
    what = "the benchmarked size" if n == args.n else f"a smaller instance of the n={args.n} workload (its cost grows as n^3)"
    return {"value": 2.0 * n ** 3 / t / 1e12, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle", "seconds": t,
            "sample": f"one oracle pass at n={n}, {what} (same realization, levels, quantizer); value = 2n^3/t"}


def run_reference(args):
    if int(os.environ.get("RANK", "0")) != 0:
        return
    from oracle import oracle as O
    # bounded sample: one step = one oracle pass at half the benchmarked size (an eighth of the work; about 4 s on 16
    # cores at n = 4096, so that warm-up plus 20 steps end within a few minutes), a quarter with few host threads
    n = args.ref_n or (args.n // 2 if O.num_threads() >= 8 else args.n // 4)
    for _ in range(args.warmup):
        _oracle_step(n, args.levels, args.realization, args.block_k, args.scale_mode)
    ts = [_oracle_step(n, args.levels, args.realization, args.block_k, args.scale_mode, seed=i)
          for i in range(args.steps)]
    t = sum(ts) / len(ts)
    val = 2.0 * n ** 3 / t / 1e12
    sample = (f"each step = one oracle pass at n={n} (bounded sample of the n={args.n} workload: same realization, levels, "
              f"quantizer and operand family, smaller matrices), value = 2n^3/t")
    out = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": t * 1e3, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "fp8_e4m3", "data": "synthetic",
           "config": {"workload": f"n={args.n} square, {args.levels} level(s), {args.realization}, A,B iid N(0,1) fp32",
                      "scale_mode": args.scale_mode, "block_k": args.block_k, "M": args.n, "N": args.n, "K": args.n,
                      "l2": "not applicable (host cores)", "multi_gpu": "replicas only", "sample_n": n},
           "cpu_baseline": {"value": val, "unit": UNIT, "cores": O.num_threads(), "kind": "oracle", "sample": sample},
           "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "gpu_launches": 0}
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    a = parse()
    if a.impl == "reference":
        run_reference(a)
    else:
        run_ours(a)
