"""Performance cases: the work a user of this library has it do, through its public entry points.

Four kinds of work, with the shapes, realizations and operand families of the library's own benchmark and error-sweep
configurations (`bench.py`, `paper_2609_26077_b200/sweep.py`):

  matmul  C = A @ B through a realization (Plan.matmul: encode, R^levels fp8 products, decode), operands on the device
  host    the same product with operands and result in pinned host memory (Plan.matmul_host)
  ref     the fp64 reference product that every trial of an error sweep is measured against (fmm_ref_gemm_fp64)
  stats   the error statistics of one result against that reference (fmm_error_stats)

listed() names the representative cases, draw() gives further ones of the same ranges, prepare() makes what a program
has in hand before the call, run() is one pass, work() the bytes and operations a pass cannot do without and
tolerance() how far another correct implementation's results may be off.
"""
from __future__ import annotations

import math

import torch

from paper_2609_26077_b200 import fmm, realizations

REALIZATIONS = ["strassen", "winograd", "phi_optimal"]
# (block_k, scale mode, weight-side tile, bf16 pre-round of the weight side): the quantizers a plan can be made with
QUANTIZERS = [(32, "fp32", 0, False), (32, "ue8m0", 0, False), (128, "fp32", 0, False), (128, "fp32", 128, True)]


def _matmul(name, M, K, N, realization, levels, quantizer, family, kind="matmul"):
    blk, mode, tile, bf16 = quantizer
    return {"name": name, "kind": kind, "M": M, "K": K, "N": N, "realization": realization, "levels": levels,
            "block_k": blk, "scale_mode": mode, "b_tile_n": tile, "b_bf16": bf16, "family": family}


def listed():
    b32, mx, b128, tiles = QUANTIZERS
    return [
        # sweep c1, the smallest product there is use for: launches and host work are the whole cost
        _matmul("c1_n256_strassen", 256, 256, 256, "strassen", 1, b32, "gaussian"),
        # a few row blocks of activations against a weight matrix, no dimension a multiple of 512
        _matmul("ragged_ue8m0", 1280, 3328, 2816, "phi_optimal", 1, mx, "llm"),
        # sweep c5: deep recursion at a moderate size, operands over six decades of magnitude
        _matmul("c5_n2048_three_levels", 2048, 2048, 2048, "phi_optimal", 3, b32, "scaled_gaussian"),
        # sweep c2, the arm every ratio is taken against: the cubic product under the paper's quantizer
        _matmul("c2_n4096_cubic", 4096, 4096, 4096, "cubic", 0, b32, "gaussian"),
        # sweep c2 at the paper's own block size
        _matmul("c2_n4096_block128", 4096, 4096, 4096, "winograd", 1, b128, "uniform"),
        # sweep c9: weight tiles of 128 x 128 and the bf16 pre-round of a deployed kernel
        _matmul("c9_n4096_weight_tiles", 4096, 4096, 4096, "phi_optimal", 1, tiles, "llm"),
        # the headline of bench.py (sweep c3)
        _matmul("c3_n8192_headline", 8192, 8192, 8192, "phi_optimal", 1, b32, "gaussian"),
        # sweep c3 at two levels with the scales the tensor cores apply themselves
        _matmul("c3_n8192_two_levels", 8192, 8192, 8192, "phi_optimal", 2, mx, "gaussian"),
        # sweep c4: the rectangular LLM shape, the largest product of the benchmark
        _matmul("c4_llm_shape", 16384, 8192, 8192, "strassen", 1, mx, "llm"),
        # bench.py's end-to-end leg: operands come from, and the result goes back to, pinned host memory
        _matmul("host_n4096", 4096, 4096, 4096, "phi_optimal", 1, b32, "gaussian", kind="host"),
        # one per trial of sweep c5
        {"name": "ref_n2048", "kind": "ref", "M": 2048, "K": 2048, "N": 2048, "family": "student_t3"},
        # one per realization and trial of sweep c2
        {"name": "stats_n4096", "kind": "stats", "M": 4096, "N": 4096},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dim(rng, unit, lo, hi):
    """A multiple of unit, spread over the logarithm of [lo, hi]; odd multiples are as likely as even ones."""
    return unit * max(1, round(_log_uniform(rng, max(lo, unit), hi) / unit))


def draw(rng):
    kind = rng.choices(["matmul", "host", "ref", "stats"], [15, 1, 2, 2])[0]
    if kind == "ref":
        while True:
            M, N, K = _dim(rng, 64, 128, 4096), _dim(rng, 64, 128, 4096), _dim(rng, 16, 128, 4096)
            if M * N * K <= 2048 ** 3:
                return {"kind": kind, "M": M, "K": K, "N": N, "family": rng.choice(["gaussian", "uniform", "student_t3"])}
    if kind == "stats":
        return {"kind": kind, "M": _dim(rng, 2, 128, 8192), "N": _dim(rng, 1, 128, 8192)}
    realization = rng.choice(REALIZATIONS + ["cubic"])
    levels = 0 if realization == "cubic" else rng.choices([1, 2, 3], [4, 2, 1])[0]
    quantizer = rng.choice(QUANTIZERS)
    family = rng.choice(["gaussian", "uniform", "llm", "scaled_gaussian", "student_t3"])
    unit = 128 << levels
    most = 4096 ** 3 if kind == "host" else 8192 ** 3
    while True:
        M, K, N = _dim(rng, unit, 256, 16384), _dim(rng, unit, 256, 8192), _dim(rng, unit, 256, 8192)
        if M * N * K <= most and (kind != "host" or M * K + K * N + M * N <= 3 * 4096 ** 2):
            break
    case = _matmul("", M, K, N, realization, levels, quantizer, family, kind)
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------------ inputs
def _operands(family, M, K, N, g):
    """The families of paper_2609_26077_b200/workloads.py, made on the device."""
    def randn(*shape):
        return torch.randn(*shape, device="cuda", generator=g)

    if family == "uniform":
        return tuple(torch.rand(*s, device="cuda", generator=g).mul_(2).sub_(1) for s in ((M, K), (K, N)))
    if family == "llm":
        return randn(M, K).mul_(torch.exp(1.5 * randn(K))), randn(K, N).mul_(0.02)
    sigma = torch.ones(2, device="cuda")
    if family in ("scaled_gaussian", "student_t3"):
        sigma = 10.0 ** (6.0 * torch.rand(2, device="cuda", generator=g) - 3.0)
    out = []
    for s, shape in zip(sigma, ((M, K), (K, N))):
        x = randn(*shape)
        if family == "student_t3":
            chi2 = randn(*shape).square_()
            for _ in range(2):
                chi2.add_(randn(*shape).square_())
            x.div_(chi2.div_(3.0).sqrt_())
        out.append(x.mul_(s))
    return tuple(out)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    kind, M, N = case["kind"], case["M"], case["N"]
    if kind == "stats":
        C = torch.randn(M, N, device="cuda", generator=g)
        ref = torch.randn(M, N, device="cuda", generator=g, dtype=torch.float64).mul_(0.05).add_(C)
        return {"kind": kind, "C": C, "ref": ref, "out3": torch.empty(3, dtype=torch.float64, device="cuda")}
    K = case["K"]
    A, B = _operands(case["family"], M, K, N, g)
    if kind == "ref":
        return {"kind": kind, "A": A, "B": B, "out": torch.empty(M, N, dtype=torch.float64, device="cuda")}
    U, V, W = (None, None, None) if case["realization"] == "cubic" else realizations.get(case["realization"])
    plan = fmm.Plan(U, V, W, levels=case["levels"], block_k=case["block_k"], scale_mode=case["scale_mode"],
                    b_tile_n=case["b_tile_n"], b_preround_bf16=case["b_bf16"])
    if kind == "host":
        A, B = A.cpu().pin_memory(), B.cpu().pin_memory()
        return {"kind": kind, "plan": plan, "A": A, "B": B, "C": torch.empty(M, N, pin_memory=True),
                "ws": plan.host_workspace(M, N, K)}
    return {"kind": kind, "plan": plan, "A": A, "B": B, "C": torch.empty(M, N, device="cuda")}


# ------------------------------------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "matmul":
        return state["plan"].matmul(state["A"], state["B"], out=state["C"])
    if kind == "host":
        return state["plan"].matmul_host(state["A"], state["B"], state["C"], state["ws"])
    if kind == "ref":
        return fmm.fmm_ref_gemm_fp64(state["A"], state["B"], out=state["out"])
    return fmm.fmm_error_stats(state["C"], state["ref"], out3=state["out3"])


def work(case):
    kind, M, N = case["kind"], case["M"], case["N"]
    if kind == "stats":
        # C once (fp32), the reference once (fp64); a subtraction, two multiply-adds and a maximum per element
        return {"bytes": 12 * M * N + 24, "flops": 6 * M * N}
    K = case["K"]
    if kind == "ref":
        return {"bytes": 4 * (M * K + K * N) + 8 * M * N, "flops": 2 * M * N * K}
    # the realization replaces each 2 x 2 x 2 block product by seven
    return {"bytes": 4 * (M * K + K * N + M * N), "flops": 2 * M * N * K * (7 / 8) ** case["levels"]}


def tolerance(case):
    if case["kind"] in ("ref", "stats"):
        return {"rel": 1e-12}           # fp64 sums in another order
    return {"rel": 1e-5}                # the quantized operands are fixed to the bit; fp32 sums in another order
