"""Both sides of a small call are encoded by one launch: codes and scales bit for bit the oracle's for every quantizer and
coefficient pattern that has such a kernel, at its smallest size, at thin and wide operands, near its largest size, and with one
launch a side right above that and for what has no such kernel (coefficients without zeros, panels that do not divide)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import MODES, coeffs, dev

pytestmark = pytest.mark.gpu

# (block, scale mode, weight tile, bf16 pre-round), M x K x N near the largest size and right above it (148 SMs, one level)
FORMS = [((32, "fp32", 0, False), (512, 1024, 512), (768, 768, 768)), ((32, "ue8m0", 0, False), (1024, 1280, 1024), (1280, 1280, 1280)),
         ((128, "fp32", 0, False), (1024, 2048, 1792), (2560, 2560, 2560)), ((128, "fp32", 128, False), (512, 2048, 1792), (2560, 2560, 2560)),
         ((128, "fp32", 0, True), (512, 512, 768), (2560, 2560, 2560)), ((128, "fp32", 128, True), (768, 2304, 1280), (2560, 2560, 2560))]


def check(name, form, shape, launches, terms=None):
    blk, mode, tile, bf16 = form
    M, K, N = shape
    levels = 0 if name == "cubic" else 1
    A, B = Wl.FAMILIES["llm"](M, K, N, seed=7)
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile, b_preround_bf16=bf16)
    a, b = dev(A), dev(B)
    ws = plan.workspace(M, N, K)
    ws.fill_(0xFF)
    plan.encode_only(a, b, workspace=ws)
    torch.cuda.synchronize()
    assert plan.last_launch_count() == launches and plan.device_status() == (0, 0)
    for side, X, coef in (("A", A, U), ("B", B, V)):
        opts = dict(b_tile=tile, b_bf16=bf16) if side == "B" else {}
        codes, scales, e8 = O.encode(X, side, U, V, levels, blk=blk, mode=MODES[mode], **opts)
        want = scales if mode == "fp32" else e8
        for t in range(plan.terms) if terms is None else terms:
            q, s = plan.quantized_operand(ws, M, N, K, t, side)
            assert np.array_equal(q, codes[t]), f"codes of {side}, term {t}"
            assert np.array_equal(s.view(np.uint8), want[t].view(np.uint8)), f"scales of {side}, term {t}"
    if M * N * K <= 512 ** 3:
        got = plan.matmul(a, b, workspace=ws).cpu().numpy().astype(np.float64)
        want = O.fused_fmm(A, B, U, V, W, levels=levels, blk=blk, mode=MODES[mode], b_tile=tile, b_bf16=bf16)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    plan.close()


@pytest.mark.parametrize("form,large,above", FORMS)
@pytest.mark.parametrize("name", ["strassen", "winograd", "phi_optimal"])
def test_one_launch(name, form, large, above):
    check(name, form, (256, 256, 256), 1)
    check(name, form, (256, 768, 512), 1)
    check(name, form, large, 1, terms=(0, 6))


@pytest.mark.parametrize("form,large,above", FORMS)
def test_one_launch_of_panels(form, large, above):
    check("cubic", form, (128, 128, 512), 1)
    check("cubic", form, (384, 640, 512), 1)


@pytest.mark.parametrize("form,large,above", FORMS)
def test_one_launch_a_side(form, large, above):
    check("phi_optimal", form, above, 2, terms=(3,))
    check("orbit_05", form, (256, 256, 512), 2)
    check("cubic", form, (256, 256, 128), 2)


class KernelNodeParams(ctypes.Structure):                  # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", ctypes.c_void_p)] + [(n, ctypes.c_uint) for n in ("gx", "gy", "gz", "bx", "by", "bz", "shared")] + \
               [(n, ctypes.c_void_p) for n in ("params", "extra", "kern", "ctx")]


def captured_grid(call):
    """Grid of the only kernel that `call` launches."""
    graph, stream, driver = torch.cuda.CUDAGraph(keep_graph=True), torch.cuda.Stream(), ctypes.CDLL("libcuda.so.1")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
        call()
    node, count, p = ctypes.c_void_p(0), ctypes.c_size_t(1), KernelNodeParams()
    assert driver.cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.byref(node), ctypes.byref(count)) == 0 and count.value == 1
    assert driver.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(p)) == 0
    return p.gx, p.gy, p.gz


# sizes (148 SMs) at which a block per combination takes the launch 1.05 to 1.65 times as long as a block for all of them
@pytest.mark.parametrize("form,shape", [((32, "ue8m0", 0, False), (512, 1024, 512)), ((32, "ue8m0", 0, False), (3072, 512, 512)),
                                        ((128, "fp32", 0, False), (1024, 1024, 1024)), ((128, "fp32", 0, False), (256, 256, 4096)),
                                        ((128, "fp32", 128, False), (1024, 1024, 1024)), ((128, "fp32", 128, True), (256, 1536, 1024)),
                                        ((128, "fp32", 0, True), (1024, 1024, 1024))])
def test_no_block_per_combination_where_warps_are_many(form, shape):
    blk, mode, tile, bf16 = form
    M, K, N = shape
    plan = fmm.Plan(*coeffs("phi_optimal"), levels=1, block_k=blk, scale_mode=mode, b_tile_n=tile, b_preround_bf16=bf16)
    a, b, ws = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda"), plan.workspace(M, N, K)
    assert captured_grid(lambda: plan.encode_only(a, b, workspace=ws))[2] == 1


# sizes on both sides of that limit: the bits do not depend on it
@pytest.mark.parametrize("form,sizes", [((32, "fp32", 0, False), ((512, 256, 512), (512, 512, 512))), ((32, "ue8m0", 0, False), ((256, 256, 1536), (512, 768, 512))),
                                        ((128, "fp32", 0, False), ((512, 1536, 256), (768, 768, 768))), ((128, "fp32", 128, False), ((512, 1536, 256), (512, 512, 1280))),
                                        ((128, "fp32", 0, True), ((512, 768, 768), (1024, 512, 1280))), ((128, "fp32", 128, True), ((512, 1536, 256), (512, 512, 1280)))])
def test_codes_around_the_limit(form, sizes):
    for shape in sizes:
        check("phi_optimal", form, shape, 1, terms=(0, 3, 6))
    check("cubic", form, (512, 512, 512), 1)
    check("cubic", form, (512, 1024, 1024), 1 if form[0] == 128 or form[1] == "ue8m0" else 2)
