"""A call is ordinary work towards what is before it on the stream, while its own kernels overlap: operands written just before
the call, a workspace and a result shared by consecutive calls, and calls captured behind every kind of graph node have to give
the bits of a call on an idle device, and no call depends on the caller's last kernel alone."""
import ctypes

import pytest
import torch

from paper_2609_26077_b200 import fmm
from gpu_common import coeffs

pytestmark = pytest.mark.gpu

CASES = [("cubic", 0, 32, "fp32", 0, 256), ("strassen", 1, 32, "fp32", 0, 512), ("phi_optimal", 1, 128, "fp32", 128, 2048),
         ("winograd", 2, 32, "ue8m0", 0, 1024), ("phi_optimal", 2, 128, "fp32", 0, 1024), ("strassen", 3, 32, "fp32", 0, 1024),
         ("strassen", 1, 32, "fp32", 0, 1280), ("winograd", 1, 128, "fp32", 0, 2560)]          # a launch for each side


def setup(name, levels, blk, mode, tile, n):
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)
    g = torch.Generator(device="cuda").manual_seed(n + levels)
    srcs = [[torch.randn(n, n, device="cuda", generator=g) for _ in range(2)] for _ in range(2)]
    ws = plan.workspace(n, n, n)
    wants = []
    for a, b in srcs:
        torch.cuda.synchronize()
        wants.append(plan.matmul(a, b, workspace=ws).clone())
        torch.cuda.synchronize()
    return plan, ws, srcs, wants


@pytest.mark.parametrize("case", CASES)
def test_operands_written_just_before_the_call(case):
    plan, ws, srcs, wants = setup(*case)
    n = case[-1]
    a, b = torch.empty(n, n, device="cuda"), torch.empty(n, n, device="cuda")
    out, ref = torch.empty(n, n, device="cuda"), torch.empty(n, n, dtype=torch.float64, device="cuda")
    got = []
    for i in range(8):
        x, y = srcs[i % 2]
        if i % 4 < 2:
            torch.mul(x, 1.0, out=a)
            b.copy_(y)                            # a copy, the last thing before the call
        else:
            a.copy_(x)
            torch.mul(y, 1.0, out=b)              # a kernel, which wrote the side whose encoder does not wait
        plan.matmul(a, b, out=out, workspace=ws)
        fmm.fmm_ref_gemm_fp64(a, b, out=ref)
        stats = fmm.fmm_error_stats(out, ref, out3=torch.empty(3, dtype=torch.float64, device="cuda"))
        got.append((out.clone(), ref.clone(), stats.clone()))
    torch.cuda.synchronize()
    assert plan.device_status() == (0, 0)
    for i, (c, r, s) in enumerate(got):
        x, y = srcs[i % 2]
        assert torch.equal(c, wants[i % 2])
        assert torch.equal(r, fmm.fmm_ref_gemm_fp64(x, y))
        torch.cuda.synchronize()
        assert torch.equal(s, fmm.fmm_error_stats(c, r, out3=torch.empty(3, dtype=torch.float64, device="cuda")))


@pytest.mark.parametrize("before", ["nothing", "kernel", "kernel_b", "memset", "copy", "event", "call"])
@pytest.mark.parametrize("case", CASES[1::2])
def test_captured_behind_every_kind_of_node(case, before):
    plan, ws, srcs, wants = setup(*case)
    n = case[-1]
    a, b = (t.clone() for t in srcs[0])
    out, stats = torch.empty(n, n, device="cuda"), torch.empty(3, dtype=torch.float64, device="cuda")
    ref = torch.empty(n, n, dtype=torch.float64, device="cuda")
    spare = torch.empty(n, n, device="cuda")
    stream, side = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        with torch.cuda.graph(graph, stream=stream):
            if before == "kernel":
                torch.mul(srcs[0][0], 1.0, out=a)
            elif before == "kernel_b":
                torch.mul(srcs[0][1], 1.0, out=b)
            elif before == "memset":
                spare.zero_()
            elif before == "copy":
                a.copy_(srcs[0][0])
            elif before == "event":
                side.wait_stream(stream)
                with torch.cuda.stream(side):
                    a.copy_(srcs[0][0])
                spare.add_(1.0)
                stream.wait_stream(side)
            elif before == "call":
                plan.matmul(srcs[1][0], srcs[1][1], out=spare, workspace=ws)
            plan.matmul(a, b, out=out, workspace=ws)
            fmm.fmm_ref_gemm_fp64(a, b, out=ref)
            fmm.fmm_error_stats(out, ref, out3=stats)
    for _ in range(3):
        if before in ("kernel", "copy", "event"):
            a.fill_(float("nan"))
        elif before == "kernel_b":
            b.fill_(float("nan"))
        out.fill_(float("nan"))
        graph.replay()
    torch.cuda.synchronize()
    assert plan.device_status() == (0, 0)
    assert torch.equal(out, wants[0]) and torch.equal(ref, fmm.fmm_ref_gemm_fp64(*srcs[0]))
    assert torch.equal(stats, fmm.fmm_error_stats(out, ref, out3=torch.empty(3, dtype=torch.float64, device="cuda")))
    if before == "call":
        assert torch.equal(spare, wants[1])


def edges(graph):
    """(from, to, type) of every edge of a captured graph; type 1 is a programmatic one."""
    driver = ctypes.CDLL("libcuda.so.1")
    count = ctypes.c_size_t(0)
    handle = ctypes.c_void_p(graph.raw_cuda_graph())
    assert driver.cuGraphGetEdges_v2(handle, None, None, None, ctypes.byref(count)) == 0
    src, dst = (ctypes.c_void_p * count.value)(), (ctypes.c_void_p * count.value)()
    data = (ctypes.c_uint8 * (8 * count.value))()          # CUgraphEdgeData: from_port, to_port, type, reserved[5]
    assert driver.cuGraphGetEdges_v2(handle, src, dst, data, ctypes.byref(count)) == 0
    return [(src[i], dst[i], data[8 * i + 2]) for i in range(count.value)]


def captured_behind_a_kernel(call):
    spare, stream = torch.zeros(64, device="cuda"), torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
        spare.add_(1.0)
        call()
    return edges(graph)


@pytest.mark.parametrize("case", CASES)
def test_first_kernel_waits_for_everything_before_it(case):
    # a programmatic dependency on the caller's last kernel would stand for that kernel alone: it may itself have been launched
    # under the tail of one that it does not wait for
    plan, ws, srcs, wants = setup(*case)
    n = case[-1]
    a, b = srcs[0]
    out, ref, out3 = torch.empty(n, n, device="cuda"), torch.empty(n, n, dtype=torch.float64, device="cuda"), torch.empty(3, dtype=torch.float64, device="cuda")
    fmm.fmm_error_stats_noalloc(out, ref, out3)
    calls = {"matmul": lambda: plan.matmul(a, b, out=out, workspace=ws), "encode": lambda: plan.encode_only(a, b, workspace=ws),
             "multiply": lambda: plan.multiply_only(n, n, n, out, workspace=ws), "ref": lambda: fmm.fmm_ref_gemm_fp64(a, b, out=ref),
             "stats": lambda: fmm.fmm_error_stats(out, ref, out3=out3), "stats_noalloc": lambda: fmm.fmm_error_stats_noalloc(out, ref, out3)}
    for name, call in calls.items():
        found = captured_behind_a_kernel(call)
        roots = {f for f, _, _ in found} - {t for _, t, _ in found}
        assert len(roots) == 1, name
        assert [kind for f, _, kind in found if f in roots] == [0], name
