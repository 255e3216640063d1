"""Rounding error of the fp32-scale products against the exact product of the quantized operands, per kernel: the sums that the
walk carries from one product to the next may cost no more than stated, compared with every product summed on its own in fp32
(one rounding per K block, as the paper's fp32 accumulation has it)."""
import numpy as np
import pytest
import torch

from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import coeffs, dev

pytestmark = pytest.mark.gpu


def dequantized(plan, ws, M, N, K, term):
    """The term's operands in fp64, (m, K blocks, blk) and (n, K blocks, blk): codes only, and the scales."""
    table = torch.from_numpy(np.arange(256, dtype=np.uint8)).view(torch.float8_e4m3fn).to(torch.float64).cuda()
    out = []
    for side in "AB":
        codes, scales = plan.quantized_operand(ws, M, N, K, term, side)
        if side == "B":
            codes, scales = codes.T, scales.T
        codes = table[torch.from_numpy(np.ascontiguousarray(codes)).cuda().long()]
        out.append((codes.reshape(codes.shape[0], -1, plan.block_k), torch.from_numpy(np.ascontiguousarray(scales)).cuda().double()))
    return out


@pytest.mark.parametrize("name", ["strassen", "winograd", "phi_optimal", "orbit_05", "orbit_10", "orbit_12"])
@pytest.mark.parametrize("blk,tile,form,bound", [
    # every product is summed on its own; what is left is the order of the seven sums
    (32, 0, (fmm.KERNEL_PERSISTENT, 2, 128, 1, 1), 1.03), (32, 0, (fmm.KERNEL_PERSISTENT, 1, 128, 1, 1), 1.03),
    (32, 0, (fmm.KERNEL_CLUSTER, 1, 64, 1, 0), 1.03), (32, 0, (fmm.KERNEL_BLOCKS_ON_CHIP, 1, 64, 1, 0), 1.03),
    (128, 0, (fmm.KERNEL_BLOCKS_ON_CHIP, 1, 64, 1, 0), 1.03), (128, 128, (fmm.KERNEL_BLOCKS_ON_CHIP, 1, 64, 1, 0), 1.03),
    # the accumulators start from the carried sum: 1.57 times for independent products (see the walk's own test)
    (32, 0, (fmm.KERNEL_PERSISTENT, 2, 128, 1, 0), 1.6), (128, 0, (fmm.KERNEL_PERSISTENT, 2, 256, 1, 0), 1.6),
    (128, 128, (fmm.KERNEL_PERSISTENT, 2, 256, 1, 0), 1.6)])
def test_rounding_error_against_separate_sums(name, blk, tile, form, bound):
    M, K, N = 512, 4096, 512
    A, B = Wl.gaussian(M, K, N, seed=3)
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=1, block_k=blk, scale_mode="fp32", b_tile_n=tile)
    plan.force_product_shape(*form)
    ws = plan.workspace(M, N, K)
    got = plan.matmul(dev(A), dev(B), workspace=ws).double()
    assert plan.device_status() == (0, 0)
    m, n = M // 2, N // 2
    exact = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    separate = torch.zeros(M, N, device="cuda")
    for r in range(len(W)):
        (qa, sa), (qb, sb) = dequantized(plan, ws, M, N, K, r)
        whole, acc = torch.zeros(m, n, dtype=torch.float64, device="cuda"), torch.zeros(m, n, device="cuda")
        for kb in range(qa.shape[1]):
            part = torch.zeros(m, n, device="cuda")
            for j in range(0, blk, 32):                   # an instruction of the tensor core multiplies 32 k
                part = (part.double() + qa[:, kb, j:j + 32] @ qb[:, kb, j:j + 32].T).float()
            whole += (qa[:, kb] @ qb[:, kb].T) * (sa[:, kb, None] * sb[None, :, kb])
            acc = (acc.double() + (part * sb[None, :, kb].float()).double() * sa[:, kb, None]).float()
        for q in range(4):
            if W[r][q] != 0:
                s = np.s_[(q >> 1) * m:(q >> 1) * m + m, (q & 1) * n:(q & 1) * n + n]
                exact[s] += float(W[r][q]) * whole
                separate[s] += float(W[r][q]) * acc
    ours, theirs = (got - exact).norm().item(), (separate.double() - exact).norm().item()
    print(f"{name} {blk} {tile} {form}: {ours / exact.norm().item():.3e} against {theirs / exact.norm().item():.3e}: {ours / theirs:.3f}")
    assert ours <= bound * theirs
