"""The product kernel that keeps a parent's output blocks on chip: forced at the sizes where its indexing can go wrong (one stage, more
stages than operand slots, both halves of a scale tile, several parents, more positions than CTAs, realizations without zeros and of
eight products), against the oracle, and to the bit against the cluster kernel, which sums in the same order; and what is chosen."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import MODES, coeffs, dev

pytestmark = pytest.mark.gpu

QUANTIZERS = [(32, "fp32", 0), (32, "ue8m0", 0), (128, "fp32", 0), (128, "fp32", 128)]
KEEP = (fmm.KERNEL_BLOCKS_ON_CHIP, 1, 64, 1, 0)
SIZES = [("strassen", 1, (256, 256, 256)), ("winograd", 1, (768, 1792, 768)), ("cubic8", 1, (256, 512, 768)), ("orbit_05", 1, (768, 256, 256)),
         ("phi_optimal", 2, (512, 1024, 1536)), ("strassen", 3, (1024, 1024, 2048))]


def make(name, levels, quantizer):
    blk, mode, tile = quantizer
    return fmm.Plan(*coeffs(name), levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)


@pytest.mark.parametrize("quantizer", QUANTIZERS)
@pytest.mark.parametrize("name,levels,shape", SIZES)
def test_matches_oracle_and_cluster_kernel(name, levels, shape, quantizer):
    M, K, N = shape
    blk, mode, tile = quantizer
    A, B = Wl.gaussian(M, K, N, seed=41)
    a, b = dev(A), dev(B)
    plan = make(name, levels, quantizer)
    plan.force_product_shape(*KEEP)
    got = plan.matmul(a, b, out=torch.full((M, N), float("nan"), device="cuda"))
    assert plan.device_status() == (0, 0)
    plan.force_product_shape(fmm.KERNEL_CLUSTER, 1, 128, 1, 0)
    assert torch.equal(got, plan.matmul(a, b))
    want = O.fused_fmm(A, B, *coeffs(name), levels=levels, blk=blk, mode=MODES[mode], b_tile=tile)
    assert np.linalg.norm(got.cpu().numpy().astype(np.float64) - want) <= 1e-5 * np.linalg.norm(want)


@pytest.mark.parametrize("quantizer", QUANTIZERS)
@pytest.mark.parametrize("m,n", [(128 * 37, 128 * 3), (128 * 10, 128 * 22)])
def test_more_positions_than_ctas(m, n, quantizer):
    # 222 and 440 tile positions, one with an odd number of rows of tiles: two and three to a CTA
    plan = make("phi_optimal", 1, quantizer)
    a, b = torch.randn(2 * m, 768, device="cuda"), torch.randn(768, 2 * n, device="cuda")
    plan.force_product_shape(*KEEP)
    got = plan.matmul(a, b)
    assert plan.device_status() == (0, 0)
    plan.force_product_shape(fmm.KERNEL_CLUSTER, 1, 128, 1, 0)
    assert torch.equal(got, plan.matmul(a, b))


@pytest.mark.parametrize("quantizer", QUANTIZERS)
def test_zero_weights_leave_a_block_alone(quantizer):
    # NaN in some products reaches the blocks that they feed and no other, and not the next position of the CTA, which starts with the
    # running sums of this one in its registers
    plan = make("strassen", 1, quantizer)
    # 8 x 48 tile positions on at most 148 CTAs: a CTA has a position in the first row of tiles first and one in a later row next
    M, N = 2048, 6144
    m, n = M // 2, N // 2
    A = torch.randn(M, 256, device="cuda")
    A[:128, :128] = float("nan")                  # the first row of tiles of A11, which feeds products of C11, C12 and C22, none of C21
    B = torch.randn(256, N, device="cuda")
    plan.force_product_shape(*KEEP)
    got = plan.matmul(A, B)
    plan.force_product_shape(fmm.KERNEL_CLUSTER, 1, 128, 1, 0)
    want = plan.matmul(A, B)
    reached = torch.zeros(M, N, dtype=torch.bool, device="cuda")
    reached[:128] = True                          # C11, C12
    reached[m:m + 128, n:] = True                 # C22
    for c in (got, want):
        assert torch.equal(torch.isnan(c), reached) and torch.isfinite(c[~reached]).all()
    assert torch.equal(got[~reached], want[~reached])


def test_choice_and_refusals():
    for quantizer in QUANTIZERS:
        plan = make("phi_optimal", 1, quantizer)
        assert tuple(plan.product_shape(2048, 2048, 512)) == KEEP                 # short terms, more tiles than clusters
        assert plan.product_shape(256, 256, 256).kernel == fmm.KERNEL_CLUSTER
        assert plan.product_shape(8192, 8192, 8192).kernel == fmm.KERNEL_PERSISTENT
        for form in [(8, 2, 64, 1, 0), (8, 1, 128, 1, 0), (8, 1, 32, 1, 0), (8, 1, 64, 2, 0), (8, 1, 64, 1, 1)]:
            with pytest.raises(fmm.FmmError) as e:
                plan.force_product_shape(*form)
            assert e.value.status == 1
        with pytest.raises(fmm.FmmError):
            make("cubic", 0, quantizer).force_product_shape(*KEEP)


@pytest.mark.parametrize("quantizer", QUANTIZERS)
def test_host_strips_take_the_same_kernel(quantizer):
    # 8 MB of operand and more go up in strips: the same bits as from device operands
    plan = make("phi_optimal", 1, quantizer)
    M, K, N = 8192, 512, 1024
    a, b = torch.randn(M, K), torch.randn(K, N)
    assert tuple(plan.product_shape(M, N, K)) == KEEP
    out = torch.empty(M, N).pin_memory()
    plan.matmul_host(a.pin_memory(), b.pin_memory(), out, plan.host_workspace(M, N, K))
    torch.cuda.synchronize()
    assert torch.equal(out, plan.matmul(a.cuda(), b.cuda()).cpu())
