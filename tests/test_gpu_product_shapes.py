"""Every tile shape of the product kernels, forced, at the sizes where its indexing can go wrong: one tile, leaves that are not
a multiple of the tile (half of a CTA pair's rows, half of a wide tile's columns hang over the edge), one K stage, more stages
than operand slots, several parents - against the oracle; what a plan cannot take is refused."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import MODES, coeffs, dev

pytestmark = pytest.mark.gpu

P, CL = fmm.KERNEL_PERSISTENT, fmm.KERNEL_CLUSTER
# (kernel, CTAs per tile, columns, K shares, output warp) by quantizer
SHAPES = {
    (32, "fp32", 0): [(P, 2, 128, 1, 0), (P, 1, 128, 1, 0), (P, 2, 128, 1, 1), (P, 1, 128, 1, 1), (CL, 1, 128, 1, 0), (CL, 1, 64, 1, 0), (CL, 1, 32, 1, 0)],
    (32, "ue8m0", 0): [(P, 2, 256, 1, 0), (P, 1, 256, 1, 0), (P, 1, 128, 1, 0), (CL, 1, 128, 1, 0)],
    (128, "fp32", 0): [(P, 2, 256, 1, 0), (P, 1, 128, 1, 0), (CL, 1, 128, 1, 0), (CL, 1, 64, 1, 0), (CL, 1, 32, 1, 0)],
    (128, "fp32", 128): [(P, 2, 256, 1, 0), (P, 1, 128, 1, 0), (CL, 1, 128, 1, 0), (CL, 1, 64, 1, 0), (CL, 1, 32, 1, 0)],
}
# for plans with products to combine, every quantizer
KEEP = (fmm.KERNEL_BLOCKS_ON_CHIP, 1, 64, 1, 0)
SIZES = [("strassen", 1, (256, 256, 256)), ("winograd", 1, (768, 1536, 768)), ("cubic8", 1, (256, 512, 768)),
         ("orbit_05", 1, (768, 256, 256)), ("phi_optimal", 2, (512, 1024, 1536)), ("strassen", 3, (1024, 1024, 1024)),
         ("cubic", 0, (384, 1024, 128)), ("cubic", 0, (128, 128, 384))]


def shapes(name, quantizer):
    return SHAPES[quantizer] + ([] if name == "cubic" else [KEEP])


def make(name, levels, quantizer):
    blk, mode, tile = quantizer
    return fmm.Plan(*coeffs(name), levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)


@pytest.mark.parametrize("quantizer", list(SHAPES))
@pytest.mark.parametrize("name,levels,shape", SIZES)
def test_every_shape_matches_oracle(name, levels, shape, quantizer):
    M, K, N = shape
    blk, mode, tile = quantizer
    A, B = Wl.gaussian(M, K, N, seed=31)
    a, b = dev(A), dev(B)
    want = O.fused_fmm(A, B, *coeffs(name), levels=levels, blk=blk, mode=MODES[mode], b_tile=tile)
    plan = make(name, levels, quantizer)
    forms = shapes(name, quantizer)
    if name == "cubic":
        forms += [(CL, 1, c, s, 0) for _, _, c, _, _ in forms[-1:] for s in (2, 4, 8) if s <= K // 128]
    d = 1 << levels
    for form in forms:
        plan.force_product_shape(*form)
        assert tuple(plan.product_shape(M, N, K)) == form
        out = torch.full((M, N), float("nan"), device="cuda")
        got = plan.matmul(a, b, out=out).cpu().numpy().astype(np.float64)
        assert plan.device_status() == (0, 0)
        for i in range(d):
            for j in range(d):
                s = np.s_[i * M // d:(i + 1) * M // d, j * N // d:(j + 1) * N // d]
                assert np.linalg.norm(got[s] - want[s]) <= 2e-5 * np.linalg.norm(want[s]), f"{form}, block ({i},{j})"
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), f"{form}"


@pytest.mark.parametrize("quantizer", list(SHAPES))
def test_shapes_that_do_not_exist_are_refused(quantizer):
    for levels, name in ((0, "cubic"), (1, "strassen")):
        known = set(shapes(name, quantizer))
        if quantizer[1] == "ue8m0" and levels:
            known.add((fmm.KERNEL_CLUSTER_TWO_TERMS, 1, 128, 1, 0))
        plan = make(name, levels, quantizer)
        chosen = tuple(plan.product_shape(256, 256, 256))
        for form in [(k, c, n, s, w) for k in (1, 2, 3, 4, 5, 8, 16) for c in (1, 2) for n in (32, 64, 128, 256) for s in (1, 2, 3) for w in (0, 1)]:
            base = (*form[:3], 1, form[4])
            if base in known and (form[3] == 1 or (form[3] == 2 and form[0] == CL and levels == 0)):
                plan.force_product_shape(*form)
                plan.force_product_shape()
            else:
                with pytest.raises(fmm.FmmError) as e:
                    plan.force_product_shape(*form)
                assert e.value.status == 1
        # a refused shape and the release of a forced one leave the library's choice
        assert tuple(plan.product_shape(256, 256, 256)) == chosen


def test_more_k_shares_than_chunks_is_a_shape_error():
    plan = make("cubic", 0, (32, "fp32", 0))
    plan.force_product_shape(CL, 1, 128, 4, 0)
    a = torch.randn(128, 256, device="cuda")
    with pytest.raises(fmm.FmmError) as e:
        plan.matmul(a, a.t().contiguous())
    assert e.value.status == 2
    plan.force_product_shape()
    plan.matmul(a, a.t().contiguous())
    assert plan.device_status() == (0, 0)


@pytest.mark.parametrize("K", [768, 1024])
@pytest.mark.parametrize("name", ["strassen", "phi_optimal"])
def test_block_32_around_the_output_warps_boundary(name, K):
    # terms of three and four K stages, more tiles than CTAs (182) and pairs (91 of an odd number of rows of tiles): sums carried,
    # written by the promoting warps and by the output warps, and separate ones
    M, N = 3328, 3584
    A, B = Wl.gaussian(M, K, N, seed=32)
    a, b = dev(A), dev(B)
    plan = make(name, 1, (32, "fp32", 0))
    want = O.fused_fmm(A, B, *coeffs(name), levels=1, blk=32, mode=O.SCALE_FP32)
    carried = []
    for form in SHAPES[(32, "fp32", 0)][:4]:
        plan.force_product_shape(*form)
        c = plan.matmul(a, b, out=torch.full((M, N), float("nan"), device="cuda"))
        assert plan.device_status() == (0, 0)
        assert np.linalg.norm(c.cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want), f"{form}"
        if form[4] == 0:
            carried.append(c)
    assert torch.equal(*carried)
