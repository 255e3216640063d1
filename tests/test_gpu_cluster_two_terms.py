"""The cluster kernel with two terms per CTA (UE8M0 scales): forced at one tile, odd and even ranks, one K stage and more than
operand slots, several parents and strips of tiles - the same bits as the cluster kernel with one term per CTA, and the
oracle's result; chosen by the library where its clusters hold all tiles and those of the other do not; refused elsewhere."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import coeffs, dev, make_plan

pytestmark = pytest.mark.gpu

TWO = fmm.KERNEL_CLUSTER_TWO_TERMS
SIZES = [("strassen", 1, (256, 256, 256)), ("cubic8", 1, (256, 512, 768)), ("winograd", 1, (768, 1536, 768)), ("orbit_05", 1, (768, 256, 256)),
         ("phi_optimal", 2, (512, 1024, 1536)), ("strassen", 3, (1024, 1024, 1024)), ("phi_optimal", 1, (2304, 1024, 2560))]


@pytest.mark.parametrize("name,levels,shape", SIZES)
def test_matches_one_term_per_cta_and_the_oracle(name, levels, shape):
    M, K, N = shape
    A, B = Wl.gaussian(M, K, N, seed=13)
    a, b = dev(A), dev(B)
    plan = make_plan(name, levels, 32, "ue8m0")
    out = []
    for kernel in (fmm.KERNEL_CLUSTER, TWO):
        plan.force_product_shape(kernel, 1, 128)
        assert plan.product_shape(M, N, K).kernel == kernel
        for _ in range(2):
            c = torch.full((M, N), float("nan"), device="cuda")
            plan.matmul(a, b, out=c)
            out.append(c)
        assert plan.device_status() == (0, 0)
    assert all(torch.equal(out[0], c) for c in out[1:])
    want = O.fused_fmm(A, B, *coeffs(name), levels=levels, blk=32, mode=O.SCALE_UE8M0)
    assert np.linalg.norm(out[2].cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)


def test_choice():
    plan = make_plan("phi_optimal", 1, 32, "ue8m0")
    # 55 and 56 tiles: between what one wave of clusters of seven and of four holds, with room on both sides
    assert plan.product_shape(1792, 2048, 2048).kernel == TWO
    assert plan.product_shape(1280, 2816, 3328).kernel == TWO
    assert plan.product_shape(1024, 1024, 1024).kernel == fmm.KERNEL_CLUSTER
    assert plan.product_shape(4096, 4096, 4096).kernel == fmm.KERNEL_PERSISTENT


def test_refused_without_terms_and_for_other_quantizers():
    for plan in (make_plan("cubic", 0, 32, "ue8m0"), make_plan("strassen", 1, 32, "fp32"), make_plan("strassen", 1, 128, "fp32")):
        with pytest.raises(fmm.FmmError) as e:
            plan.force_product_shape(TWO, 1, 128)
        assert e.value.status == 1
