"""The fp64 reference product against the CPU one: both tile sizes of its dispatch (64 x 64 outputs from 148 such tiles on,
32 x 32 below), K of one step, of fewer steps than pipeline stages and of many, and operands that are not 16-byte aligned."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(64, 16, 64), (64, 48, 192), (192, 1040, 128), (768, 80, 832), (640, 16, 960)])
@pytest.mark.parametrize("aligned", [True, False])
def test_reference_product_matches_the_cpu_product(M, K, N, aligned):
    A, B = Wl.student_t3(M, K, N, seed=3)

    def place(x):
        buf = torch.empty(x.size + 1, device="cuda")
        t = buf[0 if aligned else 1:][:x.size].view(*x.shape)
        t.copy_(torch.from_numpy(x))
        return t

    out = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
    got = fmm.fmm_ref_gemm_fp64(place(A), place(B), out=out).cpu().numpy()
    want = O.ref_gemm(A, B)
    scale = np.abs(A.astype(np.float64)) @ np.abs(B.astype(np.float64))
    assert np.all(np.abs(got - want) <= 1e-13 * scale)


def test_both_tile_sizes_give_the_same_bits():
    # the size of the problem decides between tiles of 32 and of 64: a part of a large problem is the small problem's result
    A, B = Wl.gaussian(1024, 272, 1024, seed=4)
    whole = fmm.fmm_ref_gemm_fp64(dev(A), dev(B))
    part = fmm.fmm_ref_gemm_fp64(dev(A[128:384]), dev(B[:, 64:320]))
    assert torch.equal(whole[128:384, 64:320], part)
