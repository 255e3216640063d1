"""Operands near the ends of the fp32 range: codes do not change when an operand is multiplied by a power of two, so the result
is the same to the bit, times that power - in every kernel, as long as the result itself is in range."""
import numpy as np
import pytest
import torch

from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import coeffs, dev
from test_gpu_product_shapes import SHAPES, shapes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quantizer", list(SHAPES))
@pytest.mark.parametrize("name,levels", [("cubic", 0), ("phi_optimal", 1), ("winograd", 2)])
def test_powers_of_two_pass_through(name, levels, quantizer):
    blk, mode, tile = quantizer
    M, K, N = 512, 1024, 512
    A, B = Wl.gaussian(M, K, N, seed=5)
    a, b = dev(A), dev(B)
    plan = fmm.Plan(*coeffs(name), levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)
    # elements of B up to 2^124, of its partial products with 8-bit codes up to 2^138; the clamp of the scales stays out of it
    for ea, eb in ((-30, 120), (120, -30), (-30, -30), (40, 40)):
        sa, sb = float(np.float32(2.0) ** ea), float(np.float32(2.0) ** eb)
        for form in shapes(name, quantizer):
            plan.force_product_shape(*form)
            want = plan.matmul(a, b).double() * 2.0 ** (ea + eb)
            got = plan.matmul(a * sa, b * sb)
            assert plan.device_status() == (0, 0)
            assert torch.isfinite(got).all(), f"{form} 2^{ea} 2^{eb}"
            assert torch.equal(got.double(), want), f"{form} 2^{ea} 2^{eb}"


@pytest.mark.parametrize("blk", [32, 128])
def test_small_clamp_keeps_small_products(blk):
    # a clamp below the range that the scaled-down sums leave room for: operands of 1e-17, results of 1e-33 and less
    A, B = Wl.gaussian(256, 256, 256, seed=6)
    a, b = dev(A), dev(B)
    plan = fmm.Plan(None, None, None, levels=0, block_k=blk, scale_mode="fp32", amax_floor=1e-30)
    want = plan.matmul(a, b).double() * 2.0 ** -112
    got = plan.matmul(a * 2.0 ** -56, b * 2.0 ** -56).double()
    # the sums' last places are far above the smallest subnormal number: nothing is lost but where a sum passes through zero
    assert torch.isfinite(got).all()
    assert (got - want).abs().max() <= 2.0 ** -23 * want.abs().max()


@pytest.mark.parametrize("K", [512, 1024, 3840])
def test_products_above_the_range_whose_weighted_sums_are_in_it(K):
    # U times 8 and W times 1/8: the same C from products that are 8 times larger.  Every kernel that carries sums or exchanges
    # products weights them before they leave the scaled-down range.  2, 4 and 15 K stages of a term
    U, V, W = coeffs("phi_optimal")
    U, W = np.float32(8) * np.asarray(U, np.float32), np.asarray(W, np.float32) / np.float32(8)
    M, N = 256, 512
    A, B = Wl.gaussian(M, K, N, seed=8)
    a, b = dev(A), dev(B)
    # elements of C up to 2^(e + 2) sqrt(K), products up to 2^(e + 5.5) sqrt(K)
    e = 124 - int(np.ceil(np.log2(K) / 2))
    sa, sb = 2.0 ** (e // 2), 2.0 ** (e - e // 2)
    plan = fmm.Plan(U, V, W, levels=1, block_k=32, scale_mode="fp32")
    for form in [f for f in shapes("phi_optimal", (32, "fp32", 0)) if f[4] == 0]:
        plan.force_product_shape(*form)
        want = plan.matmul(a, b).double() * 2.0 ** e
        got = plan.matmul(a * sa, b * sb)
        assert plan.device_status() == (0, 0)
        assert torch.isfinite(got).all(), f"{form}"
        assert torch.equal(got.double(), want), f"{form}"
