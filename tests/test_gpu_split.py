"""The product kernel for few output tiles (a cluster of CTAs per tile, partial products exchanged in distributed shared
memory): every mode at the sizes where its indexing can go wrong - one tile, one K stage, fewer and more K stages than
operand slots, clusters of 7 (rank 7), 8 (rank 8, or eight K shares) and 2 (a K that does not divide evenly), several
parents, and (FP32 scales) tiles of 32, 64 and 128 columns - against the oracle, and bit for bit from call to call."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import MODES, coeffs, dev

pytestmark = pytest.mark.gpu

SHAPES = [("strassen", 1, (256, 256, 256)), ("phi_optimal", 1, (256, 1792, 768)), ("winograd", 1, (768, 1024, 256)),
          ("cubic8", 1, (256, 512, 512)), ("phi_optimal", 2, (512, 1024, 1536)), ("winograd", 3, (1024, 1024, 1024)),
          ("cubic", 0, (128, 128, 128)), ("cubic", 0, (128, 1920, 256)), ("cubic", 0, (256, 4096, 128)), ("cubic", 0, (1024, 2048, 1024)),
          ("winograd", 1, (1024, 1024, 1024)), ("winograd", 1, (1280, 1280, 1280))]


@pytest.mark.parametrize("blk,mode,tile", [(32, "fp32", 0), (32, "ue8m0", 0), (128, "fp32", 0), (128, "fp32", 128)])
@pytest.mark.parametrize("name,levels,shape", SHAPES)
def test_few_tiles_match_oracle(name, levels, shape, blk, mode, tile):
    M, K, N = shape
    A, B = Wl.gaussian(M, K, N, seed=17)
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)
    a, b = dev(A), dev(B)
    want = O.fused_fmm(A, B, U, V, W, levels=levels, blk=blk, mode=MODES[mode], b_tile=tile)
    out = torch.full((M, N), float("nan"), device="cuda")
    # every tile width of the kernel this test is about, and whatever the library chooses for the size
    shares = max(s for s in (1, 2, 4, 8) if s <= K // 128) if name == "cubic" else 1
    for columns in (None, 128) if mode == "ue8m0" else (None, 128, 64, 32):
        if columns:
            plan.force_product_shape(fmm.KERNEL_CLUSTER, 1, columns, shares)
            assert plan.product_shape(M, N, K).kernel == fmm.KERNEL_CLUSTER
        out.fill_(float("nan"))
        first = plan.matmul(a, b, out=out).clone()
        out.fill_(float("nan"))
        assert torch.equal(plan.matmul(a, b, out=out), first)
        assert plan.device_status() == (0, 0)
        got = first.cpu().numpy().astype(np.float64)
        d = 1 << levels
        for i in range(d):
            for j in range(d):
                s = np.s_[i * M // d:(i + 1) * M // d, j * N // d:(j + 1) * N // d]
                assert np.linalg.norm(got[s] - want[s]) <= 2e-5 * np.linalg.norm(want[s]), f"columns {columns}, block ({i},{j})"
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want), f"columns {columns}"
