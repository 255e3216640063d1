"""Leaves that are not a multiple of the product kernel's tile: an odd number of 128-row blocks (half of a CTA pair's last
tiles hangs over the edge), of 128-column blocks (half of a 256-column tile), both, one level and two (the next term's rows
lie behind the edge), large enough for the persistent kernel - against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import MODES, coeffs, dev

pytestmark = pytest.mark.gpu

SHAPES = [("cubic", 0, (3200, 256, 3072)), ("cubic", 0, (3072, 256, 3200)), ("cubic", 0, (4224, 128, 4224)),
          ("strassen", 1, (4352, 512, 4352)), ("winograd", 2, (3584, 512, 5632))]


@pytest.mark.parametrize("blk,mode,tile", [(32, "fp32", 0), (32, "ue8m0", 0), (128, "fp32", 0), (128, "fp32", 128)])
@pytest.mark.parametrize("name,levels,shape", SHAPES)
def test_odd_leaves_match_oracle(name, levels, shape, blk, mode, tile):
    M, K, N = shape
    A, B = Wl.gaussian(M, K, N, seed=23)
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)
    want = O.fused_fmm(A, B, U, V, W, levels=levels, blk=blk, mode=MODES[mode], b_tile=tile)
    a, b = dev(A), dev(B)
    out = torch.full((M, N), float("nan"), device="cuda")
    d = 1 << levels
    m, n = M // d, N // d
    # the library's choice, and the shapes whose tiles hang over these leaves: CTA pairs, 256-column tiles
    forms = [None, (2, 128 if blk == 32 and mode == "fp32" else 256)] + ([(1, 256)] if mode == "ue8m0" else [])
    for form in forms:
        if form:
            if not (m % (128 * form[0]) or n % form[1]):
                continue                                  # the tiles of this shape end with this leaf
            plan.force_product_shape(fmm.KERNEL_PERSISTENT, *form)
        out.fill_(float("nan"))
        plan.matmul(a, b, out=out)
        assert plan.device_status() == (0, 0)
        got = out.cpu().numpy().astype(np.float64)
        for i in range(d):
            for j in range(d):
                for r, c in ((slice(0, m), slice(0, n)), (slice(m - 128, m), slice(0, n)), (slice(0, m), slice(n - 128, n))):
                    g, w = got[i * m:(i + 1) * m, j * n:(j + 1) * n][r, c], want[i * m:(i + 1) * m, j * n:(j + 1) * n][r, c]
                    assert np.linalg.norm(g - w) <= 2e-5 * np.linalg.norm(w), f"{form}, block ({i},{j}), rows {r}, columns {c}"
