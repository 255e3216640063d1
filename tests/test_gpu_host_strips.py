"""fmm_matmul_host with operands large enough to be cut into strips: the same bits as the device call, by rows and by columns,
with strip borders that leave a remainder, in every scale mode, with and without the cluster kernel, on two streams at once."""
import numpy as np
import pytest
import torch

from paper_2609_26077_b200 import fmm, workloads as Wl
from gpu_common import coeffs, dev

pytestmark = pytest.mark.gpu

# (realization, levels, M, K, N): rows in strips while M >= N, columns otherwise
CASES = [("phi_optimal", 1, 2560, 2048, 512), ("strassen", 1, 512, 2304, 2816), ("phi_optimal", 1, 4096, 1024, 4096), ("strassen", 1, 2048, 1024, 4096),
         ("cubic", 0, 3456, 1024, 256), ("cubic", 0, 256, 1152, 3968), ("phi_optimal", 2, 1024, 4096, 1024)]


@pytest.mark.parametrize("blk,mode,tile", [(32, "fp32", 0), (32, "ue8m0", 0), (128, "fp32", 0), (128, "fp32", 128)])
@pytest.mark.parametrize("name,levels,M,K,N", CASES)
def test_strips_give_the_bits_of_the_device_call(name, levels, M, K, N, blk, mode, tile):
    U, V, W = coeffs(name)
    plan = fmm.Plan(U, V, W, levels=levels, block_k=blk, scale_mode=mode, b_tile_n=tile)
    A, B = Wl.gaussian(M, K, N, 23)
    want = plan.matmul(dev(A), dev(B)).cpu()
    Ah, Bh = torch.from_numpy(A).pin_memory(), torch.from_numpy(B).pin_memory()
    streams = [torch.cuda.Stream() for _ in range(2)]
    wss = [plan.host_workspace(M, N, K) for _ in range(2)]
    outs = [torch.full((M, N), float("nan")).pin_memory() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(3):
        for s, ws, o in zip(streams, wss, outs):
            plan.matmul_host(Ah, Bh, o, ws, stream=s)
    for s in streams:
        s.synchronize()                       # the call's side streams are joined to the caller's stream
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want)
    assert plan.device_status() == (0, 0)
    assert np.isfinite(want.numpy()).all()
