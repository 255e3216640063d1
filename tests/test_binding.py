"""The Python binding without a device: what it hands to the library stays alive for the call."""
import gc
import weakref

import torch

from paper_2609_26077_b200 import fmm


class Operand:
    """The attributes of a CUDA tensor that Plan.matmul reads."""
    dtype, is_cuda, device = torch.float32, True, torch.device("cpu")

    def __init__(self, rows, cols):
        self.shape = (rows, cols)

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return 4096

    def new_empty(self, shape):
        return Operand(*shape)


def test_workspace_outlives_the_call_when_another_thread_grows_it(monkeypatch):
    plan = fmm.Plan.__new__(fmm.Plan)
    plan._h, plan._ws, plan._need = None, None, {(128, 128, 128): 4096}
    seen = []

    class Library:
        def fmm_matmul(self, *args):
            # what a second thread does that needs a larger workspace, just before this call is enqueued
            first = weakref.ref(plan._ws[0])
            plan._own_workspace(1 << 20, torch.device("cpu"))
            gc.collect()
            seen.append(first() is not None)
            return 0

    monkeypatch.setattr(fmm, "_lib", Library())
    monkeypatch.setattr(fmm, "_stream_ptr", lambda stream: 0)
    plan.matmul(Operand(128, 128), Operand(128, 128))
    assert seen == [True]
