"""The product kernel's producer / issuer warps run with 56 or 72 registers after setmaxnreg; a few spilled values in
their loops cost a quarter of the throughput of the balanced kernels.  Compile the file with ptxas statistics and
require every instantiation to be spill-free."""
import os
import re
import shutil
import subprocess
import tempfile

import pytest

from paper_2609_26077_b200 import build as B


@pytest.mark.skipif(shutil.which(B.NVCC) is None and not os.path.exists(B.NVCC), reason="nvcc not available")
def test_product_kernel_has_no_register_spills():
    src = os.path.join(B.CSRC, "fmm_gemm.cu")
    with tempfile.TemporaryDirectory() as tmp:
        cmd = [B.NVCC] + B.FLAGS + ["-Xptxas", "-v", "-c", src, "-o", os.path.join(tmp, "g.o")]
        out = subprocess.run(cmd, capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]
    text = out.stderr + out.stdout
    entries = re.findall(r"Compiling entry function '([^']*fmm_gemm_kernel[^']*)'.*?\n.*?\n\s*(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", text)
    assert len(entries) >= 8, "ptxas statistics not found"
    bench = ("ILi128ELi3ELi32ELi2", "ILi256ELi1ELi32ELi2")
    bad = [(name[-60:], st, ld) for name, _, st, ld in entries if int(st) or int(ld)]
    assert not bad, f"register spills in {bad}"
    assert all(any(b in name for name, *_ in entries) for b in bench), "benchmark kernels not found"


def allowed(kernel):
    """Bytes of spill stores and loads that a kernel may have: none, but for the A-side encoders whose blocks per SM are worth
    more than what they spill (measured, see encode_a_kernel)."""
    m = re.search(r"encode_a_kernelILi(\d+)ELi(\d)ELj(\d+)E", kernel)
    if not m:
        return 0
    blk, mode, mask = (int(x) for x in m.groups())
    if blk == 128:
        return 48 if mask else 4           # four blocks per SM; three without a known zero pattern
    return 4 if mode == 1 and mask == 0 else 0


OTHERS = [("fmm_split.cu", 10), ("fmm_keep.cu", 4), ("fmm_encode.cu", 60), ("fmm_stats.cu", 5)]


def test_every_source_file_is_compiled():
    # fmm_api.cu has no kernels
    assert sorted(["fmm_api.cu", "fmm_gemm.cu"] + [source for source, _ in OTHERS]) == sorted(B.SOURCES)
    assert "__global__" not in open(os.path.join(B.CSRC, "fmm_api.cu")).read()


@pytest.mark.parametrize("source,kernels", OTHERS)
@pytest.mark.skipif(shutil.which(B.NVCC) is None and not os.path.exists(B.NVCC), reason="nvcc not available")
def test_other_kernels_have_no_register_spills(source, kernels):
    with tempfile.TemporaryDirectory() as tmp:
        cmd = [B.NVCC] + B.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(B.CSRC, source), "-o", os.path.join(tmp, "g.o")]
        out = subprocess.run(cmd, capture_output=True, text=True)
    assert out.returncode == 0, out.stderr[-2000:]
    entries = re.findall(r"Compiling entry function '([^']*)'.*?\n.*?\n\s*\d+ bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", out.stderr + out.stdout)
    assert len(entries) >= kernels, "ptxas statistics not found"
    bad = [(name[-60:], st, ld) for name, st, ld in entries if max(int(st), int(ld)) > allowed(name)]
    assert not bad, f"register spills in {bad}"
