"""What the compiler reports of the kernels whose operand-building warps store columns too: the strip-matrix kernel spills nothing,
the window-offset kernel at most a few registers (those that also write the im2win tensor have 80 registers a thread, the others 96)."""
import concurrent.futures
import os
import re
import subprocess

import pytest

from paper_2306_14320_b200 import build

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def _spills(source, *defines):
    cmd = [NVCC, "-std=c++17", "-O3", *build.ARCH_FLAGS, *defines, "-Xcompiler", "-fPIC", "-Xptxas", "-v", "-I",
           os.path.join(os.path.dirname(os.path.dirname(build.CSRC)), "include"), "-I", build.CSRC, "-c",
           os.path.join(build.CSRC, source), "-o", os.devnull]
    text = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    return {name: int(stores) for name, stores in re.findall(r"entry function '(\S+)'.*?(\d+) bytes spill stores", text, re.S)}


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_spills():
    with concurrent.futures.ThreadPoolExecutor(2) as pool:
        window = pool.submit(_spills, "conv_tc_window.cu", "-DIM2WIN_PART=1")  # (5x5: the instantiations of 3x3 report the same)
        strip = pool.submit(_spills, "conv_tc_strip.cu")
        window, strip = window.result(), strip.result()
    strip = {k: v for k, v in strip.items() if "conv_tc_strip_kernel" in k}
    assert len(strip) == 20 and not any(strip.values()), strip
    seen = {}
    for name, stores in window.items():
        form = re.search(r"conv_tc_window_kernelILi5ELi5ELb([01])ELi([0-3])ELb([01])ELb([01])E", name)
        if form:
            seen[tuple(int(v) for v in form.groups())] = stores  # (BF16, source kind, pairs, channel tail)
    assert len(seen) == 18
    assert all(v <= (40 if kind == 3 else 0 if bf16 else 12) for (bf16, kind, _, _), v in seen.items()), seen
