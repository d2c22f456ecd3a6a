"""What the compiler reports of the tile transform's instantiations: none spills registers, and only filter heights that
the column form serves (odd, above 1; in bf16 storage 7 and 11, behind the pairs kernel, whose registers are looked at too) have it -- beside the quads in one kernel for three rows and for eleven in fp32, else alone -- and the quads' kernels do not."""
import os
import re
import subprocess

import pytest

from paper_2306_14320_b200 import build

NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_tile_transform_instantiations_do_not_spill(tmp_path):
    cmd = [NVCC, "-std=c++17", "-O3", *build.ARCH_FLAGS, "-Xcompiler", "-fPIC", "-Xptxas", "-v", "-I",
           os.path.join(os.path.dirname(os.path.dirname(build.CSRC)), "include"), "-I", build.CSRC, "-c",
           os.path.join(build.CSRC, "transform.cu"), "-o", str(tmp_path / "t.o")]
    text = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    seen = {}
    for name, body in re.findall(r"entry function '(\S+)'(.*?Used \d+ registers)", text, re.S):
        form = re.search(r"transform_tile_kernelILi(\d+)ELb([01])ELi([012])E", name)
        if form:
            spill = int(re.search(r"(\d+) bytes spill stores", body).group(1))
            seen[tuple(int(v) for v in form.groups())] = (spill, int(re.search(r"Used (\d+) registers", body).group(1)))
    columns = {(3, 0): 2, (5, 0): 1, (7, 0): 1, (7, 1): 1, (11, 0): 2, (11, 1): 1}
    assert sorted(k for k in seen if not k[2]) == sorted([(fh, 0, 0) for fh in (1, 2, 3, 4, 5, 7, 11)] + [(fh, 1, 0) for fh in (1, 2, 4)])
    assert {k[:2]: k[2] for k in seen if k[2]} == columns
    assert all(spill == 0 for spill, _ in seen.values()), seen
    pairs = [tuple(map(int, v)) for v in re.findall(r"transform_pairs_kernelILi(?:3|5|7|11)E.*?(\d+) bytes spill stores.*?Used (\d+) registers", text, re.S)]
    assert len(pairs) == 4 and all(spill == 0 and regs <= 40 for spill, regs in pairs), pairs
    # six CTAs of 256 threads per SM (34 KB of shared memory each): at most 40 registers a thread
    assert all(regs <= 40 for (fh, o, form), (_, regs) in seen.items() if fh <= 5 or (fh, o) == (7, 1)), seen
