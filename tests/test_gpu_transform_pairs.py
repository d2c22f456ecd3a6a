"""The bf16 transform by pairs of columns: bit for bit against Algorithm 1 rounded to bf16, at rows of odd and even length, strips
that start at odd elements, one column, blocks of rows and several planes per job with every 16-byte phase of the output."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import ensure_built
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

SHAPES = [(3, 5, 15, 15), (2, 3, 31, 31), (5, 7, 12, 14), (1, 2, 40, 227), (2, 3, 60, 61), (9, 11, 13, 11), (1, 1, 11, 11), (1, 3, 90, 130)]


@pytest.mark.parametrize("fh", [3, 5, 7, 11])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_bits(shape, fh):
    ensure_built()
    n, c, h, w = shape
    rng = np.random.default_rng(h * w)
    x = rng.standard_normal((n, c, h, w)).astype(np.float32)
    for s in (1, 2):
        dims = (n, c, h, w, 1, fh, 1, s)
        ref = torch.from_numpy(oracle.im2win(x, oracle.Shape(*dims)).astype(np.float32)).bfloat16().view(torch.int16).flatten()
        full = torch.full((ref.numel() + 64,), 21555, dtype=torch.int16, device="cuda")
        out = full[32:-32]
        b.transform_bf16(torch.from_numpy(x).cuda(), dims, out)
        assert b.last_device_status() == 0
        assert torch.equal(out.cpu(), ref)
        assert bool((full[:32] == 21555).all()) and bool((full[-32:] == 21555).all())
