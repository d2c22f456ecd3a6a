"""Strides far above the filter, where one block of output rows would stage many rows that it does not read: both transforms bit for
bit against Algorithm 1, and the convolution behind them, at planes that fit a CTA's shared memory and planes that do not."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import TOL, apply_config, ensure_built, gpu_conv, gpu_transform, oracle_conv, rel_l2
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 102, 1000, 3, 100), (1, 2, 34, 1900, 3, 32), (2, 3, 300, 300, 7, 299), (1, 2, 61, 1200, 5, 56), (1, 2, 40, 1601, 1, 39)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_transforms_and_convolution(shape):
    ensure_built()
    apply_config("auto")
    n, c, h, w, fh, s = shape
    dims = (n, c, h, w, 4, fh, fh, s)
    rng = np.random.default_rng(h)
    x = rng.standard_normal((n, c, h, w)).astype(np.float32)
    f = rng.standard_normal((4, c, fh, fh)).astype(np.float32)
    ref = oracle.im2win(x, oracle.Shape(*dims)).astype(np.float32).ravel()
    assert np.array_equal(gpu_transform(x, dims).view(np.uint32), ref.view(np.uint32))
    out = torch.empty(ref.size, dtype=torch.int16, device="cuda")
    b.transform_bf16(torch.from_numpy(x).cuda(), dims, out)
    assert b.last_device_status() == 0
    assert torch.equal(out.cpu(), torch.from_numpy(ref).bfloat16().view(torch.int16))
    for mode in (b.MODE_TF32, b.MODE_BF16, b.MODE_FP32):
        assert rel_l2(gpu_conv(x, f, dims, mode), oracle_conv(x, f, dims)) <= TOL[mode]
