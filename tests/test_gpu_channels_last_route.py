"""Channels-last calls of the window-offset kernel's wider families, from the input with the im2win tensor beside the result, as the
library chooses: many rounds of units behind one accumulator, and many channels under one filter row, go to the other kernels."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, mode, window", [
    ((71, 17, 75, 44, 176, 1, 3, 1), b.MODE_BF16, False), ((28, 39, 97, 73, 208, 3, 3, 1), b.MODE_BF16, False),
    ((18, 416, 29, 15, 480, 1, 3, 1), b.MODE_TF32, False), ((21, 73, 26, 44, 136, 3, 5, 1), b.MODE_TF32, True),
    ((21, 189, 49, 21, 160, 1, 3, 1), b.MODE_BF16, True)], ids=str)
def test_route_and_result(dims, mode, window):
    ensure_built()
    n, c, h, w, k, fh, fw, s = dims
    rng = np.random.default_rng(n)
    few = rng.integers(-3, 4, (2, c, h, w)).astype(np.float32)
    f = rng.integers(-3, 4, (k, c, fh, fw)).astype(np.float32)
    sh = oracle.Shape(2, *dims[1:])
    ref, hat = oracle.conv_direct(few, f, sh).astype(np.float32).transpose(0, 2, 3, 1), oracle.im2win(few, sh).reshape(2, -1)
    x = torch.from_numpy(few).cuda()[torch.arange(n, device="cuda") % 2].contiguous()
    try:
        apply_config("own choice, test build", window_xhat=0)
        out, ws = Guarded(n * ref[0].size), Guarded((b.conv_workspace_bytes(dims, b.SRC_NCHW, mode) + 3) // 4)
        b.conv_nhwc(x, b.SRC_NCHW, torch.from_numpy(f).cuda(), dims, mode, out.view, ws.view)
        assert b.last_device_status() == 0 and (b.last_kernel() == b.KERNEL_WINDOW) == window
        tensor, got = ws.check()[:n * hat.shape[1]].reshape(n, -1), out.check().reshape(n, *ref.shape[1:])
        assert all(np.array_equal(got[i], ref[i % 2]) and np.array_equal(tensor[i], hat[i % 2]) for i in range(n))
    finally:
        reset_config()
