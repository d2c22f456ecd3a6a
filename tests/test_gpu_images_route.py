"""Which calls put several whole small images into a tile of the strip-matrix kernel, as the library chooses: few channels and several
rounds of units go to the other kernels, except channels-last.  The result is the same, bit for bit on small integers."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, nhwc, images", [
    ((302, 32, 18, 4, 704), False, False), ((302, 32, 18, 4, 704), True, True), ((424, 32, 4, 23, 768), False, False),
    ((233, 32, 13, 3, 1024), False, False), ((60, 32, 9, 9, 272), False, True), ((302, 64, 18, 4, 704), False, False),
    ((302, 96, 18, 4, 704), False, True), ((200, 64, 9, 9, 256), False, True)], ids=str)
def test_route_and_result(dims, nhwc, images):
    ensure_built()
    n, c, h, w, k = dims
    full = (*dims, 3, 3, 1)
    rng = np.random.default_rng(n)
    few = rng.integers(-3, 4, (2, c, h, w)).astype(np.float32)
    f = rng.integers(-3, 4, (k, c, 3, 3)).astype(np.float32)
    ref = oracle.conv_direct(few, f, oracle.Shape(2, c, h, w, k, 3, 3, 1)).astype(np.float32)
    x = torch.from_numpy(few).cuda()[torch.arange(n, device="cuda") % 2].contiguous()
    room = max(b.workspace_bytes(full), b.conv_workspace_bytes(full, b.SRC_NCHW, b.MODE_BF16)) + 256
    try:
        apply_config("own choice, test build", no_gather=1)  # (which takes few images before)
        out, ws = Guarded(n * ref[0].size), Guarded(room // 4)
        (b.conv_nhwc if nhwc else b.conv)(x, b.SRC_NCHW_FUSED, torch.from_numpy(f).cuda(), full, b.MODE_BF16, out.view, ws.view)
        assert b.last_device_status() == 0 and (b.last_kernel() == b.KERNEL_STRIP) == images
        ws.check()
        got = out.check().reshape((n, h - 2, w - 2, k) if nhwc else (n, k, h - 2, w - 2))
        if nhwc:
            got = got.transpose(0, 3, 1, 2)
        assert all(np.array_equal(got[i], ref[i % 2]) for i in range(n))
    finally:
        reset_config()
