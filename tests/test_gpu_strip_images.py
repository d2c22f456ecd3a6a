"""The strip-matrix kernel with several whole images per tile (small images): results bit for bit on small integers (every
product and partial sum is exact), every source kind and both output orders, batches whose last tile is partly or hardly filled, images
that just fit twice and many times, several filter tiles."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

SHAPES = [  # N, C, H, W, K
    (5, 32, 9, 9, 48), (7, 64, 9, 9, 272), (3, 32, 7, 7, 16), (2, 96, 18, 4, 32), (9, 32, 10, 8, 520),
    (4, 32, 3, 3, 16), (40, 32, 5, 5, 96), (2, 32, 3, 64, 32), (131, 32, 4, 3, 240),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


@pytest.mark.parametrize("kind", ["im2win", "im2win bf16", "fused", "fused nhwc"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_result(shape, kind):
    n, c, h, w, k = shape
    dims = (n, c, h, w, k, 3, 3, 1)
    rng = np.random.default_rng(11)
    x = rng.integers(-3, 4, (n, c, h, w)).astype(np.float32)
    f = rng.integers(-3, 4, (k, c, 3, 3)).astype(np.float32)
    sh = oracle.Shape(*dims)
    ref = oracle.conv_direct(x, f, sh).astype(np.float32)
    if kind == "fused nhwc":
        ref = np.ascontiguousarray(ref.transpose(0, 2, 3, 1))
    src = torch.from_numpy(x if kind.startswith("fused") else oracle.im2win(x, sh).astype(np.float32)).cuda()
    src_kind = {"im2win": b.SRC_IM2WIN, "im2win bf16": b.SRC_IM2WIN_BF16}.get(kind, b.SRC_NCHW_FUSED)
    if kind == "im2win bf16":
        src = src.bfloat16()
    fd = torch.from_numpy(f).cuda()
    apply_config(strip_images=1, no_gather=1)
    out = Guarded(ref.size)
    ws = Guarded((b.workspace_bytes(dims) + 256 + b.conv_workspace_bytes(dims, src_kind, b.MODE_BF16)) // 4)
    (b.conv_nhwc if kind == "fused nhwc" else b.conv)(src, src_kind, fd, dims, b.MODE_BF16, out.view, ws.view)
    assert b.last_kernel() == b.KERNEL_STRIP and b.last_device_status() == 0
    ws.check()
    assert np.array_equal(out.check(), ref.ravel())
