"""Channel counts that the persistent kernel's channel groups do not divide (the last group is completed with
zeros), bit for bit on small-integer data: resident and streamed filters, padded filter copies, tiles cut per image
and tiles that span many small images."""
import numpy as np
import pytest

from paper_2306_14320_b200 import binding as b
from paper_2306_14320_b200 import workloads as wl
from gpu_helpers import apply_config, ensure_built, gpu_conv, oracle_conv, reset_config
from test_gpu_nhwc import gpu_conv_nhwc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# N, C, H, W, K, Fh, Fw, stride
SHAPES = [
    (2, 40, 19, 23, 72, 3, 5, 1), (3, 17, 9, 14, 33, 5, 3, 1), (2, 1, 12, 13, 8, 1, 3, 1), (2, 61, 30, 9, 300, 3, 1, 1),
    (3, 18, 18, 30, 108, 1, 1, 1), (1, 29, 27, 36, 600, 1, 1, 1), (7, 33, 5, 6, 20, 1, 1, 1), (9, 23, 4, 9, 18, 1, 7, 1),
    (2, 21, 24, 20, 40, 2, 2, 2), (2, 13, 20, 24, 300, 4, 4, 2), (1, 401, 17, 43, 32, 3, 3, 1), (2, 37, 20, 21, 500, 3, 3, 1),
    (5, 5, 11, 12, 24, 3, 3, 2), (2, 2, 30, 31, 16, 3, 3, 1), (2, 6, 17, 16, 24, 5, 5, 1), (1, 59, 14, 14, 280, 5, 5, 1),
    (1, 12, 33, 35, 64, 7, 7, 2), (2, 2, 37, 35, 24, 7, 7, 2), (1, 3, 40, 40, 520, 7, 7, 2), (1, 7, 51, 51, 300, 11, 11, 4),
    (11, 35, 3, 4, 24, 3, 3, 1),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()


@pytest.mark.parametrize("mode", [b.MODE_TF32, b.MODE_BF16], ids=["tf32", "bf16"])
@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "x".join(map(str, d)))
def test_odd_channel_counts_bit_exact(dims, mode):
    n, c, h, w, k, fh, fw, s = dims
    x = wl.small_ints(31 + c, n * c * h * w).reshape(n, c, h, w)
    f = wl.small_ints(32 + k, k * c * fh * fw, -2, 2).reshape(k, c, fh, fw)
    ref = oracle_conv(x, f, dims)
    try:
        apply_config("auto", no_gather=1)
        for src in (b.SRC_NCHW, b.SRC_NCHW_FUSED):
            assert np.array_equal(gpu_conv(x, f, dims, mode, src_kind=src).astype(np.float64), ref), src
            assert b.last_kernel() == b.KERNEL_PERSISTENT
            nhwc = gpu_conv_nhwc(x, f, dims, mode, src)
            assert np.array_equal(np.transpose(nhwc, (0, 3, 1, 2)).astype(np.float64), ref), src
    finally:
        reset_config()


def test_fused_source_without_workspace_is_still_refused_for_odd_channels():
    dims = (2, 40, 19, 23, 72, 3, 5, 1)
    n, c, h, w, k, fh, fw, s = dims
    ho, wo = b.out_dims(dims)
    x, f = torch.zeros((n, c, h, w), device="cuda"), torch.zeros((k, c, fh, fw), device="cuda")
    out = torch.empty((n, k, ho, wo), device="cuda")
    with pytest.raises(b.Im2winError) as e:
        b.conv(x, b.SRC_NCHW_FUSED, f, dims, b.MODE_BF16, out)
    assert e.value.code == b.EUNSUPPORTED
