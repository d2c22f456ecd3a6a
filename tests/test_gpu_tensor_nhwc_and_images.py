"""Channels-last results of the window-offset kernel that writes the im2win tensor beside them (channel tails, bulk copies, CTA pairs),
and infinities and NaN in one of several images that share a tile of the strip-matrix kernel.  Small integers: exact."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


def _data(dims, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(-3, 4, dims[:4]).astype(np.float32)
    f = rng.integers(-3, 4, (dims[4], dims[1], dims[5], dims[6])).astype(np.float32)
    return x, f, oracle.conv_direct(x, f, oracle.Shape(*dims)).astype(np.float32)


@pytest.mark.parametrize("mode", [b.MODE_TF32, b.MODE_BF16])
@pytest.mark.parametrize("c, k, fs, knobs", [
    (18, 33, (3, 3), {}), (40, 72, (3, 5), {}), (17, 48, (1, 1), {}), (64, 48, (3, 3), {"no_box": 1}), (32, 65, (5, 5), {"no_box": 1, "window_mh": 1}),
    (64, 128, (3, 3), {"window_pair": 1, "window_mh": 1}), (32, 96, (5, 5), {"window_pair": 1})], ids=str)
def test_channels_last_with_the_tensor(c, k, fs, knobs, mode):
    ran = 0
    for n, h, w in ((3, 14, 17), (2, 21, 20)):
        dims = (n, c, h, w, k, *fs, 1)
        x, f, ref = _data(dims, c + k)
        hat = oracle.im2win(x, oracle.Shape(*dims)).ravel()
        out, ws = Guarded(ref.size), Guarded((b.conv_workspace_bytes(dims, b.SRC_NCHW, mode) + 3) // 4)
        apply_config("tensor beside", force_window=1, window_xhat=1, **knobs)
        b.last_transform()
        b.conv_nhwc(torch.from_numpy(x).cuda(), b.SRC_NCHW, torch.from_numpy(f).cuda(), dims, mode, out.view, ws.view)
        assert b.last_device_status() == 0
        ran += b.last_kernel() == b.KERNEL_WINDOW and b.last_transform() == b.TRANSFORM_NONE  # (not every variant fits every shape)
        assert np.array_equal(out.check().reshape(n, *ref.shape[2:], k).transpose(0, 3, 1, 2), ref)
        assert np.array_equal(ws.check()[:hat.size], hat)
    assert ran >= 1


@pytest.mark.parametrize("bad", [0, 1, 4])
@pytest.mark.parametrize("kind", [b.SRC_NCHW, b.SRC_NCHW_FUSED, b.SRC_IM2WIN_BF16])
def test_one_image_of_a_tile_is_not_finite(kind, bad):
    for dims in ((5, 64, 9, 9, 32, 3, 3, 1), (5, 32, 6, 7, 48, 3, 3, 1)):
        x, f, ref = _data(dims, bad)
        rng = np.random.default_rng(bad)
        x[bad] = np.where(rng.random(x[bad].shape) < 0.5, np.inf, np.nan)
        out, ws = Guarded(ref.size), Guarded((max(b.conv_workspace_bytes(dims, q, b.MODE_BF16) for q in (kind, b.SRC_NCHW)) + 3) // 4)
        apply_config("images", strip_images=1, no_gather=1, window_xhat=2)
        src = torch.from_numpy(x).cuda()
        if kind == b.SRC_IM2WIN_BF16:
            hat = torch.empty(b.workspace_bytes_bf16(dims) // 2, dtype=torch.int16, device="cuda")
            b.transform_bf16(src, dims, hat)
            src = hat
        b.conv(src, kind, torch.from_numpy(f).cuda(), dims, b.MODE_BF16, out.view, ws.view)
        assert b.last_device_status() == 0 and b.last_kernel() == b.KERNEL_STRIP
        ws.check()
        got = out.check().reshape(ref.shape)
        good = [i for i in range(dims[0]) if i != bad]
        assert np.array_equal(got[good], ref[good]) and not np.isfinite(got[bad]).any()
