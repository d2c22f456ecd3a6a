"""im2win_conv from the untransformed input where the window-offset kernel writes the im2win tensor itself: the tensor bit for
bit, the result bit for bit on small integers (every product and partial sum is exact), at the edges of tiles: images of less
than a tile (one contiguous copy per stage), of a tile and a bit, planes that are no whole 16-byte chunks, rows longer than a
copy box, several filter tiles (each writes the stages of its turn), CTA pairs with an odd number of tiles."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

SHAPES = [  # N, C, H, W, K, F
    (3, 32, 9, 9, 48, 3), (2, 32, 18, 8, 16, 3), (1, 64, 58, 58, 64, 3), (2, 32, 21, 57, 80, 3), (2, 32, 9, 130, 300, 3),
    (3, 64, 7, 9, 520, 3), (1, 32, 3, 3, 16, 3), (2, 32, 19, 31, 256, 5), (3, 32, 11, 13, 40, 5), (1, 32, 5, 5, 16, 5),
    (1, 96, 6, 140, 32, 3),
]
CONFIGS = {"own": {}, "one block": {"window_mh": 1, "window_pair": 2}, "pairs": {"window_pair": 1}, "copies": {"no_box": 1},
           "streamed": {"window_bres": 2, "window_two": 1}}


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


@pytest.mark.parametrize("mode", [b.MODE_TF32, b.MODE_BF16])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_tensor_and_result(shape, mode):
    n, c, h, w, k, fs = shape
    dims = (n, c, h, w, k, fs, fs, 1)
    rng = np.random.default_rng(7)
    x = rng.integers(-3, 4, (n, c, h, w)).astype(np.float32)
    f = rng.integers(-3, 4, (k, c, fs, fs)).astype(np.float32)
    sh = oracle.Shape(*dims)
    ref, hat = oracle.conv_direct(x, f, sh).astype(np.float32), oracle.im2win(x, sh).ravel()
    xd, fd = torch.from_numpy(x).cuda(), torch.from_numpy(f).cuda()
    ran = 0
    for name, knobs in CONFIGS.items():
        apply_config(window_xhat=1, **knobs)
        out, ws = Guarded(ref.size), Guarded((b.conv_workspace_bytes(dims, b.SRC_NCHW, mode) + 3) // 4)
        b.conv(xd, b.SRC_NCHW, fd, dims, mode, out.view, ws.view)
        ran += b.last_kernel() == b.KERNEL_WINDOW  # (not every variant fits every shape)
        assert b.last_device_status() == 0, name
        assert np.array_equal(ws.check()[:hat.size].view(np.uint32), hat.view(np.uint32)), name
        assert np.array_equal(out.check(), ref.ravel()), name
    assert ran >= 2


def test_product_library_takes_it_without_a_transform():
    """The library's own choice on a layer of the kind it is for, at several batch sizes: tensor and result as above."""
    apply_config("auto")
    for n in (8, 33):
        dims = (n, 64, 30, 30, 64, 3, 3, 1)
        rng = np.random.default_rng(n)
        x = rng.integers(-3, 4, dims[:4]).astype(np.float32)
        f = rng.integers(-3, 4, (64, 64, 3, 3)).astype(np.float32)
        sh = oracle.Shape(*dims)
        out, ws = Guarded(n * 64 * 28 * 28), Guarded(b.conv_workspace_bytes(dims, b.SRC_NCHW, b.MODE_TF32) // 4)
        b.conv(torch.from_numpy(x).cuda(), b.SRC_NCHW, torch.from_numpy(f).cuda(), dims, b.MODE_TF32, out.view, ws.view)
        assert b.last_device_status() == 0
        hat = oracle.im2win(x, sh).ravel()
        assert np.array_equal(ws.check()[:hat.size], hat)
        assert np.array_equal(out.check(), oracle.conv_direct(x, f, sh).astype(np.float32).ravel())


def _route():
    """(kernel, source kind of the window-offset kernel, transform kernel) of the last call; clears the last."""
    plan = (ctypes.c_int * 8)()
    b.lib().im2win_debug_last_plan(plan)
    return b.last_kernel(), plan[0] // 1000, b.last_transform()


@pytest.mark.parametrize("dims, mode", [
    ((8, 64, 30, 30, 64, 3, 3, 1), b.MODE_TF32), ((33, 64, 30, 30, 64, 3, 3, 1), b.MODE_TF32),
    # where it is preferred on the input beside a transform, from 2e9 multiplications on
    ((66, 16, 48, 48, 176, 5, 5, 1), b.MODE_TF32), ((15, 256, 51, 51, 31, 3, 3, 1), b.MODE_TF32), ((10, 96, 40, 45, 350, 3, 3, 1), b.MODE_BF16),
], ids=str)
def test_the_librarys_own_choice_needs_no_transform(dims, mode):
    n = dims[0]
    rng = np.random.default_rng(n)
    few = rng.integers(-3, 4, (2, *dims[1:4])).astype(np.float32)
    f = rng.integers(-3, 4, (dims[4], dims[1], dims[5], dims[6])).astype(np.float32)
    sh = oracle.Shape(2, *dims[1:])
    hat, ref = oracle.im2win(few, sh).reshape(2, -1).view(np.uint32), oracle.conv_direct(few, f, sh).astype(np.float32).reshape(2, -1)
    x = torch.from_numpy(few).cuda()[torch.arange(n, device="cuda") % 2].contiguous()
    for config, knobs in (("own choice, test build", {"window_xhat": 0}), ("auto", {})):
        apply_config(config, **knobs)
        out, ws = Guarded(n * ref.shape[1]), Guarded((b.conv_workspace_bytes(dims, b.SRC_NCHW, mode) + 3) // 4)
        if knobs:
            _route()
        b.conv(x, b.SRC_NCHW, torch.from_numpy(f).cuda(), dims, mode, out.view, ws.view)
        assert b.last_device_status() == 0
        assert not knobs or _route() == (b.KERNEL_WINDOW, 3, b.TRANSFORM_NONE)
        tensor, result = ws.check()[:n * hat.shape[1]].view(np.uint32).reshape(n, -1), out.check().reshape(n, -1)
        assert all(np.array_equal(tensor[i], hat[i % 2]) and np.array_equal(result[i], ref[i % 2]) for i in range(n))
