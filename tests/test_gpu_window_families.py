"""The window-offset kernel on rectangular filters and on channel counts that are no whole filter blocks, from the input: results
(and the im2win tensor, where the call leaves it) bit for bit on small integers; channels beyond the last must not be read as
data (infinities and NaN in the next image beside them)."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

FILTERS = [(1, 1), (1, 3), (3, 1), (1, 7), (7, 1), (3, 5), (5, 3), (3, 4), (3, 3), (5, 5)]
SHAPES = [(2, 17, 20, 21, 48), (3, 40, 13, 18, 72), (2, 33, 9, 100, 100), (3, 36, 9, 8, 260)]  # N, C, H, W, K


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


def _call(x, f, dims, mode, kind, nhwc=False):
    ho, wo = b.out_dims(dims)
    out = Guarded(dims[0] * dims[4] * ho * wo)
    room = max(b.workspace_bytes(dims), b.conv_workspace_bytes(dims, b.SRC_NCHW, mode), b.conv_workspace_bytes(dims, kind, mode))
    ws = Guarded((room + 3) // 4)
    (b.conv_nhwc if nhwc else b.conv)(torch.from_numpy(x).cuda(), kind, torch.from_numpy(f).cuda(), dims, mode, out.view, ws.view)
    assert b.last_kernel() == b.KERNEL_WINDOW and b.last_device_status() == 0
    got = out.check()
    return (got.reshape(dims[0], ho, wo, dims[4]).transpose(0, 3, 1, 2) if nhwc else got.reshape(dims[0], dims[4], ho, wo)), ws.check()


@pytest.mark.parametrize("fs", FILTERS, ids=lambda f: "%dx%d" % f)
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_result_and_tensor(shape, fs):
    n, c, h, w, k = shape
    dims = (n, c, h, w, k, *fs, 1)
    rng = np.random.default_rng(c * k)
    x = rng.integers(-3, 4, (n, c, h, w)).astype(np.float32)
    f = rng.integers(-3, 4, (k, c, *fs)).astype(np.float32)
    sh = oracle.Shape(*dims)
    ref, hat = oracle.conv_direct(x, f, sh).astype(np.float32), oracle.im2win(x, sh).ravel()
    for mode in (b.MODE_TF32, b.MODE_BF16):
        for knobs in ({}, {"no_box": 1, "window_mh": 1}):
            apply_config(force_window=1, window_xhat=1, **knobs)
            got, ws = _call(x, f, dims, mode, b.SRC_NCHW)
            assert np.array_equal(got, ref) and np.array_equal(ws[:hat.size], hat)
            assert np.array_equal(_call(x, f, dims, mode, b.SRC_NCHW_FUSED, nhwc=bool(knobs))[0], ref)


@pytest.mark.parametrize("fs", [(3, 3), (1, 1), (3, 4)], ids=lambda f: "%dx%d" % f)
def test_channels_beyond_the_last_are_not_data(fs):
    dims = (2, 18, 16, 16, 32, *fs, 1)
    rng = np.random.default_rng(3)
    x = rng.integers(-3, 4, dims[:4]).astype(np.float32)
    f = rng.integers(-3, 4, (32, 18, *fs)).astype(np.float32)
    ref = oracle.conv_direct(x, f, oracle.Shape(*dims)).astype(np.float32)
    x[1] = np.where(rng.random(x[1].shape) < 0.5, np.inf, np.nan)  # (the next image, behind the first one's last channel)
    for mode in (b.MODE_TF32, b.MODE_BF16):
        apply_config(force_window=1, window_xhat=1)
        for kind in (b.SRC_NCHW, b.SRC_NCHW_FUSED):
            got, _ = _call(x, f, dims, mode, kind)
            assert np.array_equal(got[0], ref[0]) and not np.isfinite(got[1]).any()


def test_refused_without_room_for_the_tensor_as_before():
    """A fused call whose channel count or filter no fused kernel of the published list takes wants room for the im2win tensor."""
    apply_config("auto")
    for dims in ((8, 40, 40, 40, 64, 3, 5, 1), (8, 64, 40, 40, 64, 3, 4, 1)):
        n, c, h, w, k, fh, fw, s = dims
        ho, wo = b.out_dims(dims)
        x, f = torch.zeros((n, c, h, w), device="cuda"), torch.zeros((k, c, fh, fw), device="cuda")
        out = torch.empty((n, k, ho, wo), device="cuda")
        ws = torch.empty(b.workspace_bytes(dims) - 4, dtype=torch.uint8, device="cuda")
        with pytest.raises(b.Im2winError) as e:
            b.conv(x, b.SRC_NCHW_FUSED, f, dims, b.MODE_BF16, out, ws)
        assert e.value.code == b.EUNSUPPORTED
