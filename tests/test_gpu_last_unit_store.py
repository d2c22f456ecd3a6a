"""The columns that the warps behind a unit's operand store themselves, behind a CTA's last unit or (one accumulator) behind every
one: bit for bit on small integers, with one operand stage per unit, several units per CTA, and one and two accumulators."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

WINDOW = {"force_window": 1}
STRIP = {"force_strip": 1, "no_window": 1}
CONFIGS = {
    "window one block": {**WINDOW, "window_mh": 1, "window_pair": 2}, "window two": {**WINDOW, "window_mh": 2, "window_pair": 2},
    "window two, epilogue warps alone": {**WINDOW, "window_mh": 2, "window_pair": 2, "window_nohelp": 1},
    "window pairs": {**WINDOW, "window_mh": 1, "window_pair": 1}, "window pairs two": {**WINDOW, "window_mh": 2, "window_pair": 1},
    "window pairs two, epilogue warps alone": {**WINDOW, "window_mh": 2, "window_pair": 1, "window_nohelp": 1},
    "strip one block": {**STRIP, "strip_mh": 1, "strip_pair": 2}, "strip two": {**STRIP, "strip_mh": 2, "strip_pair": 2},
    "strip pairs": {**STRIP, "strip_mh": 1, "strip_pair": 1}, "strip pairs two": {**STRIP, "strip_mh": 2, "strip_pair": 1},
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


@pytest.mark.parametrize("images", [37, 120])
@pytest.mark.parametrize("filters", [64, 160])  # two blocks of 64 columns leave room for two accumulators, of 160 for one
@pytest.mark.parametrize("config", CONFIGS)
def test_result(config, filters, images):
    rng = np.random.default_rng(filters)
    for mode, c in ((b.MODE_TF32, 16), (b.MODE_BF16, 32)):
        dims = (images, c, 30, 32, filters, 3, 3, 1)
        few = rng.integers(-3, 4, (3, *dims[1:4])).astype(np.float32)
        f = rng.integers(-3, 4, (filters, c, 3, 3)).astype(np.float32)
        ref = oracle.conv_direct(few, f, oracle.Shape(3, *dims[1:])).astype(np.float32).reshape(3, -1)
        x = torch.from_numpy(few).cuda()[torch.arange(images, device="cuda") % 3].contiguous()
        apply_config(config, **CONFIGS[config])
        out, ws = Guarded(images * ref.shape[1]), Guarded(b.conv_workspace_bytes(dims, b.SRC_NCHW, mode) // 4)
        for _ in range(3):
            out.view.fill_(-7.0e37)
            b.conv(x, b.SRC_NCHW_FUSED, torch.from_numpy(f).cuda(), dims, mode, out.view, ws.view)
            assert b.last_kernel() == (b.KERNEL_WINDOW if config.startswith("window") else b.KERNEL_STRIP)
            assert b.last_device_status() == 0
            got = out.check().reshape(images, -1)
            assert all(np.array_equal(got[i], ref[i % 3]) for i in range(images))
