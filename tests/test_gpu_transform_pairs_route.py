"""The bf16 transform by pairs of columns and, with that kernel switched off, its fallbacks: which kernel ran, bit for bit the same
results, and a bounded wait that runs out."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b

pytestmark = pytest.mark.gpu

SHAPES = [(3, 5, 15, 15), (2, 3, 31, 31), (5, 7, 12, 14), (1, 2, 40, 227), (2, 3, 60, 61), (9, 11, 13, 11), (1, 1, 11, 11), (1, 3, 90, 130)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    ensure_built()
    yield
    reset_config()


@pytest.mark.parametrize("route", ["pairs", "fallback"])
@pytest.mark.parametrize("fh", [3, 5, 7, 11])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_route_and_bits(shape, fh, route):
    n, c, h, w = shape
    rng = np.random.default_rng(h * w)
    x = rng.standard_normal((n, c, h, w)).astype(np.float32)
    apply_config(transform_pairs=2 if route == "fallback" else 0)
    for s in (1, 2):
        dims = (n, c, h, w, 1, fh, 1, s)
        ref = torch.from_numpy(oracle.im2win(x, oracle.Shape(*dims)).astype(np.float32)).bfloat16().view(torch.int16).flatten()
        full = torch.full((ref.numel() + 64,), 21555, dtype=torch.int16, device="cuda")
        out = full[32:-32]
        b.transform_bf16(torch.from_numpy(x).cuda(), dims, out)
        assert b.last_device_status() == 0
        took = b.last_transform()
        planned = b.lib().im2win_debug_tile_plan(ctypes.byref(b.Shape(*dims)), 2, (ctypes.c_int64 * 11)()) == b.OK
        assert planned or fh > 3  # (tall filters: blocks of few rows are left to the others)
        assert (took == b.TRANSFORM_PAIRS) == (route == "pairs" and planned) and took != b.TRANSFORM_NONE
        assert torch.equal(out.cpu(), ref)
        assert bool((full[:32] == 21555).all()) and bool((full[-32:] == 21555).all())


def test_bounded_wait_expiry_is_reported_and_the_context_survives():
    """As for the tile kernel: an input copy that is announced and never issued, on a problem of one CTA."""
    dims = (1, 1, 8, 8, 1, 3, 3, 1)
    x = torch.randn((1, 1, 8, 8), device="cuda")
    out = torch.empty(6 * 24, dtype=torch.int16, device="cuda")
    apply_config("hook", test_skip_copy=1)
    b.transform_bf16(x, dims, out)
    rc, status = b.last_device_status_rc()  # (synchronises; the wait takes about a second)
    assert b.last_transform() == b.TRANSFORM_PAIRS
    assert rc == b.ETIMEOUT and status == 109, (rc, status)
    b.set_option("test_skip_copy", 0)
    assert b.last_device_status() == 0
    b.transform_bf16(x, dims, out)
    assert b.last_device_status() == 0
    ref = oracle.im2win(x.cpu().numpy(), oracle.Shape(*dims)).astype(np.float32)
    assert torch.equal(out.cpu(), torch.from_numpy(ref).bfloat16().view(torch.int16).flatten())
