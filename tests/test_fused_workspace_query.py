"""im2win_conv_workspace_bytes for fused calls: no room is asked for a filter copy that only the window-offset kernel's wider families
(rectangular filters, channel tails) would read, which take such calls only with room for the im2win tensor; and with it they do."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import SENTINEL, Guarded, apply_config, ensure_built, reset_config
from paper_2306_14320_b200 import binding as b


@pytest.mark.parametrize("mode", [b.MODE_TF32, b.MODE_BF16])
def test_query_holds_what_a_fused_call_can_use(mode):
    for fs in ((1, 1), (1, 3), (3, 1), (1, 7), (7, 1), (3, 5), (5, 3), (3, 4)):
        for c in (17, 40, 64, 96):
            dims = (8, c, 40, 40, 96, *fs, 1)
            assert b.conv_workspace_bytes(dims, b.SRC_NCHW_FUSED, mode) == b.conv_workspace_bytes(dims, b.SRC_IM2WIN, mode)
    for fs in ((3, 3), (5, 5)):
        assert (b.conv_workspace_bytes((8, 40, 40, 40, 96, *fs, 1), b.SRC_NCHW_FUSED, mode)
                <= b.conv_workspace_bytes((8, 40, 40, 40, 96, *fs, 1), b.SRC_IM2WIN, mode))
        assert b.conv_workspace_bytes((8, 64, 40, 40, 96, *fs, 1), b.SRC_NCHW_FUSED, mode) >= 64 * 96 * fs[0] * fs[1] * (2 if mode else 4)


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [b.MODE_TF32, b.MODE_BF16])
@pytest.mark.parametrize("dims, family", [((3, 64, 20, 24, 48, 3, 5, 1), True), ((3, 64, 17, 20, 80, 1, 7, 1), True), ((2, 40, 20, 21, 72, 3, 3, 1), True),
                                          ((2, 64, 20, 20, 64, 3, 3, 1), False), ((2, 64, 20, 20, 96, 5, 5, 1), False)], ids=str)
def test_a_fused_call_with_exactly_the_queried_workspace(dims, family, mode):
    """The window-offset kernel forced: with the queried size the families are other kernels' (or refused, as any call that no fused
    specialisation takes), the square filters on whole filter blocks run; with room for the tensor all of them do."""
    ensure_built()
    rng = np.random.default_rng(dims[1])
    x = rng.integers(-3, 4, dims[:4]).astype(np.float32)
    f = rng.integers(-3, 4, (dims[4], dims[1], dims[5], dims[6])).astype(np.float32)
    ref = oracle.conv_direct(x, f, oracle.Shape(*dims)).astype(np.float32).ravel()
    queried = b.conv_workspace_bytes(dims, b.SRC_NCHW_FUSED, mode)
    xd, fd = torch.from_numpy(x).cuda(), torch.from_numpy(f).cuda()
    try:
        apply_config("window", force_window=1)
        for nbytes in (queried, max(queried, b.workspace_bytes(dims))):
            out, ws = Guarded(ref.size), Guarded((nbytes + 3) // 4 + 64)
            try:
                b.conv(xd, b.SRC_NCHW_FUSED, fd, dims, mode, out.view, ws.view, nbytes)
            except b.Im2winError as e:
                assert e.code == b.EUNSUPPORTED and family and nbytes == queried
                continue
            assert b.last_device_status() == 0 and np.array_equal(out.check(), ref)
            assert (ws.check()[nbytes // 4 + 1:] == np.float32(SENTINEL)).all()
            assert (b.last_kernel() == b.KERNEL_WINDOW) == (not family or nbytes >= b.workspace_bytes(dims))
    finally:
        reset_config()
