"""The transform's column-by-column transposition (odd row lengths, odd filter heights), bit for bit against Algorithm 1
written as a stack of shifted rows: whole planes and row blocks, ragged last blocks, one-column images, both storages."""
import pytest

from paper_2306_14320_b200 import binding as b
from gpu_helpers import ensure_built

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# N, C, H, W, Fh, stride
SHAPES = [
    (2, 32, 21, 25, 3, 2), (3, 5, 9, 9, 3, 1), (2, 7, 15, 15, 5, 1), (2, 3, 111, 111, 7, 2), (1, 1, 11, 11, 11, 1), (1, 2, 7, 1, 7, 1),
    (2, 3, 227, 227, 11, 4), (1, 2, 60, 1001, 3, 1), (130, 40, 5, 3, 3, 1), (1, 3, 225, 225, 7, 2), (2, 3, 61, 301, 11, 3),
]


@pytest.mark.parametrize("bf16", [False, True], ids=["fp32", "bf16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_odd_rows_bit_exact(shape, bf16):
    ensure_built()
    n, c, h, w, fh, s = shape
    dims = (n, c, h, w, 1, fh, 1, s)
    ho, _ = b.out_dims(dims)
    x = torch.randn((n, c, h, w), device="cuda")
    out = torch.full((n * c * ho * w * fh + 16,), -7.0, device="cuda", dtype=torch.bfloat16 if bf16 else torch.float32)
    (b.transform_bf16 if bf16 else b.transform)(x, dims, out[:-16])
    assert b.last_device_status() == 0
    ref = torch.stack([x[:, :, u:u + (ho - 1) * s + 1:s] for u in range(fh)], -1).reshape(-1).to(out.dtype)
    assert torch.equal(out[:-16], ref) and bool((out[-16:] == -7.0).all())
