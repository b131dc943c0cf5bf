"""The cast to rows of no 16-byte alignment: from one column to past a CTA's width, and the
memory beside the rows."""
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("rows,cols,ldx,ldy", [(1, 1, 1, 1), (9, 3, 3, 3), (300, 31, 32, 33), (70, 2049, 2056, 2051),
                                               (5, 5003, 5003, 5005), (20000, 65, 72, 65)])
def test_cast_to_unaligned_rows(ops, rows, cols, ldx, ldy):
    x = torch.randn((rows, ldx), device="cuda")[:, :cols]
    for src, out in ((x, "bf16"), (x.to(torch.bfloat16), "f32"), (x, "f32")):
        flat = torch.full((rows * ldy + 1,), 3.0, device="cuda", dtype=torch.float32 if out == "f32" else torch.bfloat16)
        y = flat[1:].view(rows, ldy)
        ops.cast(src, out, out=y[:, :cols])
        assert torch.equal(y[:, :cols], src.to(y.dtype)) and bool((y[:, cols:] == 3.0).all()) and float(flat[0]) == 3.0
