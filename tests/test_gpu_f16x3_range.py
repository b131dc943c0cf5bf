"""The FP32 product on FP16 planes takes operands of any common magnitude, or one row far
from the others: the scale per row follows them, the 3xTF32 product is not needed."""
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("ea,eb,row,er", [
    (-43, 0, 0, 0), (0, 40, 0, 0), (-55, -55, 0, 0), (55, 55, 0, 0),
    (0, 0, 5, -57), (0, 0, 2999, 74), (-57, 74, 17, 0),     # sums up to 2^6 of the entries
])
def test_magnitudes(ops, ea, eb, row, er):
    m, n, l, b, N, e, mask = 3000, 8192, 3001, 1024, 4, 0, 0b1111      # K = 4096
    g = torch.Generator(device="cuda")
    g.manual_seed(60 + ea + row)
    A = torch.randn((m, n), generator=g, device="cuda") * 2.0 ** ea
    B = torch.randn((n, l), generator=g, device="cuda") * 2.0 ** eb
    A[row] *= 2.0 ** er
    p = ops.plan(n, b, N, e, 3)
    C = ops.matmul(p, A, B, mask, "f32")
    T = ops.matmul(p, A, B, mask, "tf32x2")
    At, Bt = ops.sketch_left(p, A, "f32")[0].double(), ops.sketch_right(p, B, "f32")[0].double()
    ref, mag = At @ Bt.t() / 4, At.abs() @ Bt.abs().t() / 4
    # as for operands of magnitude one: 16 truncated accumulations (2^-23) and chunk sums,
    # two splits (2^-23 each), the dropped lo.lo (2^-22), four roundings
    bound = (16 * 2.0 ** -23 + (b * N / 256 + 12) * 2.0 ** -24) * mag
    assert bool(((C.double() - ref).abs() <= bound).all())
    assert not torch.equal(C, T)
    assert ops.device_status() == 0
