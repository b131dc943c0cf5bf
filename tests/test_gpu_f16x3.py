"""The FP32 product on FP16 planes: parity with the oracle at its tile edges, no
larger an error than the 3xTF32 product of the same operands, and operands that the
planes do not suit (wide rows, huge and tiny magnitudes, Inf and NaN), which must
give what the 3xTF32 product gives."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _operands(m, n, l, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randn((m, n), generator=g, device="cuda"), torch.randn((n, l), generator=g, device="cuda"))


def _reference(ops, p, A, B, mask):
    """FP64 product of the library's own FP32 sums (so only the GEMM's error shows), and the
    product of their magnitudes."""
    At, Bt = ops.sketch_left(p, A, "f32")[0].double(), ops.sketch_right(p, B, "f32")[0].double()
    cols = torch.cat([torch.arange(j * p.b, (j + 1) * p.b) for j in range(p.P) if mask >> j & 1]).cuda()
    k = bin(mask).count("1")
    return At[:, cols] @ Bt[:, cols].t() / k, At[:, cols].abs() @ Bt[:, cols].abs().t() / k


@pytest.mark.parametrize("m,n,l,b,N,e,mask", [
    (1500, 9000, 1601, 704, 4, 1, 0b11011),     # ragged tiles of 256 x 160, odd ldc, K = 44 chunks
    (2560, 8192, 1920, 512, 4, 2, 0b101101),    # whole tiles
    (4001, 4096, 4003, 64, 5, 1, 0b011111),     # K = 320: a chunk of one step
    (6001, 4096, 6003, 192, 3, 1, 0b1011),      # K = 576: the third chunk of one step
    (257, 20000, 12801, 1024, 2, 0, 0b11),      # a second tile row of one row
])
def test_f16x3_parity(ops, m, n, l, b, N, e, mask):
    A, B = _operands(m, n, l, m)
    p = ops.plan(n, b, N, e, 5)
    ref, mag = _reference(ops, p, A, B, mask)
    C = ops.matmul(p, A, B, mask, "f32").double()
    T = ops.matmul(p, A, B, mask, "tf32x2").double()
    # 16 truncated accumulations of FP32 per chunk (2^-23 each), FP32 chunk sums, 2^-24 per split and dropped term
    K = bin(mask).count("1") * b
    assert bool(((C - ref).abs() <= (16 * 2.0 ** -23 + (K / 256 + 8) * 2.0 ** -24) * mag + 1e-30).all())
    assert float((C - ref).norm()) <= float((T - ref).norm())
    assert bool((C == ops.matmul(p, A, B, mask, "f32").double()).all())
    assert ops.device_status() == 0


@pytest.mark.parametrize("kind", ["wide", "huge", "tiny", "inf", "nan"])
def test_rows_the_planes_do_not_suit(ops, kind):
    m, n, l, b, N, e, mask = 1300, 2048, 1500, 1024, 4, 0, 0b1111
    A, B = _operands(m, n, l, 3)
    if kind == "wide":
        A *= 1e-6
        A[7, 100] = 1e6
        B[100] = 0.0
    elif kind == "huge":
        A[3] *= 1e25
    elif kind == "tiny":
        B[:, 11] *= 1e-20
    else:
        A[5, 17] = float(kind)
    p = ops.plan(n, b, N, e, 1)
    C, T = ops.matmul(p, A, B, mask, "f32"), ops.matmul(p, A, B, mask, "tf32x2")
    assert bool(((C == T) | (C.isnan() & T.isnan())).all())


def test_f16x3_symmetric_and_zero_rows(ops):
    m, n, b, N, e, mask = 1400, 6000, 1024, 4, 1, 0b11101
    A, _ = _operands(m, n, 1, 9)
    A[100:356] = 0.0
    p = ops.plan(n, b, N, e, 2)
    H = ops.matmul(p, A, None, mask, "f32", symmetric=True).cpu().numpy()
    h, s = oracle.hash_tables(n, b, N, e, 2)
    A64 = A.cpu().numpy()
    assert oracle.rel_frob(H, oracle.oversketch(A64, A64.T, h, s, b, mask)) <= 1e-5
    assert (H[100:356] == 0).all() and (H[:, 100:356] == 0).all()
