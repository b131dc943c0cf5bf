"""The backward pass's data movement at its edges: the tiles of the transposed gather
into dX (64 x 128), ragged and unaligned rows of dG, the cast, and the BF16 strip
transpose (64 x 128), against FP64 torch."""
import numpy as np
import pytest

import oracle
from helpers import assert_fp32_within, gpu_lib, sketch_bounds_left

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("m,n,l,b,P,mask", [
    (1, 63, 5, 64, 2, 0b11), (127, 64, 3, 64, 3, 0b101), (128, 65, 129, 64, 2, 0b10), (129, 200, 513, 64, 3, 0b111),
    (136, 1000, 520, 128, 5, 0b11011), (260, 777, 1026, 64, 2, 0b11), (8, 129, 8, 128, 2, 0b01),
])
def test_gradients_at_tile_edges(ops, m, n, l, b, P, mask, dt):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n)
    p = ops.plan(n, b, P, 0, 3)
    At = torch.randn((m, p.z), generator=g, device="cuda").to(torch.bfloat16)
    Bt = torch.randn((l, p.z), generator=g, device="cuda").to(torch.bfloat16)
    dC = torch.randn((m, l), generator=g, device="cuda")
    dX, dG = ops.matmul_backward(p, At, Bt, dC, mask, dt, dt)
    h, s = oracle.hash_tables(n, b, P, 0, 3)
    ht, st = torch.from_numpy(h.astype(np.int64)).cuda(), torch.from_numpy(s.astype(np.float64)).cuda()
    kept = [j for j in range(P) if mask >> j & 1]
    d = dC.to(torch.bfloat16).double() / len(kept)
    X, G = torch.zeros((m, n), dtype=torch.float64, device="cuda"), torch.zeros((n, l), dtype=torch.float64, device="cuda")
    for j in kept:
        X += (d @ Bt[:, j * b:(j + 1) * b].double())[:, ht[j]] * st[j]
        G += (At[:, j * b:(j + 1) * b].double().t() @ d)[ht[j]] * st[j][:, None]
    tol = 1e-5 if dt is torch.float32 else 4e-3      # FP32 accumulation; one BF16 rounding of the result
    assert float((dX.double() - X).norm()) <= tol * float(X.norm())
    assert float((dG.double() - G).norm()) <= tol * float(G.norm())
    assert float((dX.double() - X).abs().max()) <= 4 * tol * float(X.abs().max())
    assert float((dG.double() - G).abs().max()) <= 4 * tol * float(G.abs().max())


@pytest.mark.parametrize("rows,cols,ldx,ldy,off", [(1, 1, 1, 8, 0), (3, 7, 8, 8, 0), (100, 2056, 2056, 2056, 0),
                                                   (33, 129, 136, 192, 0), (5, 64, 65, 72, 1), (70000, 9, 12, 16, 0)])
def test_cast_edges(ops, rows, cols, ldx, ldy, off):
    x = torch.randn(off + rows * ldx, device="cuda")[off:].view(rows, ldx)[:, :cols]
    for src, out in ((x, "bf16"), (x.to(torch.bfloat16), "f32"), (x, "f32")):
        y = torch.full((rows, ldy), 3.0, device="cuda", dtype=torch.float32 if out == "f32" else torch.bfloat16)
        ops.cast(src, out, out=y[:, :cols])
        assert torch.equal(y[:, :cols], src.to(y.dtype)) and bool((y[:, cols:] == 3.0).all())


@pytest.mark.parametrize("m,n,off", [(1, 129, 0), (63, 128, 0), (64, 256, 0), (65, 1000, 8), (255, 384, 3), (257, 1024, 0),
                                     (130, 4095, 0)])
def test_bf16_left_sketch_edges(ops, m, n, off):
    rng = np.random.default_rng(m + n)
    A = torch.zeros((m, n + off), dtype=torch.bfloat16, device="cuda")[:, off:]
    A.copy_(torch.from_numpy(rng.standard_normal((m, n)).astype(np.float32)))
    b, P = 64, 2
    p = ops.plan(n, b, P, 0, 6)
    h, s = oracle.hash_tables(n, b, P, 0, 6)
    ref, bound = sketch_bounds_left(A.float().cpu().numpy(), h, s, b)
    At, _ = ops.sketch_left(p, A, "f32")
    assert_fp32_within(At.cpu().numpy(), ref, bound)
