"""Masked products of few rows, columns or K steps, whole and in parts: FP8 and 3xTF32
tiles of which rows, columns or whole pieces lie outside C, with a beta."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("steps", [1, 3, 4, 7, 8, 16, 32])          # of 128: whole, then 2, 4 and 8 parts
@pytest.mark.parametrize("m,l", [(1, 3), (22, 198), (33, 225), (65, 636), (127, 128), (128, 33), (300, 450)])
@pytest.mark.parametrize("kind", ["fp8", "tf32x2"])
def test_thin(ops, kind, m, l, steps):
    b, P = (128 * steps, 1) if steps < 8 else (128 * steps // 8, 8)
    rng = np.random.default_rng(1000 * m + steps)
    p = ops.plan(b * P, b, P, 0, 0)
    mask = (1 << P) - 1
    A64, B64 = (rng.integers(-8, 9, size=(r, p.z)).astype(np.float64) / 4 for r in (m, l))   # exact in E4M3 and TF32
    flat = torch.full((m * (l + 1) + 1,), 0.5, device="cuda")
    C = flat[1:].view(m, l + 1)[:, :l]
    if kind == "fp8":
        A, B = (torch.from_numpy(x.astype(np.float32)).cuda().to(torch.float8_e4m3fn) for x in (A64, B64))
        sa, sb = (torch.full((p.z // 128, (r + 3) // 4 * 4), 2.0, device="cuda") for r in (m, l))
        ops.gemm_masked(p, A, B, mask, a_scales=sa, b_scales=sb, beta=2.0, C=C)
        A64 = 4 * A64
    else:
        A, B = (torch.zeros((2, r, p.z), device="cuda") for r in (m, l))
        A[0].copy_(torch.from_numpy(A64))
        B[0].copy_(torch.from_numpy(B64))
        ops.gemm_masked(p, A[0], B[0], mask, dtype="tf32x2", beta=2.0, C=C)
    ref = oracle.masked_product(A64, B64.T, b, mask) + 1.0
    # every sum is a multiple of 2^-4 (2^-2) below 2^17: exact up to 1/k and the beta term
    mag = oracle.masked_product(np.abs(A64), np.abs(B64).T, b, mask) + 1.0
    assert (np.abs(C.double().cpu().numpy() - ref) <= 4 * 2.0 ** -24 * mag).all()
    rest = flat.clone()
    rest[1:].view(m, l + 1)[:, :l] = 0.5
    assert bool((rest == 0.5).all())
    assert ops.device_status() == 0
