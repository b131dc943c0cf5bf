"""The staged FP8 quantisation over few and many slices per row and in all (a warp takes
one slice, or four of a row)."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("m,b,P,mask", [
    (1, 128, 2, 0b01),               # one slice
    (7, 128, 9, 0b101101101),        # six slices a row
    (3300, 128, 5, 0b10101),         # three a row, past one warp per slice: a part of four
    (1000, 640, 4, 0b1101),          # fifteen a row: three turns of four, one of three
    (2000, 256, 4, 0b1111),          # eight
])
def test_staged_quantisation(ops, m, b, P, mask):
    n = 1500
    g = torch.Generator(device="cuda")
    g.manual_seed(m + b)
    A = torch.randn((m, n), generator=g, device="cuda") * torch.exp2(torch.randint(-30, 30, (m, 1), generator=g, device="cuda").float())
    A[m // 2] = 0.0
    p = ops.plan(n, b, P, 0, 3)
    staged = torch.empty(ops.sketch_workspace(p, m) + 512 + 4 * m * p.z, dtype=torch.uint8, device="cuda")
    sums, _ = ops.sketch_left(p, A, "f32", block_mask=mask)
    codes, scales = ops.sketch_left(p, A, "fp8", block_mask=mask, workspace=staged)
    sl = [j * b // 128 + t for j in range(P) if mask >> j & 1 for t in range(b // 128)]
    cols = np.concatenate([np.arange(128 * t, 128 * t + 128) for t in sl])
    q, e = oracle.quantize_fp8_rows(sums.cpu().numpy()[:, cols])     # the sums are the same bits
    assert np.array_equal(codes.float().cpu().numpy()[:, cols].astype(np.float64), q)
    assert np.array_equal(scales.cpu().numpy()[sl][:, :m].T.astype(np.float64), np.ldexp(1.0, e))
