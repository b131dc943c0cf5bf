"""The FP8 product on CTA pairs at its edges: an odd count of row tiles, ragged
columns, K steps that leave a stage or a scale group partly filled, blocks of one
step with some dropped, several tiles per pair, an odd ldc with a beta, and scales
over a wide range whose padding must not be read."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _operand(rng, rows, z):
    """E4M3 codes without NaN, power-of-two scales per (row, 128 columns), exact FP64 values."""
    codes = rng.integers(0, 256, size=(rows, z), dtype=np.uint8)
    codes[(codes & 0x7F) == 0x7F] = 0x38
    q = torch.from_numpy(codes).cuda().view(torch.float8_e4m3fn)
    e = rng.integers(-40, 41, size=(z // 128, rows))
    sc = np.full((z // 128, (rows + 3) // 4 * 4), np.nan, np.float32)
    sc[:, :rows] = np.ldexp(1.0, e)
    vals = q.float().cpu().numpy().astype(np.float64) * np.repeat(np.ldexp(1.0, e).T, 128, axis=1)
    return q, torch.from_numpy(sc).cuda(), vals


@pytest.mark.parametrize("m,l,b,N,e,mask,pad,beta", [
    (1300, 1500, 1024, 2, 1, 0b101, 0, 0.0),                # 77 one-CTA tiles: the first past the split ones
    (2561, 2100, 128, 15, 6, 0b11111101111110110111, 3, 0.5),   # 17 steps, each its own block; one row in the last tile
    (2000, 1999, 896, 2, 0, 0b11, 1, 0.0),                  # 14 steps: a scale group of two
    (4000, 4000, 640, 3, 1, 0b1101, 0, -1.0),               # 15 steps, several tiles per pair
])
def test_fp8_pairs(ops, m, l, b, N, e, mask, pad, beta):
    rng = np.random.default_rng(m)
    z = (N + e) * b
    A, sa, A64 = _operand(rng, m, z)
    B, sb, B64 = _operand(rng, l, z)
    p = ops.plan(z, b, N, e, 0)
    C0 = torch.from_numpy(rng.standard_normal((m, l + pad)).astype(np.float32)).cuda()
    C = C0.clone()
    ops.gemm_masked(p, A, B, mask, a_scales=sa, b_scales=sb, beta=beta, C=C[:, :l])
    old = C0.double()
    cols = torch.from_numpy(oracle.selected_columns(mask, N + e, b)).cuda()
    k = bin(mask).count("1")
    Ad, Bd = torch.from_numpy(A64).cuda()[:, cols], torch.from_numpy(B64).cuda()[:, cols]
    ref = Ad @ Bd.t() / k + beta * old[:, :l]
    mag = Ad.abs() @ Bd.abs().t() / k + abs(beta) * old[:, :l].abs()
    # exact products, K truncated FP32 additions (2^-23 each)
    assert bool(((C[:, :l].double() - ref).abs() <= k * b * 2.0 ** -23 * mag + 1e-30).all())
    assert torch.equal(C[:, l:], C0[:, l:])
    assert ops.device_status() == 0
