"""Products of few tiles: a tile's K steps shared by the CTAs of a cluster (TF32 planes,
FP8), and the one-CTA BF16 kernel, at ragged tiles, odd leading dimensions, an uneven
last share of K and a beta."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _operand(rng, rows, z, dt):
    """Device operand, its scales (FP8) and its exact FP64 values."""
    x = rng.standard_normal((rows, z)).astype(np.float32)
    if dt == "tf32x2":
        hi = (x.view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32)
        return torch.from_numpy(np.stack([hi, x - hi])).cuda()[0], None, x.astype(np.float64)
    if dt == "bf16":
        t = torch.from_numpy(x).to(torch.bfloat16).cuda()
        return t, None, t.float().cpu().numpy().astype(np.float64)
    codes, e = oracle.quantize_fp8_rows(x)
    q = torch.from_numpy(np.asarray(codes, np.float32)).to(torch.float8_e4m3fn)
    sc = np.full((z // 128, (rows + 3) // 4 * 4), np.nan, np.float32)      # padding rows are never read
    sc[:, :rows] = np.ldexp(1.0, np.asarray(e, np.int64)).T
    return q.cuda(), torch.from_numpy(sc).cuda(), oracle.dequantize_fp8_rows(codes, e)


@pytest.mark.parametrize("dt", ["tf32x2", "bf16", "fp8"])
@pytest.mark.parametrize("m,l,b,N,e,mask,pad,beta", [
    (128, 128, 256, 2, 0, 0b11, 0, 0.0),         # one tile
    (300, 257, 384, 4, 1, 0b10111, 3, 0.5),      # ragged tiles, odd ldc, shares that start inside a block
    (1, 515, 1152, 3, 1, 0b1101, 0, 0.0),        # one row
    (513, 700, 128, 5, 0, 0b11111, 1, -1.5),     # shares of different lengths
    (1000, 900, 640, 2, 1, 0b101, 4, 0.0),       # two CTAs per tile, or none to share with
    (130, 4000, 128, 1, 0, 0b1, 0, 0.0),         # too little K to share
])
def test_few_tiles(ops, dt, m, l, b, N, e, mask, pad, beta):
    rng = np.random.default_rng(m + l)
    z = (N + e) * b
    A, sa, A64 = _operand(rng, m, z, dt)
    B, sb, B64 = _operand(rng, l, z, dt)
    p = ops.plan(max(z, 64), b, N, e, 0)
    C0 = torch.from_numpy(rng.standard_normal((m, l + pad)).astype(np.float32)).cuda()
    C = C0.clone()
    kw = dict(dtype=dt, a_scales=sa, b_scales=sb, beta=beta)
    ops.gemm_masked(p, A, B, mask, C=C[:, :l], **kw)
    old = C0.cpu().numpy().astype(np.float64)
    ref = oracle.masked_product(A64, B64.T, b, mask) + beta * old[:, :l]
    mag = oracle.masked_product(np.abs(A64), np.abs(B64).T, b, mask) + abs(beta) * np.abs(old[:, :l])
    # K truncated FP32 additions (2^-23 each); with planes lo * lo and lo's own rounding (2^-20 each) as well
    K = bin(mask).count("1") * b
    bound = (K * 2.0 ** -23 + (4 * 2.0 ** -20 if dt == "tf32x2" else 0.0)) * mag + 1e-30
    assert (np.abs(C[:, :l].cpu().numpy() - ref) <= bound).all()
    assert torch.equal(C[:, l:], C0[:, l:])
    again = C0.clone()
    ops.gemm_masked(p, A, B, mask, C=again[:, :l], **kw)
    assert torch.equal(again, C)
    assert ops.device_status() == 0
