"""Scaled FP32 gathers in the mixed order of CTAs: every strip, block and tile once,
for one and several blocks and strips, ragged tiles, in place and packed."""
import numpy as np
import pytest

import oracle
from helpers import assert_fp32_within, gpu_lib, max_bucket

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("n,l,b,P,mask", [
    (3000, 128, 40, 3, 0b101),          # one strip
    (3000, 640, 48, 1, 0b1),            # one block
    (5000, 513, 33, 4, 0b1110),         # ragged tile per block, five strips, the last one column wide
    (2000, 1300, 256, 6, 0b110111),     # many tiles
])
def test_scaled_sketches_cover_every_tile(ops, n, l, b, P, mask):
    rng = np.random.default_rng(n + l)
    B = rng.standard_normal((n, l)).astype(np.float32)
    s = (2.0 ** rng.integers(-3, 4, n)).astype(np.float32)        # exact products
    p = ops.plan(n, b, P, 0, 2)
    h, sg = oracle.hash_tables(n, b, P, 0, 2)
    ref = oracle.sketch_right(B.astype(np.float64) * s[:, None], h, sg, b).T
    mag = oracle.sketch_right(np.abs(B.astype(np.float64)) * s[:, None], h, np.ones_like(sg), b).T
    bound = (max_bucket(h, b) + 1) * 2.0 ** -23 * mag
    cols = np.concatenate([np.arange(j * b, (j + 1) * b) for j in range(P) if mask >> j & 1])
    Bd, sd = torch.from_numpy(B).cuda(), torch.from_numpy(s).cuda()
    nan = float("nan")
    for fn, X, kw in ((ops.sketch_right, Bd, dict(row_scale=sd)), (ops.sketch_left, Bd.t().contiguous(), dict(col_scale=sd))):
        out = torch.full((l, (p.z + 3) // 4 * 4), nan, device="cuda")[:, :p.z]
        Y, _ = fn(p, X, "f32", out=out, block_mask=mask, **kw)
        Y = Y.cpu().numpy()
        assert_fp32_within(Y[:, cols], ref[:, cols], bound[:, cols])
        assert np.isnan(np.delete(Y, cols, axis=1)).all()         # unlisted blocks untouched
