"""The one-pass sparse-row sketch at its edges: one and two rows per CTA at a time,
rows and block widths that are no multiple of anything, buckets longer than the
sorting network, rows that overflow a region, index ranges at 2^20."""
import numpy as np
import pytest

import oracle
from helpers import assert_bf16_within, assert_fp32_within, gpu_lib, sketch_bounds_left

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _sparse(rng, m, n, density):
    A = np.zeros((m, n), np.float32)
    for r in range(m):
        d = density if np.isscalar(density) else density[r % len(density)]
        k = int(round(d * n))
        A[r, rng.choice(n, size=k, replace=False)] = rng.standard_normal(k)
    return A


@pytest.mark.parametrize("m,n,b,P,mask,density,dtype,off", [
    (40, 30011, 4096, 3, 0b101, 0.02, "f32", 0),               # one row per CTA at a time, rows not 16-byte aligned
    (331, 30016, 4096, 2, 0b11, 0.02, "f32", 0),               # two rows at a time, three rows in some CTAs
    (457, 9001, 100, 3, 0b110, 0.01, "f32", 0),                # b no multiple of 8, unaligned rows
    (310, 16388, 130, 2, 0b11, [0.0, 0.1, 0.0005], "f32", 4),  # long buckets, empty rows, rows offset by 16 bytes
    (400, 20000, 512, 2, 0b10, 0.03, "bf16", 0),               # BF16 operand
    (320, 40960, 256, 2, 0b11, [0.001, 0.9, 0.01], "f32", 0),  # dense rows overflow their regions
])
def test_onepass_rows(ops, m, n, b, P, mask, density, dtype, off):
    rng = np.random.default_rng(m + n)
    A = _sparse(rng, m, n, density)
    Ad = torch.zeros((m, n + off), device="cuda")[:, off:]
    Ad.copy_(torch.from_numpy(A))
    if dtype == "bf16":
        Ad = Ad.to(torch.bfloat16)
        A = Ad.float().cpu().numpy()
    p = ops.plan(n, b, P, 0, 4)
    h, s = oracle.hash_tables(n, b, P, 0, 4)
    ref, bound = sketch_bounds_left(A, h, s, b)
    cols = np.concatenate([np.arange(j * b, (j + 1) * b) for j in range(P) if mask >> j & 1])
    At, _ = ops.sketch_left_sparse(p, Ad, "f32", block_mask=mask)
    assert_fp32_within(At.cpu().numpy()[:, cols], ref[:, cols], bound[:, cols])
    again, _ = ops.sketch_left_sparse(p, Ad, "f32", block_mask=mask)
    assert torch.equal(At[:, cols], again[:, cols])
    if b % 8 == 0:
        Ab, _ = ops.sketch_left_sparse(p, Ad, "bf16", block_mask=mask)
        assert torch.equal(Ab[:, cols], At[:, cols].to(torch.bfloat16))


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 4])
def test_onepass_index_range(ops, n):
    """Nonzeros at the ends of the row and of the warps' shares, at and past the 16-bit index range."""
    m, b = 160, 1024
    rng = np.random.default_rng(n)
    A = torch.zeros((m, n), device="cuda")
    cols = np.unique(np.concatenate([[0, 1, n - 1, n - 2], np.arange(0, n, 65536), np.arange(65535, n, 65536),
                                     rng.choice(n, 300, replace=False)]))
    vals = rng.standard_normal((m, len(cols))).astype(np.float32)
    A[:, torch.from_numpy(cols).cuda()] = torch.from_numpy(vals).cuda()
    p = ops.plan(n, b, 2, 0, 9)
    h, s = oracle.hash_tables(n, b, 2, 0, 9)
    ref, bound = sketch_bounds_left(vals, h[:, cols], s[:, cols], b)
    At, _ = ops.sketch_left_sparse(p, A, "f32")
    assert_fp32_within(At.cpu().numpy(), ref, bound)
    Ab, _ = ops.sketch_left_sparse(p, A, "bf16")
    assert_bf16_within(Ab.double().cpu().numpy(), ref, bound)


def test_onepass_fp8_and_tables(ops):
    m, n, b, P = 306, 24000, 384, 2
    rng = np.random.default_rng(5)
    A = _sparse(rng, m, n, 0.02)
    h, s = oracle.hash_tables(n, b, P, 0, 8)
    p, q = ops.plan(n, b, P, 0, 8), ops.plan_from_tables(h, s, b, P, 0)
    Ad = torch.from_numpy(A).cuda()
    X, Y = ops.sketch_left_sparse(p, Ad, "f32")[0], ops.sketch_left_sparse(q, Ad, "f32")[0]
    assert torch.equal(X, Y)
    Q, sc = ops.sketch_left_sparse(p, Ad, "fp8")
    scale = sc[:, :m].t().repeat_interleave(128, dim=1)
    assert torch.equal(Q.float(), (X / scale).to(torch.float8_e4m3fn).float())
    amax = X.abs().view(m, -1, 128).amax(dim=2)
    assert bool((amax <= 448 * sc[:, :m].t()).all()) and bool(((amax == 0) | (amax > 224 * sc[:, :m].t())).all())
