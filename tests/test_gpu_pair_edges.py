"""The BF16 product on CTA pairs at its edges: contractions past the short ones that the
one-CTA kernel takes, with rows and columns below and around a tile pair, odd and
misaligned C, alpha and beta, and the memory around C."""
import numpy as np
import pytest

import oracle
from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _bf16(rng, rows, cols):
    t = torch.from_numpy(rng.standard_normal((rows, cols)).astype(np.float32)).to(torch.bfloat16).cuda()
    return t, t.double().cpu().numpy()


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (0.25, -1.5)])
@pytest.mark.parametrize("m,l,ldc,off", [
    (1, 1, 1, 0), (31, 33, 40, 0), (129, 255, 255, 0), (127, 257, 260, 0), (256, 256, 256, 0), (257, 513, 516, 1),
    (300, 700, 701, 0), (255, 100, 104, 3), (513, 31, 32, 2),
])
def test_pair_edges(ops, m, l, ldc, off, alpha, beta):
    rng = np.random.default_rng(m * 1000 + l)
    b, N, e, mask = 1024, 3, 1, 0b1011               # K = 3072
    z = (N + e) * b
    A, A64 = _bf16(rng, m, z)
    B, B64 = _bf16(rng, l, z)
    p = ops.plan(z, b, N, e, 0)
    flat = torch.full((off + m * ldc + 8,), 7.25, device="cuda")
    C = flat[off:off + m * ldc].view(m, ldc)[:, :l]
    ops.gemm_masked(p, A, B, mask, alpha=alpha, beta=beta, C=C)
    ref = alpha * oracle.masked_product(A64, B64.T, b, mask) + beta * 7.25
    mag = alpha * oracle.masked_product(np.abs(A64), np.abs(B64).T, b, mask) + abs(beta) * 7.25
    # K FP32 additions of exact products (truncated: 2^-23 each), the scaling and the beta term
    assert (np.abs(C.double().cpu().numpy() - ref) <= 2 * (N * b + 2) * 2.0 ** -24 * mag).all()
    rest = flat.clone()
    rest[off:off + m * ldc].view(m, ldc)[:, :l] = 7.25
    assert bool((rest == 7.25).all()), "the write-out touched memory outside C"
    assert ops.device_status() == 0


def test_pair_reproducible(ops):
    rng = np.random.default_rng(8)
    A, _ = _bf16(rng, 700, 4096)
    B, _ = _bf16(rng, 901, 4096)
    assert torch.equal(ops.gemm_bf16(A, B), ops.gemm_bf16(A, B))
