"""The GEMMs' write-out at its edges: rows and columns at and around the 32 x 32
pieces, row pitches with and without 16-byte alignment, beta, and the memory
around C."""
import numpy as np
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.mark.parametrize("beta", [0.0, -0.5])
@pytest.mark.parametrize("m,l,ldc,off", [
    (1, 1, 1, 0), (31, 33, 40, 0), (32, 32, 32, 0), (33, 31, 31, 0), (129, 255, 255, 0), (127, 257, 260, 0),
    (256, 288, 288, 1), (300, 100, 104, 3), (257, 512, 516, 0),
])
def test_write_out_edges(ops, m, l, ldc, off, beta):
    """C = A B^T + beta C in a view with guard columns (and an unaligned start)."""
    rng = np.random.default_rng(m * 1000 + l)
    K = 64
    A = torch.from_numpy(rng.standard_normal((m, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    B = torch.from_numpy(rng.standard_normal((l, K)).astype(np.float32)).to(torch.bfloat16).cuda()
    flat = torch.full((off + m * ldc + 8,), 7.25, device="cuda")
    C = flat[off:off + m * ldc].view(m, ldc)[:, :l]
    ops.gemm_bf16(A, B, beta=beta, C=C)
    a, b = A.double().cpu().numpy(), B.double().cpu().numpy()
    ref = a @ b.T + beta * 7.25
    # K FP32 additions of exact products, the scaling and the beta term
    bound = 2 * (K + 2) * 2.0 ** -24 * (np.abs(a) @ np.abs(b).T + abs(beta) * 7.25)
    assert (np.abs(C.double().cpu().numpy() - ref) <= bound).all()
    rest = flat.clone()
    rest[off:off + m * ldc].view(m, ldc)[:, :l] = 7.25
    assert bool((rest == 7.25).all()), "the write-out touched memory outside C"
