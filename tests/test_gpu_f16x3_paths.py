"""The FP32 product on FP16 planes at the edges of its tiles and through its other entry
points, at sizes well inside its dispatch rule: every case asserts that the result is
not the 3xTF32 one, so the planes did run."""
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


@pytest.mark.parametrize("m,n,l,b,N,e,mask", [
    (12001, 4096, 12003, 64, 5, 1, 0b011111),    # K = 320: one chunk of four steps and one of one
    (9001, 4096, 9003, 192, 3, 1, 0b1011),       # K = 576: the third chunk of one step
    (4097, 8192, 4097, 1024, 4, 1, 0b11011),     # one row past 16 tile pairs
    (4353, 4096, 4001, 512, 2, 1, 0b101),        # one row past 17 pairs, one column past 25 tiles
    (3841, 8192, 4000, 256, 8, 2, 0b1110111101),  # whole tiles of columns, eight kept blocks
])
def test_planes_at_tile_edges(ops, m, n, l, b, N, e, mask):
    A, B = _operands(m, n, l, m)
    p = ops.plan(n, b, N, e, 5)
    At, Bt = ops.sketch_left(p, A, "f32")[0].double(), ops.sketch_right(p, B, "f32")[0].double()
    cols = torch.cat([torch.arange(j * b, (j + 1) * b) for j in range(N + e) if mask >> j & 1]).cuda()
    k = bin(mask).count("1")
    ref, mag = At[:, cols] @ Bt[:, cols].t() / k, At[:, cols].abs() @ Bt[:, cols].abs().t() / k
    pad = torch.full((m, l + 3), 7.25, device="cuda")
    C = ops.matmul(p, A, B, mask, "f32", C=pad[:, :l])
    T = ops.matmul(p, A, B, mask, "tf32x2")
    # a chunk's 16 truncated accumulations (2^-23), K / 256 chunk sums, two splits, the
    # dropped lo.lo (2^-22) and four roundings
    bound = (16 * 2.0 ** -23 + (k * b / 256 + 12) * 2.0 ** -24) * mag + 1e-30
    assert bool(((C.double() - ref).abs() <= bound).all())
    assert float((C.double() - ref).norm()) <= float((T.double() - ref).norm())
    assert not torch.equal(C, T)
    assert bool((pad[:, l:] == 7.25).all())
    assert ops.device_status() == 0


def test_planes_from_host_buffers(ops):
    m, n, l, b, N, e, mask = 2600, 6000, 2500, 1024, 4, 1, 0b10111
    A, B = _operands(m, n, l, 1)
    p = ops.plan(n, b, N, e, 2)
    C = ops.matmul_host(p, A.cpu().pin_memory(), B.cpu().pin_memory(), mask, "f32")
    torch.cuda.synchronize()
    assert torch.equal(C, ops.matmul(p, A, B, mask, "f32").cpu())
    assert not torch.equal(C, ops.matmul(p, A, B, mask, "tf32x2").cpu())


@pytest.mark.parametrize("sparse_a", [False, True])
def test_planes_of_a_scaled_gram_matrix(ops, sparse_a):
    m, n, b, N, e, mask = 3000, 40000, 1024, 4, 1, 0b11101
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    u = torch.rand((m, n), generator=g, device="cuda")
    A = torch.where(u < 0.02, u * 100 - 1, 0.0)
    s = torch.rand(n, generator=g, device="cuda") + 0.25
    p = ops.plan(n, b, N, e, 4)
    C = ops.matmul(p, A, None, mask, "f32", col_scale=s, symmetric=True, sparse_a=sparse_a)
    T = ops.matmul(p, A, None, mask, "tf32x2", col_scale=s, symmetric=True, sparse_a=sparse_a)
    assert not torch.equal(C, T)
    h, sg = oracle.hash_tables(n, b, N, e, 4)
    rows = np.arange(0, m, 37)
    At = oracle.sketch_left(A[rows].cpu().numpy(), h, sg, b, s.cpu().numpy())
    ref = oracle.masked_product(At, At.T, b, mask)
    assert oracle.rel_frob(C[rows][:, rows].cpu().numpy(), ref) <= 1e-5
