"""Entries far below their row's largest in the FP32 product on FP16 planes: where the
other operand is zero beside them the product consists of nothing else, so they must
come out as well as any other (listed and added back, or the whole product as 3xTF32)."""
import numpy as np
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N_, B_, BLOCKS, MASK = 8192, 2048, 2, 0b11      # K = 4096


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


@pytest.fixture(scope="module")
def plan(ops):
    return ops.plan(N_, B_, BLOCKS, 0, 11)


def _columns(p, count):
    """Indices with no two in one bucket of any block: their sketch is exact."""
    h = p.tables()[0]
    used, out = [set() for _ in range(p.P)], []
    for i in range(p.n):
        if all(int(h[j, i]) not in used[j] for j in range(p.P)):
            out.append(i)
            for j in range(p.P):
                used[j].add(int(h[j, i]))
            if len(out) == count:
                return out
    raise AssertionError("too few free buckets")


def _check(ops, p, A, B, **kw):
    """Elementwise bound against FP64 (the sketches are exact); returns C."""
    C = ops.matmul(p, A, B, MASK, "f32", **kw)
    A64, B64 = A.double(), (A.t() if B is None else B).double()
    keep = (A64 != 0).any(0) | (B64 != 0).any(1)
    A64, B64 = A64[:, keep], B64[keep]
    mag = A64.abs() @ B64.abs()
    # a chunk's 16 truncated accumulations (2^-23 each) and K / 256 chunk sums; two splits
    # (2^-23 each), the dropped lo.lo (2^-22) and four roundings of what is added back
    K = BLOCKS * B_
    bound = (16 * 2.0 ** -23 + (K / 256 + 12) * 2.0 ** -24) * mag
    err = (C.double() - A64 @ B64).abs()
    assert bool((err <= bound + 1e-37).all()), float((err / (mag + 1e-300)).max())
    assert torch.equal(C, ops.matmul(p, A, B, MASK, "f32", **kw))
    assert ops.device_status() == 0
    return C


@pytest.mark.parametrize("side", ["A", "B"])
# two listed entries a row: the list may take about 8000 in a product of this size
@pytest.mark.parametrize("rows,listed", [(1, True), (1000, True), (3900, True), (4160, False)])
@pytest.mark.parametrize("exp", [-36, -40, -46, -52])
def test_small_column_beside_zeros(ops, plan, side, rows, listed, exp):
    """One column at 2^exp of the hundred beside it, the other operand zero but there."""
    m = 4160
    cols = _columns(plan, 101)
    g = torch.Generator(device="cuda")
    g.manual_seed(100 - exp)
    X = torch.zeros((m, N_), device="cuda")
    X[:, cols[:100]] = torch.randn((m, 100), generator=g, device="cuda")
    # a row's entries spread over less than a factor of two: exactly `rows` rows are below the line
    X[:rows, cols[100]] = (1 + torch.rand(rows, generator=g, device="cuda")) * 2.0 ** exp
    Y = torch.zeros((m, N_), device="cuda")
    Y[:, cols[100]] = 1 + torch.rand(m, generator=g, device="cuda")
    # no chance entries: the hundred kept away from zero
    X[:, cols[:100]] += X[:, cols[:100]].sign() * 2.0 ** -8
    A, B = (X, Y.t().contiguous()) if side == "A" else (Y, X.t().contiguous())
    C = _check(ops, plan, A, B)
    T = ops.matmul(plan, A, B, MASK, "tf32x2")
    assert torch.equal(C, T) == (not listed)    # past the list: the 3xTF32 product itself


def test_small_entries_on_both_sides(ops, plan):
    """The same sketch columns small in A and in B: each loss is counted once."""
    m, l = 4099, 4001
    cols = _columns(plan, 64)
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A, B = torch.zeros((m, N_), device="cuda"), torch.zeros((N_, l), device="cuda")
    A[:, cols[:30]] = 1 + torch.rand((m, 30), generator=g, device="cuda")
    B[cols[30:60]] = 1 + torch.rand((30, l), generator=g, device="cuda")
    for q, c in enumerate(cols[60:64]):
        A[q::37, c] = 2.0 ** -(34 + 3 * q)
        B[c, q::41] = -2.0 ** -(33 + 2 * q)
        A[7 + 300 * q, c] = 1.5                # and large in a row each
    # every product here is exact in either arithmetic; 2 * (4 * 111 + 4 * 98) entries are listed
    C = _check(ops, plan, A, B)
    assert float(C[0, 0]) != 0.0


def test_small_entries_symmetric(ops, plan):
    m = 4097
    cols = _columns(plan, 33)
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    A = torch.zeros((m, N_), device="cuda")
    A[:900, cols[:32]] = 1 + torch.rand((900, 32), generator=g, device="cuda")
    A[:900, cols[32]] = 2.0 ** -44
    A[900:, cols[32]] = 1 + torch.rand(m - 900, generator=g, device="cuda")
    C = _check(ops, plan, A, None, symmetric=True)
    assert not torch.equal(C, ops.matmul(plan, A, None, MASK, "tf32x2", symmetric=True))
