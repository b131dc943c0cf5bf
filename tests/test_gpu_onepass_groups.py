"""One or two rows at a time in the sparse-row sketch, chosen by the nonzeros a sample
of A finds: on both sides of the line, and with rows far from the average, every row
gets the bits that a call of few rows (one at a time) gives it."""
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("out_dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("m,n,ld,b,per_row,dense_row,in_dtype", [
    (305, 65536, 65536, 2048, 900, None, "f32"),        # below 1024 a row: two groups
    (305, 65536, 65536, 2048, 1200, None, "f32"),       # above: one
    (333, 65537, 65539, 512, 4000, 17, "f32"),          # rows of no alignment, one of them full
    (305, 65536, 65536, 1024, 14, 304, "bf16"),
    (160, 1 << 20, 1 << 20, 4096, 15500, None, "f32"),  # more than two groups hold, no more than one
    (160, 1 << 20, 1 << 20, 2048, 12000, 3, "f32"),
    (160, 1 << 20, 1 << 20, 2048, 23000, None, "bf16"),  # more than either holds
])
def test_rows_do_not_depend_on_the_groups(m, n, ld, b, per_row, dense_row, in_dtype, out_dtype):
    ops = gpu_lib()
    g = torch.Generator(device="cuda")
    g.manual_seed(per_row)
    A = torch.zeros((m, ld), device="cuda")
    for r in range(0, m, 32):
        u = torch.rand((min(32, m - r), n), generator=g, device="cuda")
        A[r:r + 32, :n] = torch.where(u < per_row / n, u * (n / per_row) - 0.5, 0.0)
    if dense_row is not None:
        A[dense_row, :n] = torch.randn(n, generator=g, device="cuda")
    A[1] = 0.0
    A = A.to(torch.bfloat16 if in_dtype == "bf16" else torch.float32)[:, :n]
    p = ops.plan(n, b, 3, 1, 7)
    s = torch.rand(n, generator=g, device="cuda") + 0.5
    for scale in (None, s):
        At, sc = ops.sketch_left_sparse(p, A, out_dtype, col_scale=scale, block_mask=0b1011)
        keep = torch.cat([torch.arange(j * b, (j + 1) * b) for j in (0, 1, 3)]).cuda()
        for r in range(0, m, 100):
            few, fsc = ops.sketch_left_sparse(p, A[r:r + 100], out_dtype, col_scale=scale, block_mask=0b1011)
            x, y = At[r:r + 100], few
            if out_dtype == "fp8":
                x, y = x.view(torch.uint8), y.view(torch.uint8)
                k = torch.cat([torch.arange(j * b // 128, (j + 1) * b // 128) for j in (0, 1, 3)]).cuda()
                rows = min(100, m - r)
                assert torch.equal(sc[k, r:r + rows], fsc[k, :rows])
            assert torch.equal(x[:, keep], y[:, keep])
