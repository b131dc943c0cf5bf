"""The bounded waits of the tensor-core kernels beside the one tile of
test_gpu_wait_timeout.py: products on CTA pairs (BF16, FP8, FP32 on FP16 planes,
MN-major and per-block forms) and tiles whose K is shared by a cluster.  The hook
leaves one K step of the first tile unloaded; the wait for it runs out, the pair
waits for the copies and MMAs it issued and returns, the host reads the status, and
the next launch gives what the one before the hook gave."""
import numpy as np
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LIMIT_NS = 200_000


@pytest.fixture(scope="module")
def ops():
    return gpu_lib()


def _bf16(rows, cols, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn((rows, cols), generator=g, device="cuda").to(torch.bfloat16)


def _fp8(rows, z, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    q = torch.randn((rows, z), generator=g, device="cuda").to(torch.float8_e4m3fn)
    return q, torch.ones((z // 128, (rows + 3) // 4 * 4), device="cuda")


def _runs_out(ops, skip_kb, run):
    before = run()
    assert ops.device_status(reset=True) == 0
    ops.test_wait_timeout(LIMIT_NS, skip_kb)
    run()
    assert ops.device_status(reset=True) == 6        # OS_ERR_TIMEOUT
    after = run()                                    # the hook was consumed by that launch
    assert ops.device_status(reset=True) == 0
    for x, y in zip(before, after):
        assert torch.equal(x, y)


# the first step (no MMA issued), one in the first round of the ring, one past it
@pytest.mark.parametrize("skip_kb", [0, 3, 9])
@pytest.mark.parametrize("kind", ["bf16", "fp8", "f16x3", "blocks"])
def test_pair_wait_runs_out(ops, kind, skip_kb):
    if kind == "bf16":           # K > 2560: on pairs
        A, B = _bf16(700, 4096, 1), _bf16(513, 4096, 2)
        _runs_out(ops, skip_kb, lambda: [ops.gemm_bf16(A, B)])
    elif kind == "fp8":          # 77 one-CTA tiles: past the shared ones
        (A, sa), (B, sb) = _fp8(1300, 2048, 3), _fp8(1500, 2048, 4)
        p = ops.plan(2048, 1024, 2, 0, 0)
        _runs_out(ops, skip_kb, lambda: [ops.gemm_masked(p, A, B, 0b11, a_scales=sa, b_scales=sb)])
    elif kind == "f16x3":
        g = torch.Generator(device="cuda")
        g.manual_seed(5)
        A = torch.randn((4096, 8192), generator=g, device="cuda")
        B = torch.randn((8192, 4000), generator=g, device="cuda")
        p = ops.plan(8192, 2048, 2, 0, 1)
        assert not torch.equal(ops.matmul(p, A, B, 0b11, "f32"), ops.matmul(p, A, B, 0b11, "tf32x2"))
        _runs_out(ops, skip_kb, lambda: [ops.matmul(p, A, B, 0b11, "f32")])
    else:
        A, B = _bf16(512, 2048, 6), _bf16(512, 2048, 7)
        p = ops.plan(2048, 512, 3, 1, 0)
        masks = torch.tensor([[0b1011, 0b1101], [0b0111, 0b1110]], dtype=torch.int64, device="cuda")
        _runs_out(ops, skip_kb, lambda: [ops.gemm_masked_blocks(p, A, B, masks, 256, 256)])


@pytest.mark.parametrize("skip_kb", [0, 2])
def test_backward_wait_runs_out(ops, skip_kb):
    """The first of the backward pass's two MN-major products is the one that gives up."""
    m, l, b = 256, 512, 128
    p = ops.plan(3000, b, 3, 1, 0)
    At, BtT = _bf16(m, p.z, 8), _bf16(l, p.z, 9)
    dC = _bf16(m, l, 10).float()
    _runs_out(ops, skip_kb, lambda: list(ops.matmul_backward(p, At, BtT, dC, 0b1011, torch.float32, torch.float32)))


@pytest.mark.parametrize("skip_kb", [0, 5])
@pytest.mark.parametrize("kind", ["tf32x2", "fp8"])
def test_shared_tile_wait_runs_out(ops, kind, skip_kb):
    """A lone tile whose K steps are dealt to a cluster: its first CTA gives up."""
    p = ops.plan(4096, 1024, 4, 0, 0)
    if kind == "fp8":
        skip_kb = min(skip_kb, 3)        # of 32 steps of 128, four per CTA of eight
        (A, sa), (B, sb) = _fp8(128, p.z, 11), _fp8(200, p.z, 12)
        run = lambda: [ops.gemm_masked(p, A, B, 0b1111, a_scales=sa, b_scales=sb)]
    else:
        g = torch.Generator(device="cuda")
        g.manual_seed(13)
        X = torch.randn((2, 128, p.z), generator=g, device="cuda")
        hi = (X.view(torch.int32) & -8192).view(torch.float32)   # TF32 planes: hi in [0], lo behind it
        A, B = torch.stack((hi[0], X[0] - hi[0])), torch.stack((hi[1], X[1] - hi[1]))
        run = lambda: [ops.gemm_masked(p, A[0], B[0], 0b1111, dtype="tf32x2")]
    _runs_out(ops, skip_kb, run)
