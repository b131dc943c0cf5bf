"""dX of very many rows: more strips than one launch's grid holds, and more rows than the
gather from T^T addresses (these go through T)."""
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,l,n,b,N,xd", [
    (65535 * 128, 8, 70, 128, 1, "bfloat16"),          # the last that fits one launch (MN-major)
    (65535 * 128 + 1, 8, 70, 128, 1, "bfloat16"),
    (65535 * 128 * 2 + 77, 3, 5, 2, 2, "float32"),
    (2 ** 30 - 4, 1, 3, 2, 2, "bfloat16"),             # the last pitch of T^T
    (2 ** 30, 1, 3, 2, 2, "bfloat16"),
])
def test_tall_dx(m, l, n, b, N, xd):
    ops = gpu_lib()
    p = ops.plan(n, b, N, 0, 4)
    mask = (1 << N) - 1
    g = torch.Generator(device="cuda")
    g.manual_seed(m % 1000)
    BtT = torch.randn((l, p.z), generator=g, device="cuda").to(torch.bfloat16)
    dC = torch.randn((m, l), generator=g, device="cuda")
    dX, dG = ops.matmul_backward(p, None, BtT, dC, mask, getattr(torch, xd), torch.float32, need_dg=False)
    assert dG is None
    # the adjoint at sampled rows, at both ends and around the launches' edges
    rows = torch.randint(0, m, (2000,), generator=g, device="cuda")
    edge = torch.tensor([r for q in (0, 65535 * 128, 2 * 65535 * 128, m) for r in range(q - 130, q + 130) if 0 <= r < m],
                        device="cuda")
    rows = torch.cat((rows, edge))
    h, s, _, _ = p.tables()
    S = torch.zeros((p.z, n), dtype=torch.float64, device="cuda")
    i = torch.arange(n, device="cuda")
    for j in range(N):
        S[torch.from_numpy(h[j].astype("int64")).cuda() + j * b, i] = torch.from_numpy(s[j].astype("float64")).cuda()
    d = dC[rows].to(torch.bfloat16).double()
    ref, mag = d @ (BtT.double() @ S) / N, d.abs() @ (BtT.double().abs() @ S.abs()) / N
    # l + N FP32 roundings (2^-23: the accumulation truncates) and one to the output
    bound = (l + N + 1) * 2.0 ** -23 * mag + (2.0 ** -8 if xd == "bfloat16" else 0.0) * ref.abs() + 1e-30
    assert bool(((dX[rows].double() - ref).abs() <= bound).all())
    assert ops.device_status() == 0
    del dX, dC
    torch.cuda.empty_cache()
