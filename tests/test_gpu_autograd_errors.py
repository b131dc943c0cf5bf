"""Operands the layer refuses raise OverSketchError, as the sketches it calls do."""
import pytest

from helpers import gpu_lib

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("kind", ["g_vector", "x_vector", "x_scalar", "g_columns", "x_columns", "g_host", "x_host"])
def test_refused_operands(kind, recompute):
    ops = gpu_lib()
    from paper_1811_02653_gb300.autograd import oversketch_matmul
    p = ops.plan(512, 64, 3, 1, 0)
    X, G = torch.randn((64, 512), device="cuda"), torch.randn((512, 96), device="cuda")
    if kind == "g_vector":
        G = G[:, 0].contiguous()
    elif kind == "x_vector":
        X = X[0]
    elif kind == "x_scalar":
        X = X[0, 0]
    elif kind == "g_columns":
        G = G.t().contiguous().t()
    elif kind == "x_columns":
        X = X.t().contiguous().t()
    elif kind == "g_host":
        G = G.cpu()
    else:
        X = X.cpu()
    with pytest.raises(ops.OverSketchError):
        oversketch_matmul(X, G, p, 0b1011, recompute=recompute)
