"""The work that users have this framework do, as cases that can be timed and compared.

A case is a dict of plain values; `prepare` makes its inputs, plan and workspace,
`run` is one pass through the public entry points, `work` the bytes and operations
that pass cannot do without, and `exact` the same outputs from FP64 torch.

The kinds of a case:

* ``matmul``  -- one product (A S)(S^T B)/k of dense operands on the device: a
                 single call, with the plan and the workspace kept, as in a loop over products.
* ``gram``    -- the symmetric product A D A^T of a sparse A stored dense (the normal
                 matrix of an interior-point method): one call, sketch of the nonzeros.
* ``batched`` -- many uneven products in one call, straggler masks on the device.
* ``train``   -- forward and backward of the product as a layer of a network:
                 C, dX and dG.
* ``newton``  -- the Hessian of one Newton iteration of the barrier LP solver, with
                 one straggler per block of the Hessian.
* ``blocks``  -- the accuracy experiment's product: both sketches, then the product
                 with its own kept sketch blocks for every block of C.
* ``host``    -- the product from and to pinned host memory.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1811_02653_gb300 import lp, ops
from paper_1811_02653_gb300.autograd import oversketch_matmul

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _mask(P, dropped):
    m = (1 << P) - 1
    for j in dropped:
        m &= ~(1 << j)
    return m


def listed():
    return [
        # the smallest product, all defaults (FP32 in, FP32 accuracy): launches and latency
        dict(name="small-f32", kind="matmul", m=512, n=4096, l=512, b=256, N=4, e=1, mask=_mask(5, [2]),
             gemm="f32", a="f32", bt="f32", spike=0),
        # an ordinary product of no round size: ragged tiles, rows of no 16-byte alignment
        dict(name="ragged-bf16", kind="matmul", m=2003, n=20011, l=1777, b=640, N=6, e=2, mask=_mask(8, [0, 5]),
             gemm="bf16", a="f32", bt="f32", spike=0),
        # the headline product: two 4.3 GB operands with a shared low-rank part
        dict(name="square-bf16", kind="matmul", m=16384, n=65536, l=16384, b=1024, N=8, e=2, mask=_mask(10, [1, 6]),
             gemm="bf16", a="f32", bt="f32", spike=64),
        # the same at half the size in the other two arithmetics a caller can choose:
        # FP32 accuracy (the default) and FP8 with block scales
        dict(name="square-f32", kind="matmul", m=8192, n=32768, l=8192, b=1024, N=8, e=2, mask=_mask(10, [1, 6]),
             gemm="f32", a="f32", bt="f32", spike=64),
        dict(name="square-fp8", kind="matmul", m=8192, n=32768, l=8192, b=1024, N=8, e=2, mask=_mask(10, [1, 6]),
             gemm="fp8", a="f32", bt="f32", spike=64),
        # the interior-point normal matrix: a 1 % dense constraint matrix of 17 GB
        dict(name="gram-sparse", kind="gram", m=4096, n=1048576, b=4096, N=6, e=1, mask=_mask(7, [3]),
             gemm="bf16", a="f32", density=0.01),
        # many products of uneven sizes at once
        dict(name="batched", kind="batched", count=16, m_lo=256, m_hi=4096, n_lo=8192, n_hi=131072, N=4, e=1, a="f32"),
        # a layer's training step in BF16, the size of the autograd workload
        dict(name="train-bf16", kind="train", m=4096, n=65536, l=4096, b=2048, N=4, e=1, mask=_mask(5, [2]),
             a="bf16", bt="bf16", recompute=False),
        # a small layer's training step in FP32, odd width, sketches recomputed in backward
        dict(name="train-f32", kind="train", m=1024, n=16384, l=1501, b=512, N=4, e=1, mask=_mask(5, [4]),
             a="f32", bt="f32", recompute=True),
        # one Newton iteration's Hessian at the paper's proportions (n = 40 b, m = 5 b, z = 20 b)
        dict(name="newton-hessian", kind="newton", n=40960, m=5120, b=1024, N=19, e=1),
        # the accuracy experiment (m = l = 10 b, n = 60 b, z = 30 b, 4 stragglers per block of C)
        dict(name="blocks-study", kind="blocks", m=5120, n=30720, l=5120, b=512, N=26, e=4),
        # a product of host buffers: what a caller without device tensors pays
        dict(name="host-bf16", kind="host", m=4096, n=16384, l=4096, b=512, N=4, e=1, mask=_mask(5, [1]),
             gemm="bf16", a="f32", bt="f32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _blocks(rng, n, lo_k, hi_k, unit):
    """A block width (a multiple of `unit`, between n/64 and n/16), the numbers of
    blocks and a mask that drops e of them."""
    b = max(unit, _log(rng, max(unit, n // 64), max(unit, n // 16)) // unit * unit)
    N, e = rng.randint(lo_k, hi_k), rng.randint(0, 2)
    return b, N, e, _mask(N + e, rng.sample(range(N + e), e))


def draw(rng: random.Random):
    kind = rng.choice(["matmul", "matmul", "matmul", "train", "train", "gram", "batched", "newton", "blocks", "host"])
    if kind == "matmul":
        gemm = rng.choice(["f32", "f32", "bf16", "bf16", "fp8"])
        m, n, l = _log(rng, 300, 12288), _log(rng, 4096, 65536), _log(rng, 300, 12288)
        if rng.random() < 0.5:
            m, n, l = max(256, m // 128 * 128), n // 1024 * 1024, max(256, l // 128 * 128)
        b, N, e, mask = _blocks(rng, n, 2, 8, {"f32": 32, "bf16": 64, "fp8": 128}[gemm])
        return dict(kind=kind, m=m, n=n, l=l, b=b, N=N, e=e, mask=mask, gemm=gemm, a=rng.choice(["f32", "f32", "bf16"]),
                    bt=rng.choice(["f32", "f32", "bf16"]), spike=rng.choice([0, 64]))
    if kind == "train":
        m, n, l = _log(rng, 256, 4096), _log(rng, 4096, 65536), _log(rng, 256, 4096)
        if rng.random() < 0.6:
            m, l = max(256, m // 64 * 64), max(256, l // 64 * 64)
        b, N, e, mask = _blocks(rng, n, 2, 5, 64)
        dt = rng.choice(["f32", "bf16"])
        return dict(kind=kind, m=m, n=n, l=l, b=b, N=N, e=e, mask=mask, a=dt, bt=dt, recompute=rng.random() < 0.3)
    if kind == "gram":
        m, n = _log(rng, 256, 4096), _log(rng, 65536, 1048576)
        N, e = rng.randint(3, 6), rng.randint(0, 1)
        return dict(kind=kind, m=m, n=n, b=128 * _log(rng, 4, 32), N=N, e=e,
                    mask=_mask(N + e, rng.sample(range(N + e), e)), gemm=rng.choice(["f32", "bf16", "bf16"]), a="f32",
                    density=math.exp(rng.uniform(math.log(0.002), math.log(0.02))))
    if kind == "batched":
        return dict(kind=kind, count=rng.randint(2, 14), m_lo=256, m_hi=_log(rng, 512, 4096), n_lo=8192,
                    n_hi=_log(rng, 16384, 131072), N=4, e=1, a=rng.choice(["f32", "f32", "bf16"]))
    if kind == "newton":
        b = 256 * rng.randint(1, 4)
        return dict(kind=kind, n=b * rng.randint(16, 40), m=b * rng.randint(2, 5), b=b, N=rng.randint(8, 19), e=rng.randint(0, 1))
    if kind == "blocks":
        b = 256 * rng.randint(1, 2)
        return dict(kind=kind, m=b * rng.randint(4, 10), n=b * rng.randint(30, 60), l=b * rng.randint(4, 10), b=b,
                    N=rng.randint(10, 26), e=rng.randint(1, 4))
    m, n, l = _log(rng, 512, 4096), _log(rng, 4096, 16384), _log(rng, 512, 4096)
    b, N, e, mask = _blocks(rng, n, 2, 6, 64)
    return dict(kind="host", m=m, n=n, l=l, b=b, N=N, e=e, mask=mask, gemm="bf16", a="f32", bt="f32")


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + 17)
    return g


def _hash_seed(seed, p=0):
    return (seed * 7919 + p) % (1 << 31)


def _randn(g, rows, cols, dtype=torch.float32, std=1.0):
    x = torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float32)
    if std != 1.0:
        x.mul_(std)
    return x if dtype is torch.float32 else x.to(dtype)


def _operands(c, seed):
    """A and B of a dense product: N(0, 1), with a shared rank-`spike` part of scale 10."""
    g = _gen(seed)
    A, B = _randn(g, c["m"], c["n"]), _randn(g, c["n"], c["l"])
    if c.get("spike"):
        r = c["spike"]
        U, V, W = _randn(g, c["m"], r), _randn(g, c["n"], r), _randn(g, c["l"], r)
        s = 10.0 / math.sqrt(r)
        A.addmm_(U, V.t(), alpha=s)
        B.addmm_(V, W.t(), alpha=s)
    return A.to(DTYPES[c["a"]]), B.to(DTYPES[c["bt"]])


def _sparse(c, seed):
    """A of Bernoulli(density) N(0, 1) entries stored dense, and sqrt(D), D = 10^U(-6, 6)."""
    g = _gen(seed)
    A = torch.empty((c["m"], c["n"]), dtype=torch.float32, device="cuda")
    step = max(1, (1 << 28) // c["n"])
    for r in range(0, c["m"], step):
        part = A[r:r + step]
        part.normal_(generator=g)
        part.mul_(torch.rand(part.shape, generator=g, device="cuda") < c["density"])
    d = torch.pow(10.0, torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64) * 12.0 - 6.0)
    return A, d.sqrt().float()


def _batch_shapes(c):
    """m, l uniform, n log-uniform in multiples of 2048, b = n / 32 (the batch of the workloads)."""
    rng = random.Random(1000 * c["count"] + c["n_hi"])
    out = []
    for _ in range(c["count"]):
        m, l = rng.randint(c["m_lo"], c["m_hi"]), rng.randint(c["m_lo"], c["m_hi"])
        n = int(round(math.exp(rng.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]))) / 2048)) * 2048
        out.append((m, min(max(n, 8192), 131072), l))
    return out


def _block_masks(rows, cols, P, e, seed):
    """int64 kept-block masks, e of P bits cleared at independent places per block."""
    r = np.random.default_rng([seed, P, e])
    out = np.empty((rows, cols), dtype=np.int64)
    for i in range(rows):
        for j in range(cols):
            out[i, j] = _mask(P, r.choice(P, size=e, replace=False).tolist())
    return out


def _newton_inputs(c, seed):
    """The LP's data (A of N(0, 1/m)) and a point's slacks, which span a few decades."""
    g = _gen(seed)
    A = _randn(g, c["n"], c["m"], std=1.0 / math.sqrt(c["m"]))
    s = torch.pow(10.0, torch.rand(c["n"], generator=g, device="cuda", dtype=torch.float64) * 3.0 - 2.5)
    nb = (c["m"] + c["b"] - 1) // c["b"]
    return A, s, _block_masks(nb, nb, c["N"] + c["e"], c["e"], seed)


def prepare(case, seed):
    c, k = case, case["kind"]
    if k == "batched":
        g = _gen(seed)
        shapes, dt = _batch_shapes(c), DTYPES[c["a"]]
        st = dict(case=c, plans=[ops.plan(n, n // 32, c["N"], c["e"], _hash_seed(seed, p)) for p, (m, n, l) in enumerate(shapes)],
                  A=[], B=[], C=[])
        for m, n, l in shapes:
            st["A"].append(_randn(g, m, n, dt))
            st["B"].append(_randn(g, n, l, dt))
            st["C"].append(torch.empty((m, l), dtype=torch.float32, device="cuda"))
        P = c["N"] + c["e"]
        st["masks"] = torch.tensor([_mask(P, [p % P]) for p in range(c["count"])], dtype=torch.int64, device="cuda")
        ms, ns, ls = zip(*shapes)
        st["ws"] = torch.empty(ops.matmul_batched_workspace(st["plans"], ms, ns, ls, dt, dt), dtype=torch.uint8, device="cuda")
        return st
    if k == "newton":
        A, s, masks = _newton_inputs(c, seed)
        g = torch.Generator()
        g.manual_seed(seed)
        bvec = 1.0 + torch.randn(c["n"], generator=g, dtype=torch.float64).abs()
        cvec = torch.randn(c["m"], generator=g, dtype=torch.float64)
        solver = lp.SketchedBarrierLP(A, bvec, cvec, blk=c["b"], N=c["N"], e=c["e"], seed=_hash_seed(seed))
        return dict(case=c, solver=solver, s=s, masks=masks)
    plan = ops.plan(c["n"], c["b"], c["N"], c["e"], _hash_seed(seed))
    st = dict(case=c, plan=plan)
    if k == "gram":
        st["A"], st["d"] = _sparse(c, seed)
        st["ws"] = torch.empty(ops.workspace_size(plan, c["m"], c["m"], torch.float32, c["gemm"], symmetric=True),
                               dtype=torch.uint8, device="cuda")
        return st
    if k == "blocks":
        # A(x, y) = x + y with B = A^T, shifted by the seed; integers, exact in FP32
        x = torch.arange(1, c["m"] + 1, device="cuda", dtype=torch.float32) + (seed % 64)
        y = torch.arange(1, c["n"] + 1, device="cuda", dtype=torch.float32)
        st["A"] = x[:, None] + y[None, :]
        st["B"] = (y[:, None] + (torch.arange(1, c["l"] + 1, device="cuda", dtype=torch.float32) + (seed % 64))[None, :])
        nb = lambda q: (q + c["b"] - 1) // c["b"]
        st["masks"] = torch.from_numpy(_block_masks(nb(c["m"]), nb(c["l"]), c["N"] + c["e"], c["e"], seed)).cuda()
        return st
    if k == "train":
        g = _gen(seed)
        dt = DTYPES[c["a"]]
        st["X"] = _randn(g, c["m"], c["n"], dt, 0.02).requires_grad_()
        st["G"] = _randn(g, c["n"], c["l"], dt, 0.02).requires_grad_()
        st["dC"] = _randn(g, c["m"], c["l"])
        return st
    A, B = _operands(c, seed)
    if k == "host":
        st["A"] = torch.empty(A.shape, dtype=A.dtype, pin_memory=True).copy_(A)
        st["B"] = torch.empty(B.shape, dtype=B.dtype, pin_memory=True).copy_(B)
        st["C"] = torch.empty((c["m"], c["l"]), dtype=torch.float32, pin_memory=True)
        st["ws"] = torch.empty(ops.matmul_host_workspace(plan, c["m"], c["l"], A.dtype, B.dtype, c["gemm"]),
                               dtype=torch.uint8, device="cuda")
        return st
    st["A"], st["B"] = A, B
    st["ws"] = torch.empty(ops.workspace_size(plan, c["m"], c["l"], A.dtype, c["gemm"], b_dtype=B.dtype),
                           dtype=torch.uint8, device="cuda")
    return st


# ---------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "matmul":
        return ops.matmul(state["plan"], state["A"], state["B"], c["mask"], c["gemm"], workspace=state["ws"])
    if k == "gram":
        return ops.matmul(state["plan"], state["A"], None, c["mask"], c["gemm"], col_scale=state["d"], symmetric=True,
                          workspace=state["ws"], sparse_a=True)
    if k == "batched":
        return ops.matmul_batched(state["plans"], state["A"], state["B"], state["C"], state["masks"], state["ws"])
    if k == "train":
        C = oversketch_matmul(state["X"], state["G"], state["plan"], c["mask"], c["recompute"])
        dX, dG = torch.autograd.grad(C, (state["X"], state["G"]), state["dC"])
        return [C.detach(), dX, dG]
    if k == "newton":
        return state["solver"].hessian(state["s"], state["masks"])
    if k == "blocks":
        At, _ = ops.sketch_left(state["plan"], state["A"], "bf16")
        BtT, _ = ops.sketch_right(state["plan"], state["B"], "bf16")
        return ops.gemm_masked_blocks(state["plan"], At, BtT, state["masks"], c["b"], c["b"])
    return ops.matmul_host(state["plan"], state["A"], state["B"], c["mask"], c["gemm"], C=state["C"], workspace=state["ws"])


# ---------------------------------------------------------------- what a pass cannot do without

def _product_work(m, n, l, b, k, ea, eb, density=1.0):
    """Operands read once, C written once; one signed addition per element and kept
    block, and the product of the sketches."""
    return m * n * ea + n * l * eb + 4 * m * l, density * k * n * (m + l) + 2.0 * m * k * b * l


def work(case):
    c, k = case, case["kind"]
    size = {"f32": 4, "bf16": 2}
    if k == "batched":
        by = fl = 0
        for m, n, l in _batch_shapes(c):
            x, y = _product_work(m, n, l, n // 32, c["N"], size[c["a"]], size[c["a"]])
            by, fl = by + x, fl + y
        return {"bytes": by, "flops": fl}
    if k == "newton":
        return {"bytes": 4 * (c["n"] * c["m"] + c["m"] ** 2) + 8 * c["n"],
                "flops": (c["N"] + c["e"]) * c["n"] * c["m"] + 2.0 * c["m"] ** 2 * c["N"] * c["b"]}
    if k == "blocks":
        by, _ = _product_work(c["m"], c["n"], c["l"], c["b"], c["N"], 4, 4)
        return {"bytes": by, "flops": (c["N"] + c["e"]) * c["n"] * (c["m"] + c["l"]) + 2.0 * c["m"] * c["l"] * c["N"] * c["b"]}
    kept = bin(c["mask"]).count("1")
    if k == "gram":
        m, n = c["m"], c["n"]
        return {"bytes": 4 * (m * n + n + m * m), "flops": 2 * c["density"] * kept * m * n + 1.0 * m * (m + 1) * kept * c["b"]}
    m, n, l = c["m"], c["n"], c["l"]
    by, fl = _product_work(m, n, l, c["b"], kept, size[c["a"]], size[c["bt"]])
    if k == "train":
        by += 4 * m * l + n * (m + l) * size[c["a"]]
        fl += kept * n * (m + l) + 4.0 * m * kept * c["b"] * l
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- the same in FP64

def _mix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _tables(n, b, P, seed):
    """Buckets (int64) and signs (FP64) of the P blocks, on the device."""
    gamma = np.uint64(0x9E3779B97F4A7C15)
    i = np.arange(1, n + 1, dtype=np.uint64) * gamma
    h, s = [], []
    with np.errstate(over="ignore"):
        for j in range(P):
            key = _mix(np.uint64(seed) + np.uint64(j + 1) * gamma)
            w = _mix(key + i)
            h.append((((w >> np.uint64(32)) * np.uint64(b)) >> np.uint64(32)).astype(np.int64))
            s.append(1.0 - 2.0 * (w & np.uint64(1)).astype(np.float64))
    return [torch.from_numpy(x).cuda() for x in h], [torch.from_numpy(x).cuda() for x in s]


def _sketch_cols(A, h, s, blocks, b, scale=None):
    """A diag(scale) S over the listed blocks, m x (len(blocks) b), FP64."""
    out = torch.zeros((A.shape[0], len(blocks) * b), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // A.shape[1])
    for r in range(0, A.shape[0], step):
        x = A[r:r + step].double()
        if scale is not None:
            x *= scale
        for t, j in enumerate(blocks):
            out[r:r + step, t * b:(t + 1) * b].index_add_(1, h[j], x * s[j])
    return out


def _sketch_rows(B, h, s, blocks, b):
    """S^T B over the listed blocks, (len(blocks) b) x l, FP64."""
    out = torch.zeros((len(blocks) * b, B.shape[1]), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // B.shape[1])
    for i in range(0, B.shape[0], step):
        x = B[i:i + step].double()
        for t, j in enumerate(blocks):
            out[t * b:(t + 1) * b].index_add_(0, h[j][i:i + step], x * s[j][i:i + step, None])
    return out


def _bits(mask):
    return [j for j in range(64) if (int(mask) >> j) & 1]


def _exact_product(A, B, n, b, P, seed, mask):
    h, s = _tables(n, b, P, seed)
    bl = _bits(mask)
    return _sketch_cols(A, h, s, bl, b) @ _sketch_rows(B, h, s, bl, b) / len(bl)


def _exact_blocks(At, Bt, masks, bs, b):
    """C with each bs x bs block summing its own kept blocks (At: m x z, Bt: z x l)."""
    C = torch.zeros((At.shape[0], Bt.shape[1]), dtype=torch.float64, device="cuda")
    for i in range(masks.shape[0]):
        for j in range(masks.shape[1]):
            bl = _bits(masks[i, j])
            idx = torch.cat([torch.arange(t * b, (t + 1) * b, device="cuda") for t in bl])
            C[i * bs:(i + 1) * bs, j * bs:(j + 1) * bs] = At[i * bs:(i + 1) * bs][:, idx] @ Bt[idx][:, j * bs:(j + 1) * bs] / len(bl)
    return C


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "batched":
        g, P, out = _gen(seed), c["N"] + c["e"], []
        for p, (m, n, l) in enumerate(_batch_shapes(c)):
            A, B = _randn(g, m, n, DTYPES[c["a"]]), _randn(g, n, l, DTYPES[c["a"]])
            out.append(_exact_product(A, B, n, n // 32, P, _hash_seed(seed, p), _mask(P, [p % P])))
        return out
    P = c["N"] + c["e"]
    if k == "newton":
        A, s, masks = _newton_inputs(c, seed)
        h, sg = _tables(c["n"], c["b"], P, _hash_seed(seed))
        Bt = _sketch_rows(A.double() / s[:, None], h, sg, range(P), c["b"])
        return _exact_blocks(Bt.t().contiguous(), Bt, masks, c["b"], c["b"])
    h, sg = _tables(c["n"], c["b"], P, _hash_seed(seed))
    if k == "gram":
        A, d = _sparse(c, seed)
        bl = _bits(c["mask"])
        At = torch.zeros(c["m"] * len(bl) * c["b"], dtype=torch.float64, device="cuda")
        step = max(1, (1 << 28) // c["n"])
        for r in range(0, c["m"], step):
            row, col = torch.nonzero(A[r:r + step], as_tuple=True)
            v = A[r:r + step][row, col].double() * d[col].double()
            for t, j in enumerate(bl):
                At.index_add_(0, (row + r) * (len(bl) * c["b"]) + t * c["b"] + h[j][col], v * sg[j][col])
        At = At.view(c["m"], -1)
        return At @ At.t() / len(bl)
    if k == "blocks":
        st = prepare(case, seed)
        At, Bt = _sketch_cols(st["A"], h, sg, range(P), c["b"]), _sketch_rows(st["B"], h, sg, range(P), c["b"])
        return _exact_blocks(At, Bt, st["masks"].cpu().numpy(), c["b"], c["b"])
    bl = _bits(c["mask"])
    if k == "train":
        g = _gen(seed)
        X, G = _randn(g, c["m"], c["n"], DTYPES[c["a"]], 0.02), _randn(g, c["n"], c["l"], DTYPES[c["a"]], 0.02)
        dC = _randn(g, c["m"], c["l"]).double()
        At, Bt = _sketch_cols(X, h, sg, bl, c["b"]), _sketch_rows(G, h, sg, bl, c["b"])
        T, U = dC @ Bt.t() / len(bl), At.t() @ dC / len(bl)
        dX = torch.zeros((c["m"], c["n"]), dtype=torch.float64, device="cuda")
        dG = torch.zeros((c["n"], c["l"]), dtype=torch.float64, device="cuda")
        for t, j in enumerate(bl):
            dX += T[:, t * c["b"]:(t + 1) * c["b"]][:, h[j]] * sg[j]
            dG += U[t * c["b"]:(t + 1) * c["b"]][h[j]] * sg[j][:, None]
        return [At @ Bt / len(bl), dX, dG]
    A, B = _operands(c, seed)
    C = _sketch_cols(A, h, sg, bl, c["b"]) @ _sketch_rows(B, h, sg, bl, c["b"]) / len(bl)
    return C.cpu() if k == "host" else C
