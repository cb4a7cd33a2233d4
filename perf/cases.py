"""What a program that uses this framework has it do, as measurable cases.

A case is a dict of plain values; its "kind" says which entry points a pass goes through:

* ``c2c``: ``Plan.forward`` then ``Plan.inverse`` of a complex array (the step of a spectral solver);
* ``r2c``: forward, complex-to-real inverse, forward again (the inverse uses its input as scratch,
  so a program that wants the spectrum afterwards transforms the field again);
* ``loss``: the spectral-weight loss and its gradient through ``torch.autograd``;
* ``batch``: one direction of many independent transforms replayed from one CUDA graph;
* ``exchange``: the global redistributions alone, from stage 0 through every stage to the last.

Arrays live on the GPU as stage buffers (every virtual rank's block, concatenated in rank order).
Plans, workspaces, output buffers and the batch's graph are made once, as a program's set-up does.
"""
from __future__ import annotations

import itertools
import math

import torch

from paper_1804_09536_gb300 import inputs
from paper_1804_09536_gb300.autograd import spectral_weight_loss
from paper_1804_09536_gb300.plan import Batch, Plan

DEV = "cuda"


def listed():
    return [
        # the smallest transform in use: a 32^3 box on a 2 x 2 pencil grid (launches and latency)
        {"name": "c2c 32^3", "kind": "c2c", "shape": "32 32 32", "grid": "2 2", "precision": "fp32"},
        # an ordinary small mesh, everything in L2
        {"name": "c2c 128^3", "kind": "c2c", "shape": "128 128 128", "grid": "2 4", "precision": "fp32"},
        # a mesh of ordinary 2/3/5 lengths, not powers of two, on a grid that does not divide it
        {"name": "c2c 180x200x240", "kind": "c2c", "shape": "180 200 240", "grid": "3 4", "precision": "fp32"},
        # the paper's own example mesh: 42 and 127 have no 2/3/5 factorisation, uneven blocks
        {"name": "c2c 42x127x256", "kind": "c2c", "shape": "42 127 256", "grid": "3 4", "precision": "fp32"},
        # the headline: a DNS-style mesh on a pencil grid, far larger than L2
        {"name": "c2c 512^3", "kind": "c2c", "shape": "512 512 512", "grid": "4 8", "precision": "fp32"},
        # the same kind of mesh through the tensor-core mode (lengths 256 and 512)
        {"name": "c2c 256x512x512 bf16x3", "kind": "c2c", "shape": "256 512 512", "grid": "4 8", "precision": "bf16x3"},
        # four dimensions on a three-dimensional grid; the largest arrays
        {"name": "c2c 128^4", "kind": "c2c", "shape": "128 128 128 128", "grid": "4 4 2", "precision": "fp32"},
        # a real field on slabs (odd Hermitian half, about the size of L2)
        {"name": "r2c 256^3 slab", "kind": "r2c", "shape": "256 256 256", "grid": "8", "precision": "fp32"},
        # a real DNS field on pencils
        {"name": "r2c 512^3", "kind": "r2c", "shape": "512 512 512", "grid": "4 8", "precision": "fp32"},
        # forward and backward of the differentiable loss
        {"name": "loss 512^3", "kind": "loss", "shape": "512 512 512", "grid": "4 8", "precision": "fp32"},
        # 48 transforms of mixed shapes and grids in one graph
        {"name": "batch of 48", "kind": "batch", "count": 48, "seed": 0, "sign": -1},
        # the redistributions of a real field's half spectrum alone (rows of 257 complex)
        {"name": "exchange 512^3 half", "kind": "exchange", "shape": "512 512 512", "grid": "4 8", "real": True},
    ]


def _smooth(n):
    for f in (2, 3, 5):
        while n % f == 0:
            n //= f
    return n == 1


_POWERS = (32, 64, 128, 256, 512)
_SMOOTH = tuple(n for n in range(24, 513) if _smooth(n))
_ANY = tuple(range(24, 513))
# innermost real lengths: twice a length with compiled real-line passes
_REAL = (64, 96, 120, 128, 160, 192, 240, 256, 320, 384, 480, 512, 640, 768)
_MOST = 1 << 27  # elements of a drawn array (the largest listed one has 1 << 28)


def _length(rng, pool):
    """One of a pool of lengths, spread over its logarithm."""
    t = math.exp(rng.uniform(math.log(pool[0]), math.log(pool[-1])))
    return min(pool, key=lambda n: abs(n - t))


def _grid(rng, g):
    return [rng.choice((1, 2, 3, 4, 8)) for _ in range(g)]


def draw(rng):
    kind = rng.choice(("c2c", "c2c", "c2c", "r2c", "r2c", "loss", "batch", "exchange"))
    if kind == "batch":
        return {"kind": kind, "count": round(math.exp(rng.uniform(math.log(4), math.log(40)))),
                "seed": rng.randrange(1, 1 << 20), "sign": rng.choice((-1, 1))}
    d = 4 if kind == "c2c" and rng.random() < 0.2 else 3
    g = 3 if d == 4 else rng.choice((1, 2, 2))
    precision = rng.choice(("fp32", "fp32", "fp32", "bf16x3", "fp16x3")) if kind == "c2c" and d == 3 else "fp32"
    pool = rng.choice((_POWERS, _SMOOTH, _SMOOTH, _ANY)) if precision == "fp32" else (256, 512)
    while True:
        shape = [_length(rng, tuple(n for n in pool if d == 3 or n <= 128)) for _ in range(d)]
        if kind == "r2c":
            shape[-1] = _length(rng, _REAL)
        if math.prod(shape) <= (_MOST if pool != _ANY else _MOST >> 2):
            break
    c = {"kind": kind, "shape": " ".join(map(str, shape)), "grid": " ".join(map(str, _grid(rng, g)))}
    if kind == "exchange":
        c["real"] = shape[-1] % 2 == 0 and rng.random() < 0.5
    else:
        c["precision"] = precision
    return c


# ------------------------------------------------------------ arrays and stage buffers

def _ints(text):
    return tuple(int(v) for v in text.split())


def _normal(shape, seed, complex_):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    x = torch.randn(*shape, *((2,) if complex_ else ()), generator=g, device=DEV)
    return torch.view_as_complex(x) if complex_ else x


def _weight(n, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + (1 << 40))
    return torch.rand(n, generator=g, device=DEV)


def _blocks(shape, grid, stage):
    """Every rank's block (slices) of a stage, in rank order: grid direction i cuts axis i before
    the exchanges have moved it to axis i + 1, in balanced contiguous parts."""
    g = len(grid)
    axis = [i if i < g - stage else i + 1 for i in range(g)]
    for rank in itertools.product(*(range(m) for m in grid)):
        cut = [slice(0, n) for n in shape]
        for i, p in enumerate(rank):
            q, r = divmod(shape[axis[i]], grid[i])
            s = q * p + min(r, p)
            cut[axis[i]] = slice(s, s + q + (p < r))
        yield tuple(cut)


def _to_stage(x, grid, stage):
    return torch.cat([x[b].reshape(-1) for b in _blocks(tuple(x.shape), grid, stage)])


def _from_stage(buf, shape, grid, stage):
    x = torch.empty(shape, dtype=buf.dtype, device=buf.device)
    at = 0
    for b in _blocks(shape, grid, stage):
        n = math.prod(max(0, s.stop - s.start) for s in b)
        x[b] = buf[at:at + n].reshape(x[b].shape)
        at += n
    return x


def _half(shape):
    return shape[:-1] + (shape[-1] // 2 + 1,)


# ------------------------------------------------------------ prepare, run

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        problems = inputs.batch_problems(case["count"], case["seed"])
        plans = [Plan(shape, grid, device=DEV) for shape, grid in problems]
        sign = case["sign"]
        stage = (lambda p: 0) if sign < 0 else (lambda p: p.g)
        ins = [_to_stage(_normal(p.shape, seed * 64 + k, True), p.grid, stage(p)) for k, p in enumerate(plans)]
        batch = Batch(plans, sign=sign, ins=ins)
        batch.set_executor("streams", 4)
        return {"kind": kind, "batch": batch, "graph": batch.graph()}
    shape, grid = _ints(case["shape"]), _ints(case["grid"])
    if kind == "exchange":
        plan = Plan(shape, grid, kind="r2c" if case["real"] else "c2c", device=DEV)
        x = _to_stage(_normal(_half(shape) if case["real"] else shape, seed, True), grid, 0)
        return {"kind": kind, "plan": plan, "x": x, "outs": [plan.empty_stage(s) for s in range(1, plan.g + 1)]}
    plan = Plan(shape, grid, kind="r2c" if kind == "r2c" else "c2c", device=DEV, precision=case["precision"])
    x = _to_stage(_normal(shape, seed, kind != "r2c"), grid, 0)
    if kind == "loss":
        return {"kind": kind, "plan": plan, "x": x.requires_grad_(True), "w": _weight(x.numel(), seed)}
    return {"kind": kind, "plan": plan, "x": x, "y": plan.empty_stage(plan.g),
            "back": plan.empty_stage(0, real=kind == "r2c")}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["graph"].replay()
        return state["batch"].outs
    plan, x = state["plan"], state["x"]
    if kind == "exchange":
        for k, out in enumerate(state["outs"]):
            plan.redistribute(plan.g - k, plan.g - k - 1, x, out)
            x = out
        return state["outs"]
    if kind == "loss":
        x.grad = None
        loss = spectral_weight_loss(x, state["w"], plan)
        loss.backward()
        # the scalar as a training log keeps it: its accuracy is that of the FP32 transform under it
        return loss.detach().float(), x.grad
    y, back = state["y"], state["back"]
    plan.forward(x, out=y)
    plan.inverse(y, out=back)
    if kind == "r2c":
        plan.forward(back, out=y)
    return y, back


# ------------------------------------------------------------ work, exact

def work(case):
    """Each call reads its input once and writes its output once; 5 n log2 n operations a transform."""
    kind = case["kind"]
    if kind == "batch":
        sizes = [math.prod(shape) for shape, _ in inputs.batch_problems(case["count"], case["seed"])]
        return {"bytes": sum(16 * n for n in sizes), "flops": sum(5 * n * math.log2(n) for n in sizes)}
    shape = _ints(case["shape"])
    n = math.prod(shape)
    if kind == "exchange":
        return {"bytes": len(_ints(case["grid"])) * 16 * (math.prod(_half(shape)) if case["real"] else n), "flops": 0}
    if kind == "r2c":  # half the complex work on half the data
        return {"bytes": 3 * (4 * n + 8 * math.prod(_half(shape))), "flops": 3 * 2.5 * n * math.log2(n)}
    if kind == "loss":  # x and the weights in, the gradient and the scalar out
        return {"bytes": 20 * n, "flops": 2 * 5 * n * math.log2(n) + 10 * n}
    return {"bytes": 32 * n, "flops": 2 * 5 * n * math.log2(n)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        outs = []
        for k, (shape, grid) in enumerate(inputs.batch_problems(case["count"], case["seed"])):
            x = _normal(shape, seed * 64 + k, True).to(torch.complex128)
            if case["sign"] < 0:
                outs.append(_to_stage(torch.fft.fftn(x, norm="forward"), grid, len(grid)))
            else:
                outs.append(_to_stage(torch.fft.ifftn(x, norm="forward"), grid, 0))
        return outs
    shape, grid = _ints(case["shape"]), _ints(case["grid"])
    g = len(grid)
    if kind == "exchange":
        x = _normal(_half(shape) if case["real"] else shape, seed, True).to(torch.complex128)
        return [_to_stage(x, grid, s) for s in range(1, g + 1)]
    if kind == "r2c":
        x = _normal(shape, seed, False).double()
        return _to_stage(torch.fft.rfftn(x, norm="forward"), grid, g), _to_stage(x, grid, 0)
    x = _normal(shape, seed, True).to(torch.complex128)
    y = torch.fft.fftn(x, norm="forward")
    if kind == "loss":
        w = _from_stage(_weight(x.numel(), seed), shape, grid, g).double()
        grad = 2 * torch.fft.ifftn(w * w * y)
        return (y * w).abs().square().sum(), _to_stage(grad, grid, 0)
    return _to_stage(y, grid, g), _to_stage(x, grid, 0)
