"""Performance cases of the stencil engine.

A case is what a program that uses this package runs again and again: a plan
(or a batch of grids) made once for one stencil and grid, and `steps` time
steps of a field on the GPU.  The listed cases are the workloads of bench.py
and of the tests with fewer steps (the 512^2 Jacobi grid, the 16384^2 and
10240^2 grids, the 512^3 set, the uneven batch) and ragged grids between
them; draw() spreads over the same stencils, sizes, types and precision forms.
"""
import math

import torch

from paper_2603_00477_gb300 import binding as B
from paper_2603_00477_gb300 import inputs

DEVICE = "cuda"


def _plan(name, shape, d, r, dims, dtype, steps, t=0, precision="native", path="auto", field="uniform",
          halo="zero"):
    case = {"kind": "plan", "shape": shape, "d": d, "r": r, "dtype": dtype, "steps": steps, "t": t,
            "precision": precision, "path": path, "field": field, "halo": halo}
    if name:
        case["name"] = name
    for i, n in enumerate(dims):
        case[f"n{i}"] = int(n)
    return case


def _batch(name, grids, lo, hi, steps, sizes_seed):
    case = {"kind": "batch", "grids": grids, "lo": lo, "hi": hi, "steps": steps, "dtype": "f32",
            "sizes_seed": sizes_seed}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # five-point Jacobi relaxation on a small FP64 grid: a handful of short
        # sweeps, launches and latency
        _plan("jacobi_f64_512", "star", 2, 1, (512, 512), "f64", 10),
        # a mid-sized FP32 grid with the fourth-order Laplacian's nine points,
        # odd extents, resident in L2, a non-zero boundary
        _plan("star2d2r_f32_1021x1531", "star", 2, 2, (1021, 1531), "f32", 20, halo="uniform"),
        # the flagship workload of bench.py: 7 x 7 weights, plain FP64 arithmetic
        _plan("box2d3r_f64_16384", "box", 2, 3, (16384, 16384), "f64", 6),
        # the same stencil at FP64 accuracy on the tensor cores (exact splitting)
        _plan("box2d3r_f64_split_10240", "box", 2, 3, (10240, 10240), "f64", 6, precision="ozaki"),
        # FP32 storage and FP32 arithmetic, smooth field: the plain form of the
        # precision study
        _plan("box2d2r_f32_16384", "box", 2, 2, (16384, 16384), "f32", 8, field="sine"),
        # the same grid, any operand form allowed: the fastest the engine offers
        _plan("box2d2r_any_16384", "box", 2, 2, (16384, 16384), "f32", 8, precision="any", field="sine"),
        # hi + lo FP16 operands (22 bits) on a ragged grid whose rows are no
        # 16-byte multiples, a non-zero boundary
        _plan("box2d2r_f16x3_7001x6007", "box", 2, 2, (7001, 6007), "f32", 8, precision="f16x3", field="sine",
              halo="uniform"),
        # TF32-class accuracy at the paper's domain and fusion depth
        _plan("box2d1r_tf32_10240_t7", "box", 2, 1, (10240, 10240), "f32", 14, t=7, precision="tf32"),
        # 3-D acoustic-style stencil, FP32, the usual power-of-two volume
        _plan("star3d2r_f32_512", "star", 3, 2, (512, 512, 512), "f32", 6),
        # 27 points, FP32, a ragged volume
        _plan("box3d1r_f32_301x417x533", "box", 3, 1, (301, 417, 533), "f32", 6, halo="uniform"),
        # 27 points, FP64
        _plan("box3d1r_f64_256", "box", 3, 1, (256, 256, 256), "f64", 6),
        # many uneven grids of mixed stencils in one captured launch
        _batch("batch_f32_64", 64, 64, 4096, 20, 5),
    ]


# the operand forms an FP32 grid can ask for
_FORMS_2D = ("native", "native", "any", "f16", "f16x3", "bf16x3", "tf32", "tf32x3", "sparse")


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, lo, hi, shape, d, r, dims):
    """Time steps in [lo, hi], fewer where the grid is large (the flagship's work is the most a case takes)."""
    per_step = 2.0 * inputs.num_weights(shape, d, r) * math.prod(dims)
    return max(1, min(rng.randint(lo, hi), int(1.2e11 / per_step)))


def draw(rng):
    kind = rng.choice(("2d_f32", "2d_f32", "2d_f32", "2d_f64", "2d_f64", "3d", "3d", "batch"))
    halo = rng.choice(("zero", "uniform"))
    if kind == "batch":
        return _batch(None, _log_int(rng, 8, 48), 64, rng.choice((512, 1024, 4096)), rng.randint(4, 20),
                      rng.randint(1, 10 ** 6))
    if kind == "3d":
        shape, r = rng.choice((("box", 1), ("star", 1), ("star", 2), ("star", 3)))
        dtype = rng.choice(("f32", "f32", "f64"))
        dims = [_log_int(rng, 33, 512) for _ in range(3)]
        return _plan(None, shape, 3, r, dims, dtype, rng.randint(1, 6), halo=halo)
    field = rng.choice(("uniform", "sine"))
    shape, r = rng.choice((("box", 1), ("box", 2), ("box", 3), ("star", 1), ("star", 2), ("star", 3)))
    side = 16384 if kind == "2d_f32" else 10240
    dims = [_log_int(rng, 200, side) for _ in range(2)]
    if kind == "2d_f64":
        precision = rng.choice(("native", "ozaki"))
        return _plan(None, shape, 2, r, dims, "f64", _steps(rng, 1, 20, shape, 2, r, dims), precision=precision,
                     field=field, halo=halo)
    form = rng.choice(_FORMS_2D)
    path = "auto"
    if form == "sparse":
        form, path = "tf32", "sparse_tensor_core"
    t = rng.choice((0, 0, 0, 1, 2, 3, 4))
    if t * r > 8:
        t = 0
    return _plan(None, shape, 2, r, dims, "f32", _steps(rng, 2, 16, shape, 2, r, dims), t=t, precision=form,
                 path=path, field=field, halo=halo)


def _dims(case):
    return tuple(case[f"n{i}"] for i in range(case["d"]))


def _torch_dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _field(dims, r, kind, halo, dtype, seed):
    """Stored field (halo of width r included) made on the device from the seed."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    stored = tuple(n + 2 * r for n in dims)
    inner = tuple(slice(r, r + n) for n in dims)
    if halo == "zero":
        u = torch.zeros(stored, dtype=dtype, device=DEVICE)
    else:
        u = torch.rand(stored, dtype=dtype, device=DEVICE, generator=gen)
    if kind == "uniform":
        u[inner] = torch.rand(dims, dtype=dtype, device=DEVICE, generator=gen)
        return u
    # eight seeded sine modes plus 1e-3 noise (the field of the precision study)
    p = inputs.uniform01(seed, 0, 32)
    y = torch.arange(dims[0], dtype=torch.float64, device=DEVICE)[:, None] / dims[0]
    x = torch.arange(dims[1], dtype=torch.float64, device=DEVICE)[None, :] / dims[1]
    f = torch.rand(dims, dtype=dtype, device=DEVICE, generator=gen).mul_(1e-3)
    for m in range(8):
        a, ky, kx, ph = p[4 * m] / 8.0, 1 + int(p[4 * m + 1] * 16), 1 + int(p[4 * m + 2] * 16), p[4 * m + 3]
        # sin(a + b) = sin a cos b + cos a sin b: two outer products instead of a full-size sine
        ay, bx = 2 * math.pi * ky * y, 2 * math.pi * (kx * x + ph)
        f.addcmul_((a * torch.sin(ay)).to(dtype), torch.cos(bx).to(dtype))
        f.addcmul_((a * torch.cos(ay)).to(dtype), torch.sin(bx).to(dtype))
    u[inner] = f
    return u


def _batch_descs(case):
    return inputs.batch_descs(case["grids"], seed=case["sizes_seed"], lo=case["lo"], hi=case["hi"])


def prepare(case, seed):
    dtype = _torch_dtype(case)
    if case["kind"] == "batch":
        grids, ins = [], []
        for i, (shape, r, ny, nx, _) in enumerate(_batch_descs(case)):
            grids.append((shape, r, ny, nx, inputs.weights(shape, 2, r, seed * 1009 + i)))
            ins.append(_field((ny, nx), r, "uniform", "zero", dtype, seed * 1009 + i))
        batch = B.Batch(grids, case["dtype"])
        batch.ensure_workspace(case["steps"], DEVICE)
        return {"batch": batch, "ins": ins, "outs": [torch.empty_like(x) for x in ins], "steps": case["steps"],
                "stream": torch.cuda.Stream()}
    shape, d, r, dims = case["shape"], case["d"], case["r"], _dims(case)
    w = inputs.weights(shape, d, r, seed)
    x = _field(dims, r, case["field"], case["halo"], dtype, seed)
    plan = B.Plan(shape, d, r, w, case["dtype"], dims, case["t"], precision=case["precision"], path=case["path"])
    plan.ensure_workspace(DEVICE)
    return {"plan": plan, "x": x, "y": torch.empty_like(x), "steps": case["steps"]}


def run(state):
    if "batch" in state:
        # a captured launch needs a stream of its own; the caller's stream waits for it
        cur, own = torch.cuda.current_stream(), state["stream"]
        own.wait_stream(cur)
        state["batch"].run(state["ins"], state["outs"], state["steps"], stream=own, graph=True)
        cur.wait_stream(own)
        return state["outs"]
    state["plan"].run(state["x"], state["y"], state["steps"])
    return state["y"]


def _cost(shape, d, r, dims, steps, itemsize):
    stored = math.prod(n + 2 * r for n in dims)
    return 2.0 * itemsize * stored, 2.0 * inputs.num_weights(shape, d, r) * math.prod(dims) * steps


def work(case):
    """One read of the stored field and one write of the result; a multiply and
    an add per weight, point and step."""
    if case["kind"] == "batch":
        costs = [_cost(s, 2, r, (ny, nx), case["steps"], 4) for s, r, ny, nx, _ in _batch_descs(case)]
    else:
        costs = [_cost(case["shape"], case["d"], case["r"], _dims(case), case["steps"],
                       8 if case["dtype"] == "f64" else 4)]
    return {"bytes": sum(c[0] for c in costs), "flops": sum(c[1] for c in costs)}


def _offsets(shape, d, r):
    rng = range(-r, r + 1)
    if d == 2:
        every = [(y, x) for y in rng for x in rng]
    else:
        every = [(z, y, x) for z in rng for y in rng for x in rng]
    return every if shape == "box" else [o for o in every if sum(c != 0 for c in o) <= 1]


def _exact_run(shape, d, r, w, dims, u, steps):
    """`steps` steps in FP64 with plain tensor arithmetic (halo cells fixed)."""
    a = u.to(torch.float64)
    inner = tuple(slice(r, r + n) for n in dims)
    for _ in range(steps):
        acc = torch.zeros(dims, dtype=torch.float64, device=u.device)
        for o, wk in zip(_offsets(shape, d, r), w):
            acc.add_(a[tuple(slice(r + c, r + c + n) for c, n in zip(o, dims))], alpha=float(wk))
        a = a.clone() if a is u else a
        a[inner] = acc
    return a


def exact(case, seed):
    dtype = _torch_dtype(case)
    if case["kind"] == "batch":
        out = []
        for i, (shape, r, ny, nx, _) in enumerate(_batch_descs(case)):
            w = inputs.weights(shape, 2, r, seed * 1009 + i)
            u = _field((ny, nx), r, "uniform", "zero", dtype, seed * 1009 + i)
            out.append(_exact_run(shape, 2, r, w, (ny, nx), u, case["steps"]))
        return out
    shape, d, r, dims = case["shape"], case["d"], case["r"], _dims(case)
    u = _field(dims, r, case["field"], case["halo"], dtype, seed)
    return _exact_run(shape, d, r, inputs.weights(shape, d, r, seed), dims, u, case["steps"])
