"""GPU parity of the packed-FMA march: box r = 2 at t = 2, single grids and batched.

The packed FMA rounds each half as the scalar one and the products keep their order, so the tiled kernel (a tile
asked for) and single steps at t = 1 give the same bits; against the oracle FP32's 1e-5 normwise (25 products of
positive weights with sum 1 round within 25 * 2^-24 per step, 7 steps).
"""
import numpy as np
import pytest

import oracle
from paper_2603_00477_gb300 import binding as B
from paper_2603_00477_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_2603_00477_gb300 import build
    build.build()
    B.load()
    return _t


# one cell, thin grids, the warp's 112 columns and their neighbours, quads (nx + 4 a multiple of 4) and words
@pytest.mark.parametrize("dims", [(1, 1), (1, 500), (500, 1), (5, 112), (7, 113), (33, 444), (130, 447), (1000, 366)])
def test_box2_t2(torch, dims):
    w = inputs.weights("box", 2, 2, 3)
    u = np.random.default_rng(31).uniform(-1, 1, size=tuple(n + 4 for n in dims)).astype(np.float32)
    x = torch.from_numpy(u).cuda()
    for steps in (2, 7):
        outs = []
        for t, tile in ((2, "0"), (1, "0"), (2, "32x64")):
            plan = B.Plan("box", 2, 2, w, "f32", dims, t)
            plan.set_option("tile", tile)
            y = torch.full_like(x, float("nan"))
            plan.run(x, y, steps)
            outs.append(y.cpu().numpy())
            plan.close()
        np.testing.assert_array_equal(outs[0], outs[1])
        np.testing.assert_array_equal(outs[0], outs[2])
        ref = oracle.run("box", 2, 2, w, dims, u.astype(np.float64), steps)
        assert oracle.rel_linf(outs[0], ref) <= 1e-5


def test_batched_box2_t2(torch):
    dims = [(1, 1), (3, 300), (64, 119), (130, 444), (700, 500)]
    rng = np.random.default_rng(32)
    grids = [("box", 2, ny, nx, inputs.weights("box", 2, 2, 40 + i)) for i, (ny, nx) in enumerate(dims)]
    ins = [torch.from_numpy(rng.uniform(-1, 1, size=(ny + 4, nx + 4)).astype(np.float32)).cuda() for ny, nx in dims]
    outs = [torch.full_like(x, float("nan")) for x in ins]
    batch = B.Batch(grids, "f32", t=2)
    batch.run(ins, outs, 7)  # the last sweep has depth 1
    B.stencil_batch_status(batch.handle)
    for (shape, r, ny, nx, w), x, y in zip(grids, ins, outs):
        plan = B.Plan(shape, 2, r, w, "f32", (ny, nx), 1, path="cuda_core")
        ref = torch.empty_like(x)
        plan.run(x, ref, 7)
        assert torch.equal(y, ref), (ny, nx)
        plan.close()
    batch.close()
