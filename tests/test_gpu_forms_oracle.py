"""GPU parity with the oracle of the forms a batch mixes (marching strips, shared-memory tiles, both in one launch)
and of the marching kernel's largest radius.

Tolerance: FP32, 1e-5 normwise (K <= 49 products of positive weights with sum 1 round within K 2^-24 per step).
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


@pytest.mark.parametrize("dims", [(1, 1), (3, 500), (64, 113), (257, 244), (130, 127), (500, 361)])
@pytest.mark.parametrize("shape,r,t", [("box", 3, 1), ("star", 3, 2)])
def test_march_radius_3(torch, shape, r, t, dims):
    w = inputs.weights(shape, 2, r, 3)
    u = np.random.default_rng(11).uniform(-1, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    plan = B.Plan(shape, 2, r, w, "f32", dims, t)
    x = torch.from_numpy(u).cuda()
    y = torch.full_like(x, float("nan"))
    for steps in (1, 2 * t + 1, 12):
        plan.run(x, y, steps)
        ref = oracle.run(shape, 2, r, w, dims, u.astype(np.float64), steps)
        assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-5
    plan.close()


# (kinds, sides): small and heavy (staged), light (marching), t = 2 with Box-2D3R staged beside marching grids,
# mostly staged, deeper than the marching kernel
@pytest.mark.parametrize("kinds,side,t", [
    ([("box", 3), ("box", 2)], 70, 0), ([("star", 1), ("box", 1)], 70, 0), ([("box", 3), ("star", 3)], 330, 1),
    ([("star", 2), ("box", 1), ("star", 3), ("box", 3)], 300, 2), ([("box", 3), ("star", 2)], 300, 2),
    ([("star", 3), ("box", 2)], 300, 3), ([("box", 1), ("star", 2)], 200, 4)])
def test_batch_forms(torch, kinds, side, t):
    grids, us = [], []
    rng = np.random.default_rng(17)
    for i in range(8):
        shape, r = kinds[i % len(kinds)]
        ny, nx = side + 7 * i, side + 5 * i - (i % 3)
        grids.append((shape, r, ny, nx, inputs.weights(shape, 2, r, 60 + i)))
        us.append(rng.uniform(-1, 1, size=(ny + 2 * r, nx + 2 * r)).astype(np.float32))
    batch = B.Batch(grids, "f32", t)
    ins = [torch.from_numpy(u).cuda() for u in us]
    outs = [torch.full_like(x, float("nan")) for x in ins]
    for steps in (1, 9):
        batch.run(ins, outs, steps)
        B.stencil_batch_status(batch.handle)
        for (shape, r, ny, nx, w), u, y in zip(grids, us, outs):
            ref = oracle.run(shape, 2, r, w, (ny, nx), u.astype(np.float64), steps)
            assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-5, (shape, r, ny, nx, steps)
    batch.close()
