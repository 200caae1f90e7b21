"""GPU parity of the 2-D FP32 marching kernel (t = 1 and 2) at the edges of its column blocks and segments.

A warp yields 4 (32 - 2t) columns (120 at t = 1, 112 at t = 2); rows that are 16-byte multiples take quads,
others words; non-zero halos are kept between fused steps.  Tolerance: FP32, 1e-5 normwise (K <= 25 products of
positive weights with sum 1 round within K 2^-24 per step, 12 steps).
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


# one row / column, fewer rows than a window, block edges (120, 112 and their neighbours), many blocks and segments;
# with r = 1, 2, 3 the stored rows take every residue mod 4
DIMS = [(1, 1), (1, 500), (500, 1), (2, 3), (5, 120), (7, 121), (30, 112), (64, 113), (333, 239), (257, 244),
        (1000, 367), (61, 2000)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shape,r,t", [("box", 1, 1), ("box", 1, 2), ("box", 2, 1), ("star", 1, 1), ("star", 1, 2),
                                       ("star", 2, 1), ("star", 2, 2), ("star", 3, 1)])
def test_march(torch, shape, r, t, dims):
    w = inputs.weights(shape, 2, r, 3)
    u = np.random.default_rng(11).uniform(-1, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    plan = B.Plan(shape, 2, r, w, "f32", dims, t)
    x = torch.from_numpy(u).cuda()
    y = torch.full_like(x, float("nan"))
    for steps in (1, 2 * t + 1, 12):
        plan.run(x, y, steps)
        ref = oracle.run(shape, 2, r, w, dims, u.astype(np.float64), steps)
        assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-5
        np.testing.assert_array_equal(y.cpu().numpy()[:r], u[:r])
    plan.close()


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_buffers(torch, offset):
    """Rows of a 16-byte length in buffers that do not start on a 16-byte boundary take the word path."""
    shape, r, dims = "box", 2, (90, 256)
    w = inputs.weights(shape, 2, r, 3)
    u = np.random.default_rng(12).uniform(-1, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    n = u.size
    xb = torch.zeros(n + 8, device="cuda")
    yb = torch.zeros(n + 8, device="cuda")
    xb[offset:offset + n] = torch.from_numpy(u.ravel()).cuda()
    plan = B.Plan(shape, 2, r, w, "f32", dims, 1)
    x, y = xb[offset:offset + n].view(u.shape), yb[:n].view(u.shape)
    plan.run(x, y, 3)
    ref = oracle.run(shape, 2, r, w, dims, u.astype(np.float64), 3)
    assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-5
    plan.close()


@pytest.mark.parametrize("shape,r,t", [("box", 2, 1), ("star", 2, 2), ("star", 3, 1)])
def test_same_bits_as_the_tiled_kernel(torch, shape, r, t):
    """Same products in the same order: a tile asked for (the tiled kernel) gives the same bits."""
    dims = (300, 444)
    w = inputs.weights(shape, 2, r, 5)
    u = np.random.default_rng(13).uniform(-1, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    x = torch.from_numpy(u).cuda()
    outs = []
    for tile in ("0", "48x64"):
        plan = B.Plan(shape, 2, r, w, "f32", dims, t)
        plan.set_option("tile", tile)
        y = torch.empty_like(x)
        plan.run(x, y, 6)
        outs.append(y.cpu().numpy())
        plan.close()
    np.testing.assert_array_equal(outs[0], outs[1])


def test_batched_marching_tiles(torch):
    """The batched kernel's marching path over thin, ragged and aligned grids: the same bits as single runs
    (remainder sweeps of depth 1 on tiles cut for depth 2 included)."""
    shapes = [("box", 1), ("box", 2), ("box", 3), ("star", 1), ("star", 2), ("star", 3)]
    dims = [(1, 1), (3, 300), (300, 2), (64, 119), (65, 241), (130, 448), (257, 700), (1100, 1000)]
    grids, ins = [], []
    rng = np.random.default_rng(21)
    for i, (ny, nx) in enumerate(dims):
        for shape, r in shapes:
            grids.append((shape, r, ny, nx, inputs.weights(shape, 2, r, 40 + i)))
            ins.append(torch.from_numpy(rng.uniform(-1, 1, size=(ny + 2 * r, nx + 2 * r)).astype(np.float32)).cuda())
    batch = B.Batch(grids, "f32")
    outs = [torch.full_like(x, float("nan")) for x in ins]
    for steps in (1, 7):
        batch.run(ins, outs, steps)
        B.stencil_batch_status(batch.handle)
        for (shape, r, ny, nx, w), x, y in zip(grids, ins, outs):
            plan = B.Plan(shape, 2, r, w, "f32", (ny, nx), 0, path="cuda_core")
            ref = torch.empty_like(x)
            plan.run(x, ref, steps)
            assert torch.equal(y, ref), (shape, r, ny, nx, steps)
            plan.close()
    batch.close()
