"""GPU parity of the 3-D FP32 z-marching kernel and the FP64 streaming kernel's chunks at tile and run edges.

The tile (quads per row, strips) and the run of planes follow the grid, so the sizes here take thin, ragged and
several-tile grids, stored rows of every residue mod 4 and unaligned buffers.  Tolerances: FP32 1e-5, FP64 1e-12
(normwise).
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


DIMS = [(1, 1, 1), (2, 3, 200), (40, 1, 5), (1, 70, 33), (9, 65, 130), (17, 33, 255), (70, 20, 62), (33, 130, 64),
        (5, 61, 513)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shape,r", [("box", 1), ("star", 1), ("star", 2), ("star", 3)])
def test_rot(torch, shape, r, dims):
    w = inputs.weights(shape, 3, r, 3)
    u = np.random.default_rng(11).uniform(-1, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    plan = B.Plan(shape, 3, r, w, "f32", dims, 1)
    x = torch.from_numpy(u).cuda()
    y = torch.full_like(x, float("nan"))
    for steps in (1, 3):
        plan.run(x, y, steps)
        ref = oracle.run(shape, 3, r, w, dims, u.astype(np.float64), steps)
        assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-5
        np.testing.assert_array_equal(y.cpu().numpy()[:r], u[:r])
    # the same grid in buffers off the 16-byte boundary (words instead of quads)
    n = u.size
    xb, yb = torch.zeros(n + 4, device="cuda"), torch.zeros(n + 4, device="cuda")
    xb[1:n + 1] = x.ravel()
    x1, y1 = xb[1:n + 1].view(u.shape), yb[1:n + 1].view(u.shape)
    plan.run(x1, y1, 3)
    np.testing.assert_array_equal(y1.cpu().numpy(), y.cpu().numpy())
    plan.close()


@pytest.mark.parametrize("dims", [(1, 5, 70), (65, 17, 64), (130, 33, 65)])
def test_stream_f64_chunks(torch, dims):
    w = inputs.weights("box", 3, 1, 3)
    u = np.random.default_rng(12).uniform(-1, 1, size=tuple(n + 2 for n in dims))
    plan = B.Plan("box", 3, 1, w, "f64", dims, 1)
    x = torch.from_numpy(u).cuda()
    y = torch.full_like(x, float("nan"))
    plan.run(x, y, 3)
    ref = oracle.run("box", 3, 1, w, dims, u, 3)
    assert oracle.rel_linf(y.cpu().numpy(), ref) <= 1e-12
    plan.close()
