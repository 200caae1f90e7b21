"""GPU parity of the 2-D tensor-core kernels (block form) at the edges of their tiles and of the band strips.

Tolerance per fused sweep: operand rounding P of the form plus one FP32 ulp
(2^-23) per issued MMA -- (16 + 2R)/2 x ceil((8 + 2R)/c) MMAs of a block's
neighbourhood (c = 8 values per 16-byte chunk, TF32: 4), three times for the
hi + lo forms -- summed over sweeps (normwise, positive weights of sum 1).
"""
import numpy as np
import pytest

import oracle
from paper_2603_00477_gb300 import binding as B
from paper_2603_00477_gb300 import inputs

from tc_bounds import P_FORM, sweeps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_2603_00477_gb300 import build
    build.build()
    B.load()
    return _t


def bound(form, R, steps, t):
    c = 4 if form.startswith("tf32") else 8
    mmas = (16 + 2 * R) // 2 * -(-(8 + 2 * R) // c) * (1 if form in ("tf32", "f16") else 3)
    return sweeps(steps, t) * (P_FORM[form] + mmas * 2.0 ** -23)


def run(torch, shape, r, w, dims, u, steps, t, form):
    plan = B.Plan(shape, 2, r, w, "f32", dims, t, precision=form, path="tensor_core")
    x = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    y = torch.full_like(x, float("nan"))
    plan.run(x, y, steps)
    B.stencil_device_status()
    out = y.cpu().numpy()
    plan.close()
    return out


FORMS = ["f16", "f16x3", "bf16x3", "tf32", "tf32x3"]
# interior rows/columns around tile edges (64 columns; rows 16 gn), stored rows of every residue mod 4
# (aligned, 8-byte and unaligned loads and stores), fewer rows than the band, one tile and many
SIZES = [(1, 1), (3, 200), (200, 3), (64, 64), (65, 127), (333, 446), (401, 334), (402, 335), (399, 337), (2100, 700)]


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("dims", SIZES)
def test_sizes(torch, form, dims):
    r, t = 2, 2
    w = inputs.weights("box", 2, r, 3)
    u = np.random.default_rng(5).uniform(0, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    out = run(torch, "box", r, w, dims, u, 5, t, form)
    ref = oracle.run("box", 2, r, w, dims, u.astype(np.float64), 5)
    assert oracle.rel_linf(out, ref) <= bound(form, r * t, 5, t)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("shape,r,t", [("box", 1, 1), ("box", 3, 1), ("star", 2, 2), ("box", 5, 1), ("box", 2, 3),
                                       ("box", 7, 1), ("star", 2, 4), ("box", 3, 3), ("star", 5, 2), ("box", 1, 11),
                                       ("star", 6, 2)])
def test_radii(torch, form, shape, r, t):
    """Every chunk count of a neighbourhood row (R = 1 .. 12), odd and even."""
    dims = (410, 390)
    w = inputs.weights(shape, 2, r, 4)
    u = np.random.default_rng(6).uniform(0, 1, size=tuple(n + 2 * r for n in dims)).astype(np.float32)
    steps = 2 * t
    out = run(torch, shape, r, w, dims, u, steps, t, form)
    ref = oracle.run(shape, 2, r, w, dims, u.astype(np.float64), steps)
    assert oracle.rel_linf(out, ref) <= bound(form, r * t, steps, t)


@pytest.mark.parametrize("form", ["f16", "f16x3", "bf16x3"])
@pytest.mark.parametrize("scale", [2.0 ** -100, 2.0 ** 60])
def test_scale_follows_the_field(torch, form, scale):
    """A field whose magnitude jumps by 2^24 from one band of 700 rows to the next (each tile's scale is the
    previous one's until it no longer fits), times a global power of two: every band is as accurate as alone."""
    dims, r, t = (2800, 700), 2, 1
    w = inputs.weights("box", 2, r, 3)
    u = np.random.default_rng(7).uniform(0.5, 1, size=tuple(n + 2 * r for n in dims))
    u[700:1400] *= 2.0 ** 24
    u[2100:] = 0.0
    u = (u * scale).astype(np.float32)
    out = run(torch, "box", r, w, dims, u, 1, t, form).astype(np.float64)
    ref = oracle.run("box", 2, r, w, dims, u.astype(np.float64), 1)
    assert oracle.rel_linf(out, ref) <= bound(form, r, 1, t)
    # rows whose tile cannot reach another band (tiles are at most 512 rows)
    for lo, hi in ((0, 170), (2700, 2800)):
        a, b = out[lo + r:hi + r, r:-r], ref[lo + r:hi + r, r:-r]
        assert np.abs(a - b).max() <= bound(form, r, 1, t) * max(np.abs(b).max(), 1e-300)


@pytest.mark.parametrize("dtype,form", [("f32", "tf32x3"), ("f64", "ozaki"), ("f64", "native")])
@pytest.mark.parametrize("dims", [(1, 300), (300, 2), (5, 6), (9, 140), (130, 11), (129, 257)])
def test_band_strips(torch, dtype, form, dims):
    """Band strips that overlap, meet or leave a middle: every interior point is written."""
    shape, r, t = "box", 2, 3
    w = inputs.weights(shape, 2, r, 8)
    npdt = np.float32 if dtype == "f32" else np.float64
    u = np.random.default_rng(9).uniform(0, 1, size=tuple(n + 2 * r for n in dims)).astype(npdt)
    plan = B.Plan(shape, 2, r, w, dtype, dims, t, precision=form, path="tensor_core")
    x = torch.from_numpy(u).cuda()
    y = torch.full_like(x, float("nan"))
    plan.run(x, y, 2 * t)
    B.stencil_device_status()
    plan.close()
    ref = oracle.run(shape, 2, r, w, dims, u.astype(np.float64), 2 * t)
    assert oracle.rel_linf(y.cpu().numpy(), ref) <= (bound(form, r * t, 2 * t, t) if dtype == "f32" else 1e-12)
