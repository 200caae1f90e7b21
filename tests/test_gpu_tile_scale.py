"""The power-of-two scale of a tile in the FP16 / BF16 forms: small values beside a large one, and no memory of other tiles.

A tile's largest |x| is scaled to [2^14, 65504].  FP16 numbers are normal from 2^-14 on, so a value of 2^-28 of
the largest or more keeps 11 bits, and one of 2^-17 or more keeps the 22 bits of hi + lo (the lo part, 2^-11 of it,
ends at 2^-24).  Outside the reach of the large value the relative error is then that of the form: its operand
rounding P plus one FP32 ulp per MMA (the bound of the block form).
"""
import numpy as np
import pytest

import oracle
from paper_2603_00477_gb300 import binding as B
from paper_2603_00477_gb300 import inputs

from tc_bounds import P_FORM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    from paper_2603_00477_gb300 import build
    build.build()
    B.load()
    return _t


def bound(form, R):
    return P_FORM[form] + (16 + 2 * R) // 2 * -(-(8 + 2 * R) // 8) * (1 if form == "f16" else 3) * 2.0 ** -23


def sweep(torch, form, r, w, dims, u):
    plan = B.Plan("box", 2, r, w, "f32", dims, 1, precision=form, path="tensor_core")
    x = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    y = torch.full_like(x, float("nan"))
    plan.run(x, y, 1)
    B.stencil_device_status()
    out = y.cpu().numpy()
    plan.close()
    return out


# one tile; aligned rows (edge tile), ragged rows; a grid with interior tiles of the aligned and the ragged loader
@pytest.mark.parametrize("dims", [(64, 60), (64, 61), (1200, 1020), (1200, 1021)])
@pytest.mark.parametrize("form,below", [("f16", 28), ("f16x3", 17), ("bf16x3", 28)])
def test_quiet_surroundings_of_a_pulse(torch, form, below, dims):
    """A pulse of 2^-5 in every 16 x 64 cells (so in every tile) over values of 2^-below of it."""
    r, pulse = 1, 2.0 ** -5
    w = inputs.weights("box", 2, r, 3)
    stored = tuple(n + 2 * r for n in dims)
    u = np.random.default_rng(5).uniform(1, 2, size=stored) * pulse * 2.0 ** -below
    hit = np.zeros(stored, dtype=bool)
    for y in range(7, stored[0], 16):
        for x in range(9, stored[1], 32):
            u[y, x] = pulse
            hit[y - r:y + r + 1, x - r:x + r + 1] = True
    u = u.astype(np.float32)
    out = sweep(torch, form, r, w, dims, u).astype(np.float64)
    ref = oracle.run("box", 2, r, w, dims, u.astype(np.float64), 1)
    inner = (slice(r, -r), slice(r, -r))
    quiet = ~hit[inner]
    err = np.abs(out - ref)[inner][quiet]
    # values in [1, 2) 2^-below pulse and weights of sum 1: the largest operand is at most twice any output
    assert (err <= 2 * bound(form, r) * ref[inner][quiet]).all(), (err / ref[inner][quiet]).max() / bound(form, r)


@pytest.mark.parametrize("dims", [(6000, 3004), (6000, 3005)])
@pytest.mark.parametrize("form", ["f16", "f16x3", "bf16x3"])
def test_a_tile_does_not_depend_on_the_tiles_before_it(torch, form, dims):
    """A pulse in every 16 x 32 cells over far smaller values; the lower half of the grid gives the same bits
    whether the upper half is as large, 4096 times larger or zero."""
    r, pulse = 1, 2.0 ** -5
    w = inputs.weights("box", 2, r, 3)
    u = np.exp2(-np.random.default_rng(8).uniform(16, 30, size=tuple(n + 2 * r for n in dims))) * pulse
    u[7::16, 9::32] = pulse
    outs = []
    for scale in (1.0, 4096.0, 0.0):
        v = u.copy()
        v[:2500] *= scale
        outs.append(sweep(torch, form, r, w, dims, v.astype(np.float32))[3200:])  # tiles hold at most 512 rows
    np.testing.assert_array_equal(outs[0], outs[1])
    np.testing.assert_array_equal(outs[0], outs[2])
