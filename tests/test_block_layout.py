"""Host checks of the 2-D tensor-core kernels' operand addressing (no GPU).

The block form (csrc/k_wide.cu) makes the weights the A operand over blocks of
16 x 8 outputs and block positions (8 across a group of 64 columns, gn down;
hx such groups per tile) the B operand.  This test lays the weight strip and a staged tile out as the kernel
does (16-bit operands: 8 values per 16-byte chunk; TF32: 4, even and odd chunks
in two planes), reads every issued MMA's core matrices back through the
descriptor arithmetic (start, LBO, SBO), and compares the sum of products with
the composite stencil evaluated directly.  Every address must lie inside the
strip and the operand buffer, and every tile must fit shared memory and TMEM.
"""
import itertools

import numpy as np
import pytest

import oracle
from paper_2603_00477_gb300 import inputs

SMEM = 227 * 1024


def geom(R, tf32, split, gn, hx, nbuf):
    ce = 4 if tf32 else 8
    rows = 16 * gn + 2 * R
    nc = -(-(8 + 2 * R) // ce)
    pc = 8 * hx + ((nc - 1) // 2 if tf32 else nc - 1)
    plane = -(-rows * pc * 16 // 128) * 128 + 64 if tf32 else 0
    in_bytes = -(-(plane + rows * pc * 16) // 128) * 128
    smem = 1024 + 8 * 4 * 72 * 4 + ((31 + 2 * R) * nc * 128 + nbuf * in_bytes) * (2 if split else 1)
    return dict(ce=ce, rows=rows, nc=nc, pc=pc, plane=plane, in_bytes=in_bytes, smem=smem)


def issue_list(R, nc, pc, tf32, plane):
    """(A start, A LBO, B start, B LBO) of every MMA of a tile, in bytes; SBOs are nc * 128 and 16 rows."""
    out = []
    for ky in range(0, 16 + 2 * R, 2):
        for y in (ky, ky + 1):
            for c in range(0, nc - 1, 2):
                out.append(((y * nc + c) * 128, 128, (y * pc + (c // 2 if tf32 else c)) * 16, plane if tf32 else 16))
        if nc & 1:
            c = nc - 1
            out.append(((ky * nc + c) * 128, nc * 128, (ky * pc + (c // 2 if tf32 else c)) * 16, pc * 16))
    return out


@pytest.mark.parametrize("tf32", [False, True])
@pytest.mark.parametrize("hx", [1, 2])
@pytest.mark.parametrize("shape,r,t", [("box", 1, 1), ("box", 2, 1), ("star", 3, 1), ("box", 2, 2), ("box", 1, 5),
                                       ("star", 2, 3), ("box", 1, 7), ("box", 2, 4), ("box", 3, 3), ("star", 5, 2),
                                       ("box", 1, 11), ("box", 6, 2)])
def test_block_operands_reproduce_the_composite(shape, r, t, hx, tf32):
    R, gn = t * r, 2
    g = geom(R, tf32, False, gn, hx, 2)
    ce, nc, pc = g["ce"], g["nc"], g["pc"]
    lines = 2 * R + 1
    wt = oracle.compose(shape, 2, r, inputs.weights(shape, 2, r, 5), t)
    # weight strip, one value per operand element
    strip = np.zeros((31 + 2 * R) * nc * 8 * ce)
    e = np.arange(strip.size)
    j, i, core = e % ce, (e // ce) % 8, e // (8 * ce)
    d, idx = core // nc - 15, ce * (core % nc) + j + i - 7
    ok = (d >= 0) & (d < lines) & (idx >= 0) & (idx < lines)
    strip[ok] = wt[d[ok], idx[ok]]
    # staged tile: item i = (row, quad of columns) at an offset linear in i
    rng = np.random.default_rng(3)
    tile = rng.uniform(-1, 1, size=(g["rows"], 8 * pc))
    esz = 4 if tf32 else 2
    buf = np.full(g["in_bytes"] // esz, np.nan)
    for row in range(g["rows"]):
        for c4 in range(2 * pc):
            it = row * 2 * pc + c4
            off = (it >> 1) * 16 + (it & 1) * g["plane"] if tf32 else it * 8
            buf[off // esz:off // esz + 4] = tile[row, 4 * c4:4 * c4 + 4]
    acc = np.zeros((hx, 128, 8 * gn))
    m, n = np.arange(128), np.arange(8 * gn)
    jj = np.arange(ce)
    mmas = issue_list(R, nc, pc, tf32, g["plane"])
    assert len(mmas) == (16 + 2 * R) // 2 * nc
    for a0, albo, b0, blbo in mmas:
        for h in range(hx):  # the groups of 64 columns: 8 units of 16 bytes apart
            for kc in range(2):  # the two 16-byte K core matrices of an instruction
                ia = (a0 + kc * albo + (m // 8) * nc * 128 + (m % 8) * 16)[:, None] // esz + jj
                ib = (b0 + h * 128 + kc * blbo + (n // 8) * 16 * pc * 16 + (n % 8) * 16)[:, None] // esz + jj
                assert ia.min() >= 0 and ia.max() < strip.size
                assert ib.min() >= 0 and ib.max() < buf.size
                acc[h] += strip[ia] @ buf[ib].T
    # output (y, x) of the tile: row m = 8 (15 - my) + 7 - mx, column n = 8 G + q of group x / 64
    want = np.zeros((16 * gn, 64 * hx))
    for a in range(lines):
        for b in range(lines):
            want += wt[a, b] * tile[a:a + 16 * gn, b:b + 64 * hx]
    y, x = np.arange(16 * gn)[:, None], np.arange(64 * hx)[None, :]
    got = acc[x // 64, 8 * (15 - y % 16) + 7 - x % 8, 8 * (y // 16) + (x % 64) // 8]
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-13)


@pytest.mark.parametrize("tf32,split", [(False, False), (False, True), (True, False), (True, True)])
def test_block_tiles_fit(tf32, split):
    """Every fused radius up to 12 has a tile of at least 64 x 64 outputs whose operands fit shared memory
    and whose two accumulator sets (four for TF32x3) fit TMEM; descriptor fields stay inside 14 bits."""
    for R in range(1, 13):
        fits = []
        for gn, hx, nbuf in itertools.product((32, 24, 16, 12, 8, 6, 4), (1, 2), (2, 1)):
            g = geom(R, tf32, split, gn, hx, nbuf)
            if 8 * gn * hx * (4 if tf32 and split else 2) <= 512 and g["smem"] <= SMEM:
                fits.append((gn, hx))
                assert (8 * gn) % 16 == 0
                for off in (g["plane"], 16 * g["pc"] * 16, g["nc"] * 128, g["smem"]):
                    assert off % 16 == 0 and off // 16 < 1 << 14
        assert max(gn * hx for gn, hx in fits) >= 4, (R, tf32, split)


@pytest.mark.parametrize("shape,r", [("box", 1), ("box", 2), ("box", 3), ("star", 2), ("box", 7)])
@pytest.mark.parametrize("t", [0, 1, 3])
def test_tf32_with_an_open_path_runs_dense(shape, r, t):
    """precision tf32, path auto: the dense block kernel at the ranking's t (an explicit sparse path is kept)."""
    from paper_2603_00477_gb300 import binding as B
    if t * r > 12:
        pytest.skip("t r > 12")
    w = inputs.weights(shape, 2, r, 1)
    p = B.Plan(shape, 2, r, w, "f32", (3000, 2000), t, precision="tf32")
    info = p.info()
    assert info["path"] == B.PATH_TENSOR_CORE and info["precision"] == B.PREC_TF32
    assert t == 0 or info["t"] == t
    p.set_option("path", "sparse_tensor_core")
    assert p.info()["path"] == B.PATH_SPARSE_TENSOR_CORE
    p.close()
