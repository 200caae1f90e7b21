"""Which 3-D grids the marching kernel with 32-bit in-plane offsets may take (host rule, no GPU).

cu3d_rot keeps row * Ex + column of a stored plane in an int; rot3d_plane_fits has to send every plane where such
an offset would wrap to the streaming kernel, and to keep every other one.
"""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = """
#include <cstdio>
#include <cstdlib>
#include "internal.h"
int main(int argc, char **argv)
{
    for (int i = 1; i + 1 < argc; i += 2) std::printf("%d ", (int)gbs::rot3d_plane_fits(atoll(argv[i]), atoll(argv[i + 1])));
}
"""


@pytest.mark.parametrize("dims,fits", [((512, 512), True), ((46338, 46338), True), ((46339, 46339), False),
                                       ((50000, 50000), False), ((1, 2 ** 29), True), ((1, 2 ** 30), False),
                                       ((2 ** 31 - 8, 1), False), ((2 ** 20, 2 ** 18), False)])
def test_planes_with_wrapping_offsets_are_left_out(tmp_path, dims, fits):
    src, exe = tmp_path / "fits.cpp", tmp_path / "fits"
    src.write_text(PROG)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2603_00477_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = 1
    ey, ex = dims[0] + 2 * r, dims[1] + 2 * r
    last = (ey - 1) * ex + ex - 1  # the largest offset of a plane
    wraps = int(np.array(last, dtype=np.int64).astype(np.int32)) != last
    out = subprocess.run([str(exe), str(ey), str(ex)], check=True, capture_output=True, text=True).stdout
    assert out.split() == [str(int(fits))]
    assert not (fits and wraps)


def test_the_launcher_asks_the_rule():
    """Both forms of the marching launch stand behind the rule."""
    with open(os.path.join(ROOT, "paper_2603_00477_gb300", "csrc", "k_cuda_core_impl.cuh")) as f:
        text = f.read()
    body = text[text.index("stencil_status launch3d(const Plan"):]
    assert body.index("rot3d_plane_fits(p.ext[1], p.ext[2])") < body.index("launch3d_rot<")
    assert text.count("launch3d_rot<SHAPE, R, ") == 2
