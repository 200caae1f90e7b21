"""How the launchers cut a grid into work items (csrc/launch_rules.h, plain host arithmetic compiled here; no GPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")

    def run(expr):
        src, exe = d / "rule.cpp", d / "rule"
        src.write_text(f'#include <cstdio>\n#include "launch_rules.h"\n'
                       f'int main() {{ std::printf("%lld", (long long)({expr})); }}\n')
        subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2603_00477_gb300", "csrc"), str(src),
                        "-o", str(exe)], check=True)
        return int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout)
    return run


# 256^3 in FP64: 64 tiles of 16 x 64 per plane.  Two CTAs per SM: 37 planes are 448 items on 304 CTAs, of which
# 144 take a second one, so that some SMs work off four (148 planes of work against 120 .. 130 of the others)
@pytest.mark.parametrize("nz,cols,occ,bad", [(256, 64, 2, 37), (100, 13, 2, 3)])
def test_streaming_chunks_leave_no_sm_with_one_item_more(call, nz, cols, occ, bad):
    c = call(f"gbs::stream_planes({nz}, {cols}, {occ}, {SMS})")
    items = -(-nz // c) * cols
    rest = items % (occ * SMS)
    assert c != bad and (items <= occ * SMS or rest == 0 or rest <= 0.8 * SMS or rest > 1.6 * SMS)


def test_streaming_chunks_that_stay(call):
    """Three CTAs per SM (radius 1): 448 items are one wave."""
    assert call(f"gbs::stream_planes(256, 64, 3, {SMS})") == 37
    assert 1 <= call(f"gbs::stream_planes(1, 1, 2, {SMS})") <= 1


# tiles of a plane as rot_tile cuts it: 128 x 44 x 112 (Star-3D3R) 3, 64^3 (Star-3D3R) 3
@pytest.mark.parametrize("nz,cols,r,c", [(128, 3, 3, 3), (64, 3, 3, 2)])
def test_marching_runs_of_a_small_grid_give_an_sm_one_cta(call, nz, cols, r, c):
    assert call(f"gbs::rot_planes({nz}, {cols}, {r}, 2, {SMS})") == c
    assert -(-nz // c) * cols <= SMS


# 512^3 Star-3D2R, 301 x 417 x 533 Box-3D1R, 256^3 Star-3D3R, a thin grid: two CTAs per SM as before
@pytest.mark.parametrize("nz,cols,r,c", [(512, 136, 2, 256), (301, 56, 1, 61), (256, 35, 3, 32), (34, 126, 3, 17)])
def test_marching_runs_that_stay(call, nz, cols, r, c):
    assert call(f"gbs::rot_planes({nz}, {cols}, {r}, 2, {SMS})") == c


# a small grid's band is cut into more pieces; pieces never number more than the SMs for being short
@pytest.mark.parametrize("ny,nx,band,length", [(300, 200, 3, 32), (100, 100, 9, 32), (1500, 1400, 6, 64), (16384, 16384, 6, 128),
                                               (1, 300, 4, 32), (2000, 2600, 4, 64)])
def test_band_pieces_of_a_small_grid(call, ny, nx, band, length):
    got = call(f"gbs::band_length({ny}, {nx}, {band}, {SMS})")
    assert got == length


@pytest.mark.parametrize("ny,nx,band", [(1, 1, 3), (2, 300, 3), (300, 2, 5), (7, 9, 4), (130, 259, 6), (33, 32, 8)])
@pytest.mark.parametrize("length", [32, 64, 128])
def test_band_pieces_cover_the_band_once(tmp_path, ny, nx, band, length):
    """Every interior point nearer than `band` to the boundary is in exactly one piece, as the kernel reads them."""
    prog = f"""
#include <cstdio>
#include <vector>
#include "launch_rules.h"
int main() {{
    const gbs::BandPieces g = gbs::band_pieces({ny}, {nx}, {band}, {length});
    std::vector<int> seen({ny} * {nx}, 0);
    for (int id = 0; id < g.n_h + g.n_v; id++) {{
        long y0, x0, by, bx;
        if (id < g.n_h) {{
            const bool b = id >= g.h;
            by = b ? g.bot : g.top; y0 = b ? {ny} - g.bot : 0;
            x0 = (long)(b ? id - g.h : id) * {length}; bx = std::min<long>({length}, {nx} - x0);
        }} else {{
            const int v = id - g.n_h; const bool r = v >= g.v;
            bx = r ? g.right : g.left; x0 = r ? {nx} - g.right : 0;
            y0 = g.top + (long)(r ? v - g.v : v) * {length}; by = std::min<long>({length}, {ny} - g.bot - y0);
        }}
        for (long y = y0; y < y0 + by; y++) for (long x = x0; x < x0 + bx; x++) seen[y * {nx} + x]++;
    }}
    int bad = 0;
    for (int y = 0; y < {ny}; y++) for (int x = 0; x < {nx}; x++) {{
        const bool in = y < {band} || x < {band} || {ny} - 1 - y < {band} || {nx} - 1 - x < {band};
        bad += seen[y * {nx} + x] != (in ? 1 : 0);
    }}
    std::printf("%d", bad);
}}
"""
    src, exe = tmp_path / "b.cpp", tmp_path / "b"
    src.write_text(prog)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2603_00477_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "0"


@pytest.mark.parametrize("args,tiles", [("0, 3, 1, 512, 512, 16, 32", 1), ("0, 3, 1, 2048, 2048, 64, 128", 1),
                                        ("0, 3, 1, 4096, 4096, 64, 128", 0), ("0, 3, 1, 512, 90, 16, 32", 0),
                                        ("1, 3, 1, 512, 512, 16, 32", 0), ("0, 2, 1, 512, 512, 16, 32", 0)])
def test_tiled_or_marching(call, args, tiles):
    assert call(f"gbs::tiles_beat_march({args})") == tiles


@pytest.mark.parametrize("args,early", [("true, 3, 1, 100000, 456", 0), ("false, 3, 3, 500, 456", 1),
                                        ("false, 4, 1, 460, 304", 0), ("false, 6, 1, 1128, 304", 1),
                                        ("false, 6, 2, 1128, 304", 0), ("false, 7, 3, 552, 304", 0)])
def test_when_the_next_sweep_is_let_in(call, args, early):
    assert call(f"gbs::next_sweep_early({args})") == early


# 600 tiles: three CTAs per SM leave some SMs with five, two with four; the others keep what the occupancy allows
@pytest.mark.parametrize("tiles,occ,ctas", [(600, 3, 2), (512, 3, 3), (65536, 3, 3), (100, 3, 3), (456, 3, 3), (600, 2, 2),
                                            (600, 1, 1)])
def test_fp64_tiles_per_sm(call, tiles, occ, ctas):
    assert call(f"gbs::f64_tile_ctas({tiles}, {occ}, {SMS})") == ctas
