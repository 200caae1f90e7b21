// launch_rules.h -- how the launchers cut a grid into work items (plain host arithmetic, no CUDA).
#pragma once

#include <algorithm>
#include <cstdint>

namespace gbs {

// Where the tiled 2-D FP32 kernel is faster than the marching one although that has the depth: box r = 3 at t = 1
// (shape 0) on grids that the tile divides, where every tile takes the tiled kernel's fixed-strip sub-step.  A
// warp of the marching kernel walks six rows of halo at 196 FMAs a row for its few rows.  Marching and
// tiled, one sweep: 256^2 6.6 and 4.3 us, 512^2 8.8 and 5.1, 1024^2 10.2 and 9.3, 2048^2 19.2 and 16.6,
// 4096^2 51.7 and 55.7; 512 x 90, not divided, 5.1 and 7.1.
inline bool tiles_beat_march(int shape, int r, int t, int64_t ny, int64_t nx, int tile_y, int tile_x)
{
    return shape == 0 && r == 3 && t == 1 && ny % tile_y == 0 && nx % tile_x == 0 && ny * nx <= 6000000;
}

// When a sweep of the tiled 2-D kernel lets the blocks of the next sweep in (chained launches): at its start, or when
// a block's work is done.  Blocks let in early take the slots of the blocks that finish first, the next
// sweep's blocks with one tile more among them, and share those SMs; where the FMA pipe is the bound (FP64, and
// FP32 from radius 4 on) that costs more than the head start gives, unless one-step sweeps have three tiles
// per block or more.  Eight sweeps, unchained / early / late: Box-2D4R FP32 1440 x 2560 189 / 218 / 169 us, Star-2D6R
// 1440 x 2560 300 / 326 / 282, Star-2D7R t = 3 2048 x 2048 1043 / 1118 / 1033, Star-2D6R 3000 x 3000 826 / 705 / 806,
// Box-2D4R 3000 x 3000 439 / 392 / 419.
inline bool next_sweep_early(bool f64, int r, int t, int64_t tiles, int64_t resident)
{
    return !f64 && (r <= 3 || (t == 1 && tiles >= 3 * resident));
}

// Items of the busiest SM when persistent CTAs, `occ` resident per SM, work off `items`.  Up to one wave the CTAs
// are spread evenly; beyond it those that take one item more were measured to share an SM as soon as they are more
// than ~4/5 of the SMs (as if smaller GPCs were filled twice before larger ones once): 448 items on 304 CTAs
// take as long as four on some SMs, not three.
inline int64_t busiest_items(int64_t items, int occ, int sms)
{
    const int64_t wave = (int64_t)occ * sms, full = items / wave, rest = items % wave;
    if (full == 0) return (rest + sms - 1) / sms;
    return occ * full + (rest > 0 ? std::min<int64_t>(occ, (5 * rest + 4 * sms - 1) / (4 * sms)) : 0);
}

// Persistent CTAs per SM of the tiled 2-D kernel in FP64, at most `occ`: the FP64 pipe is the bound and two CTAs fill
// it, so the fewest items on the busiest SM count.  Box-2D5R 480 x 640: 600 tiles on 456 CTAs are five on some
// SMs (640 us for eight sweeps), on 304 CTAs four (547 us).
inline int f64_tile_ctas(int64_t tiles, int occ, int sms)
{
    int best = occ;
    for (int o = occ - 1; o >= 2; o--)
        if (busiest_items(tiles, o, sms) < busiest_items(tiles, best, sms)) best = o;
    return best;
}

// Output planes per work item of the 3-D streaming kernel (`cols` tiles of a plane side by side, `occ` resident
// CTAs per SM).  The FMA pipe is the bound and an SM's CTAs share it, so a sweep takes about (items of the busiest
// SM) x (planes + a start-up worth one plane).  Box-3D2R FP64 256^3, four sweeps: 18,150 us with 37 planes (448
// items counted as three on the busiest of 152 SMs), 14,030 us with 29, 16,060 us with 64.  64 planes whatever the grid:
// Box-3D1R FP64 256^3 908 us per sweep, 778 us with 37.
inline int64_t stream_planes(int64_t nz, int64_t cols, int occ, int sms)
{
    int64_t best = nz, best_cost = -1;
    for (int64_t n = 1; n <= std::min<int64_t>(nz, 64); n++) {
        const int64_t c = (nz + n - 1) / n;
        const int64_t cost = busiest_items((nz + c - 1) / c * cols, occ, sms) * (c + 1);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

// Output planes per work item of the 3-D marching kernel (an item stages 2 r planes more than it
// writes, and starts up for about four).  Two CTAs on an SM take 1.3 to 1.5 times the time of one per
// plane (Star-3D3R: 0.97 and 1.48 us), so a sweep of few items is faster with one CTA per SM and longer
// runs: 128 x 44 x 112, 192 items of two planes 15.3 us, 129 of three 10.8 us (13.2 us with the
// fixed tiles before); 64^3, 192 items of one 12.9 us, 96 of two 9.8 us.
inline int64_t rot_planes(int64_t nz, int64_t cols, int r, int occ, int sms)
{
    const int64_t slots = (int64_t)occ * sms;
    int64_t best = nz, best_cost = -1;
    for (int64_t n = 1; n <= std::min<int64_t>(nz, 512); n++) {
        const int64_t c = (nz + n - 1) / n, items = (nz + c - 1) / c * cols;
        const int64_t rounds = items <= sms ? 10 : 14 * ((items + slots - 1) / slots);  // x 1/10
        const int64_t cost = rounds * (c + 2 * r + 4);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

// Pieces of the four band strips (k_band.cu) of an ny x nx interior cut into lengths of `len`:
// horizontal ones (top, and bottom if there is one) first, then vertical ones.
struct BandPieces {
    int top, bot;      // rows of the top and bottom strips (bot < band only when they would overlap)
    int left, right;   // columns of the left and right strips
    int h, v;          // pieces of one horizontal and one vertical strip
    int n_h, n_v;      // pieces of both
};

inline BandPieces band_pieces(int64_t ny, int64_t nx, int band, int len)
{
    BandPieces g;
    g.top = (int)std::min<int64_t>(band, ny);
    g.bot = (int)std::min<int64_t>(band, ny - g.top);
    g.left = (int)std::min<int64_t>(band, nx);
    g.right = (int)std::min<int64_t>(band, nx - g.left);
    const int64_t mid = ny - g.top - g.bot;
    g.h = (int)((nx + len - 1) / len);
    g.v = (int)((mid + len - 1) / len);
    g.n_h = g.h * (1 + (g.bot > 0));
    g.n_v = g.v * (1 + (g.right > 0));
    return g;
}

// Outputs of a piece along its strip: 128, halved down to 32 while that still leaves a CTA per SM at
// most.  A piece is one CTA's work, and in FP64 bound by its SM's two FMAs per cycle: exact splitting,
// Box-2D3R t = 2 on 300 x 200, eight steps: 309 us with 128, 277 us with the small tiles before pieces.
inline int band_length(int64_t ny, int64_t nx, int band, int sms)
{
    int len = 128;
    while (len > 32) {
        const BandPieces g = band_pieces(ny, nx, band, len / 2);
        if (g.n_h + g.n_v > sms) break;
        len /= 2;
    }
    return len;
}

}  // namespace gbs
