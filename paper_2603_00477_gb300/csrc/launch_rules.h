// launch_rules.h -- how the launchers cut a grid into work items (plain host arithmetic, no CUDA).
#pragma once

#include <algorithm>
#include <cstdint>

namespace gbs {

// Output planes per work item of the 3-D streaming kernel (`cols` tiles of a plane
// side by side, `occ` resident CTAs per SM).  The FMA pipe is the bound and an SM's
// CTAs share it, so a sweep takes about (items of the busiest SM) x (planes + a start-up
// worth one plane).  Up to one wave the CTAs are spread evenly; beyond it the persistent
// CTAs that take one item more share an SM as soon as they are more than ~4/5 of the SMs
// (the block scheduler fills the smaller GPCs twice before the larger ones once): 448
// items on 304 CTAs are four on some SMs, not three (Box-3D2R FP64 256^3, 37 planes:
// 18,150 us for four sweeps against 14,030 us with 29 planes and 16,060 us with 64).
// 64 planes whatever the grid: Box-3D1R FP64 256^3 908 us per sweep, 778 us with 37.
inline int64_t stream_planes(int64_t nz, int64_t cols, int occ, int sms)
{
    const int64_t wave = (int64_t)occ * sms;
    int64_t best = nz, best_cost = -1;
    for (int64_t n = 1; n <= std::min<int64_t>(nz, 64); n++) {
        const int64_t c = (nz + n - 1) / n, items = (nz + c - 1) / c * cols;
        const int64_t full = items / wave, rest = items % wave;
        int64_t busiest = occ * full;
        if (full == 0) busiest = (rest + sms - 1) / sms;
        else if (rest > 0) busiest += std::min<int64_t>(occ, (5 * rest + 4 * sms - 1) / (4 * sms));
        const int64_t cost = busiest * (c + 1);
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

}  // namespace gbs
