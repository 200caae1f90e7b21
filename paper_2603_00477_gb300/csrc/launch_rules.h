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
// 18,150 us for four sweeps against 14,580 us with 29 planes and 16,060 us with 64).
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

}  // namespace gbs
