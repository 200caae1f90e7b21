// k_cuda_core_impl.cuh -- host launchers of the CUDA-core sweeps
// (templates; instantiated in k_cu2d_*.cu and k_cu3d.cu so that the
// instantiations compile in parallel).
#pragma once

#include <algorithm>
#include <string>

#include "cu_kernels.cuh"
#include "launch.h"
#include "launch_rules.h"

namespace gbs {
namespace cuimpl {


template <typename T>
constexpr int kV = sizeof(T) == 8 ? 4 : 8;  // strip height: FP64 needs fewer accumulators
constexpr size_t kMaxSmem = 227 * 1024;

// 2-D FP32, t = 1 or 2, radius <= 3: the marching kernel.  The segment of output
// rows per work item is chosen so that the items fill k = 1 .. 4 rounds of the
// resident warps: the time is ~ k (segment + 2 t r + a start-up of ~12 rows).
template <int SHAPE, int R, int T, bool VEC>
stencil_status launch2d_march(const Plan &p, const void *in, void *out, cudaStream_t st)
{
    using Wt = cu::Weights<float, cu::Taps<SHAPE, 2, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 2, R>::K; k++) wt.w[k] = (float)p.w[k];
    auto kern = cu::cu2d_march<SHAPE, R, T, VEC>;
    int occ = 0;
    stencil_status s = occupancy((const void *)kern, cu::kMarchThreads, 0, &occ);
    if (s != STENCIL_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int CW = cu::march_cols<R, T>();
    const int xb = R - R % 4;  // quads start on 16-byte boundaries of aligned rows
    const int64_t ny = p.dims[1], ncb = (p.ext[2] - R - xb + CW - 1) / CW;
    const int64_t warps = (int64_t)std::max(1, occ) * std::max(1, sms) * (cu::kMarchThreads / 32);
    int64_t seg = 0, best = 0;
    for (int64_t k = 1; k <= 4; k++) {
        const int64_t nseg = std::min(ny, k * warps / ncb);
        if (nseg < 1) continue;
        const int64_t c = (ny + nseg - 1) / nseg, cost = k * (c + 2 * R * T + 12);
        if (seg == 0 || cost < best) {
            best = cost;
            seg = c;
        }
    }
    if (seg == 0) seg = ny;  // more column blocks than four rounds hold
    const int64_t items = ncb * ((ny + seg - 1) / seg);
    if (items > 0x7fffffff || seg > 0x3fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const int64_t per_cta = cu::kMarchThreads / 32;
    const unsigned grid =
        (unsigned)std::min<int64_t>((items + per_cta - 1) / per_cta, (int64_t)std::max(1, occ) * std::max(1, sms));
    const cudaError_t e = launch_chained(kern, grid, cu::kMarchThreads, 0, st, (const float *)in,
                                         (float *)out, wt, p.ext[1], p.ext[2], (int)ncb, (int)seg, (int)items, xb);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu2d_march launch");
}

template <typename T, int SHAPE, int R>
stencil_status launch2d(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    using Wt = cu::Weights<T, cu::Taps<SHAPE, 2, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 2, R>::K; k++) wt.w[k] = (T)p.w[k];
    const int *tile = p.tile;
    if constexpr (sizeof(T) == 4 && R <= 3) {
        // a tile asked for by option or picked by the autotuner runs the tiled kernel
        int def[3];
        cu_default_tile(p, p.t, def);
        if (t <= 2 && tile[1] == def[1] && tile[2] == def[2] &&
            !tiles_beat_march(SHAPE, R, t, p.dims[1], p.dims[2], tile[1], tile[2])) {
            const bool vec = p.ext[2] % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0 &&
                             reinterpret_cast<uintptr_t>(out) % 16 == 0;
            if (t == 1)
                return vec ? launch2d_march<SHAPE, R, 1, true>(p, in, out, st)
                           : launch2d_march<SHAPE, R, 1, false>(p, in, out, st);
            if constexpr (cu::march_has<SHAPE, R, 2>())
                return vec ? launch2d_march<SHAPE, R, 2, true>(p, in, out, st)
                           : launch2d_march<SHAPE, R, 2, false>(p, in, out, st);
        }
    }
    const int BY = tile[1], BX = tile[2];
    const size_t H = BY + 2 * t * R, W = BX + 2 * t * R;
    const size_t bufb = cu::buf_elems<T>((int)H, (int)W) * sizeof(T);
    // weights (FP64) + two staging buffers (+ a work buffer for t > 1)
    const size_t smem = cu::weight_smem_bytes<T, cu::Taps<SHAPE, 2, R>::K>() + bufb * (t > 1 ? 3 : 2);
    if (smem > kMaxSmem) return fail(STENCIL_ERR_UNSUPPORTED, "CUDA-core tile does not fit in shared memory");
    auto kern = cu::cu2d_sweep<T, SHAPE, R, kV<T>>;
    stencil_status s = ensure_smem((const void *)kern, smem);
    if (s != STENCIL_OK) return s;
    int occ_blocks = 0;
    s = occupancy((const void *)kern, cu::kThreads, smem, &occ_blocks);
    if (s != STENCIL_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cu::Tiles tiles{};
    if (sizeof(T) == 4 && p.ext[2] % 4 == 0 && BX % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0) {
        // shift the tile grid left so that each staged window starts on a
        // 16-byte boundary (window start = R + bx BX - t R - xshift)
        tiles.xshift = (int)(((int64_t)R * (1 - t) % 4 + 4) % 4);
        tiles.vec16 = 1;
    }
    tiles.ntx = (int)((p.dims[2] + tiles.xshift + BX - 1) / BX);
    const int64_t ntiles = (p.dims[1] + BY - 1) / BY * tiles.ntx;
    if (ntiles > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    if (sizeof(T) == 8) occ_blocks = f64_tile_ctas(ntiles, std::max(1, occ_blocks), std::max(1, sms));
    const int64_t resident = (int64_t)std::max(1, occ_blocks) * std::max(1, sms);
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles, resident);
    tiles.next_early = next_sweep_early(sizeof(T) == 8, R, t, ntiles, resident);
    const cudaError_t e = launch_chained(kern, grid, cu::kThreads, smem, st, (const T *)in, (T *)out, wt,
                                         p.ext[1], p.ext[2], BY, BX, t, tiles, (int)ntiles);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu2d_sweep launch");
}

// 3-D, t = 1: the streaming kernel (tile 16 RPT x 64 in y, x; chunks of
// planes in z).
template <typename T, int SHAPE, int R>
stencil_status launch3d_stream(const Plan &p, const void *in, void *out, cudaStream_t st)
{
    using Wt = cu::Weights<T, cu::Taps<SHAPE, 3, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 3, R>::K; k++) wt.w[k] = (T)p.w[k];
    const size_t smem = cu::stream_smem_bytes<T, R>(cu::Taps<SHAPE, 3, R>::K);
    if (smem > kMaxSmem) return fail(STENCIL_ERR_UNSUPPORTED, "3-D streaming tile does not fit in shared memory");
    auto kern = cu::cu3d_stream<T, SHAPE, R>;
    stencil_status s = ensure_smem((const void *)kern, smem);
    if (s != STENCIL_OK) return s;
    int occ = 0;
    s = occupancy((const void *)kern, cu::kThreads, smem, &occ);
    if (s != STENCIL_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int BY = 16 * cu::stream_rows_per_thread<T>(), BX = 64;
    const int64_t tyy = (p.dims[1] + BY - 1) / BY, txx = (p.dims[2] + BX - 1) / BX, nz = p.dims[0];
    const int64_t cz = stream_planes(nz, tyy * txx, std::max(1, occ), std::max(1, sms));
    const int64_t items = (nz + cz - 1) / cz * tyy * txx;
    if (items > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const unsigned grid = (unsigned)std::min<int64_t>(items, (int64_t)std::max(1, occ) * std::max(1, sms));
    const cudaError_t e = launch_chained(kern, grid, cu::kThreads, smem, st, (const T *)in, (T *)out, wt,
                                         p.ext[0], p.ext[1], p.ext[2], (int)txx, (int)tyy, (int)cz, (int)items);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu3d_stream launch");
}

// 3-D, t = 1, FP32: z-marching with rotating partial sums (cu3d_rot).
template <int SHAPE, int R, bool VEC>
stencil_status launch3d_rot(const Plan &p, const void *in, void *out, cudaStream_t st)
{
    using Wt = cu::Weights<float, cu::Taps<SHAPE, 3, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 3, R>::K; k++) wt.w[k] = (float)p.w[k];
    const int xb = R - R % 4;  // the first tile's first column: a multiple of 4
    const cu::RotTile tile =
        cu::rot_tile<R, cu::rot_rows_per_thread<SHAPE, R>()>(p.dims[1], p.dims[2] + R - xb, VEC);
    if (tile.nq == 0 || tile.smem > kMaxSmem)
        return fail(STENCIL_ERR_UNSUPPORTED, "3-D marching tile does not fit in shared memory");
    auto kern = cu::cu3d_rot<SHAPE, R, VEC>;
    stencil_status s = ensure_smem((const void *)kern, tile.smem);
    if (s != STENCIL_OK) return s;
    int occ = 0;
    s = occupancy((const void *)kern, cu::kThreads, tile.smem, &occ);
    if (s != STENCIL_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t nz = p.dims[0], cols = (int64_t)tile.tiles_x * tile.tiles_y;
    const int64_t slots = (int64_t)std::max(1, occ) * std::max(1, sms);
    const int64_t cz = rot_planes(nz, cols, R, std::max(1, occ), std::max(1, sms));
    const int64_t items = ((nz + cz - 1) / cz) * cols;
    if (items > 0x7fffffff || cz > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const unsigned grid = (unsigned)std::min<int64_t>(items, slots);
    const cudaError_t e = launch_chained(kern, grid, cu::kThreads, tile.smem, st, (const float *)in,
                                         (float *)out, wt, p.ext[0], p.ext[1], p.ext[2], tile.nq, tile.ns,
                                         tile.tiles_x, tile.tiles_y, (int)items, (int)cz, xb);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu3d_rot launch");
}

template <typename T, int SHAPE, int R>
stencil_status launch3d(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    if (t == 1) {
        // FP32 star r <= 3 and box r = 1 with planes of 32-bit offsets: rotating partial sums; the rest streams
        if constexpr (sizeof(T) == 4 && ((SHAPE == 1 && R <= 3) || (SHAPE == 0 && R == 1)))
            if (rot3d_plane_fits(p.ext[1], p.ext[2]))
                return p.ext[2] % 4 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0 &&
                               reinterpret_cast<uintptr_t>(out) % 16 == 0
                           ? launch3d_rot<SHAPE, R, true>(p, in, out, st)
                           : launch3d_rot<SHAPE, R, false>(p, in, out, st);
        return launch3d_stream<T, SHAPE, R>(p, in, out, st);
    }
    using Wt = cu::Weights<T, cu::Taps<SHAPE, 3, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 3, R>::K; k++) wt.w[k] = (T)p.w[k];
    const int *tile = p.tile;
    const int BZ = tile[0], BY = tile[1], BX = tile[2];
    const size_t Z = BZ + 2 * t * R, H = BY + 2 * t * R, W = BX + 2 * t * R;
    const size_t smem =
        cu::weight_smem_bytes<T, cu::Taps<SHAPE, 3, R>::K>() + Z * H * W * sizeof(T) * (t > 1 ? 3 : 2);
    if (smem > kMaxSmem) return fail(STENCIL_ERR_UNSUPPORTED, "CUDA-core tile does not fit in shared memory");
    auto kern = cu::cu3d_sweep<T, SHAPE, R, kV<T>>;
    stencil_status s = ensure_smem((const void *)kern, smem);
    if (s != STENCIL_OK) return s;
    int occ_blocks = 0;
    s = occupancy((const void *)kern, cu::kThreads, smem, &occ_blocks);
    if (s != STENCIL_OK) return s;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t nz = p.dims[0], ny = p.dims[1], nx = p.dims[2];
    const int64_t tx = (nx + BX - 1) / BX, ty = (ny + BY - 1) / BY, tz = (nz + BZ - 1) / BZ;
    const int64_t ntiles = tx * ty * tz;
    if (ntiles > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const int64_t resident = (int64_t)std::max(1, occ_blocks) * std::max(1, sms);
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles, resident);
    const cudaError_t e = launch_chained(kern, grid, cu::kThreads, smem, st, (const T *)in, (T *)out, wt,
                                         p.ext[0], p.ext[1], p.ext[2], BZ, BY, BX, t, (int)tx, (int)ty, (int)ntiles);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu3d_sweep launch");
}


// Launcher of one (dtype, shape) group for the radii RLO..RHI.
template <typename T, int SHAPE, int RLO, int RHI>
stencil_status launch2d_range(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    if constexpr (RLO <= RHI) {
        if (p.pat.r == RLO) return launch2d<T, SHAPE, RLO>(p, in, out, t, st);
        return launch2d_range<T, SHAPE, RLO + 1, RHI>(p, in, out, t, st);
    }
    return fail(STENCIL_ERR_UNSUPPORTED, "no CUDA-core kernel for this (shape, d, r)");
}

}  // namespace cuimpl

// One translation unit each (the large FP32 radii compile longest, so they
// are split by radius).
stencil_status launch_cu2d_f32_box_r13(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f32_box_r45(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f32_box_r6(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f32_box_r7(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f32_star_r14(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f32_star_r57(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu2d_f64(const Plan &p, const void *in, void *out, int t, cudaStream_t st);
stencil_status launch_cu3d(const Plan &p, const void *in, void *out, int t, cudaStream_t st);

}  // namespace gbs
