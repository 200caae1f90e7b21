// k_band.cu -- the band fix-up of a fused tensor-core sweep: the interior
// points within (t-1) r of the boundary, computed stepwise on CUDA cores (the
// composite kernel is exact only farther in, because the fixed halo has to be
// re-imposed between the steps).
//
// The band is four thin strips: `band` rows along the top and bottom over the
// whole width, `band` columns at the left and right of the rows between.  A
// CTA takes a piece of 32 to 128 outputs along a strip, stages the piece grown
// by t r on every side and runs the t sub-steps in shared memory (ping-pong
// between two buffers), the last one straight to global memory.  The work is
// a few thousand points per CTA and bound by latency (t + 1 barriers), so what
// counts is that every SM has a piece and no piece stages more than it needs:
// tiles of the main CUDA-core sweep (64 x 128 for a band of 6 points) took
// 98 us for Box-2D2R FP32 at t = 4 on 16384^2, this form 18 us.
#include <algorithm>

#include "cu_kernels.cuh"
#include "launch.h"
#include "launch_rules.h"

namespace gbs {
namespace {

constexpr int kBandThreads = 256;
constexpr int kBandV = 4;         // outputs of a thread (rows of a column)

struct BandGeom {
    int64_t ny, nx;  // interior extents
    int len;         // outputs of a piece along its strip (band_length)
    BandPieces p;
};

template <typename T, int SHAPE, int R>
__global__ void __launch_bounds__(kBandThreads)
    cu2d_band(const T *in, T *__restrict__ out,
              const __grid_constant__ cu::Weights<T, cu::Taps<SHAPE, 2, R>::K> wt, int64_t Ex, int t,
              const BandGeom g)
{
    cu::chain_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the piece: interior rows [iy0, iy0 + BY), columns [ix0, ix0 + BX)
    int64_t iy0, ix0;
    int BY, BX;
    const int id = blockIdx.x;
    if (id < g.p.n_h) {
        const bool bottom = id >= g.p.h;
        BY = bottom ? g.p.bot : g.p.top;
        iy0 = bottom ? g.ny - g.p.bot : 0;
        ix0 = (int64_t)(bottom ? id - g.p.h : id) * g.len;
        BX = (int)min((int64_t)g.len, g.nx - ix0);
    } else {
        const int v = id - g.p.n_h;
        const bool right = v >= g.p.v;
        BX = right ? g.p.right : g.p.left;
        ix0 = right ? g.nx - g.p.right : 0;
        iy0 = g.p.top + (int64_t)(right ? v - g.p.v : v) * g.len;
        BY = (int)min((int64_t)g.len, g.ny - g.p.bot - iy0);
    }
    const int64_t Ey = g.ny + 2 * R;
    const int H = BY + 2 * t * R, W = BX + 2 * t * R;
    const int64_t Y0 = iy0 + R - (int64_t)t * R, X0 = ix0 + R - (int64_t)t * R;  // stored coordinates of (0, 0)
    T *src = reinterpret_cast<T *>(smem_raw), *dst = src + H * W;
    const int tid = threadIdx.x;
    // cells outside the stored array are zero and never used by an interior point
    for (int e = tid; e < H * W; e += kBandThreads) {
        const int y = e / W, x = e - (e / W) * W;
        const int64_t gy = Y0 + y, gx = X0 + x;
        src[e] = (gy >= 0 && gy < Ey && gx >= 0 && gx < Ex) ? __ldcg(in + gy * Ex + gx) : T(0);
    }
    __syncthreads();
    for (int s = 1; s <= t; ++s) {
        const int lo = s * R, hiY = H - s * R, hiX = W - s * R;
        const int cw = hiX - lo, strips = (hiY - lo + kBandV - 1) / kBandV;
        const bool last = s == t;
        for (int item = tid; item < cw * strips; item += kBandThreads) {
            const int x = lo + item % cw, y0 = lo + (item / cw) * kBandV;
            T acc[kBandV];
#pragma unroll
            for (int j = 0; j < kBandV; ++j) acc[j] = T(0);
#pragma unroll
            for (int q = 0; q < kBandV + 2 * R; ++q) {
                const int yy = y0 - R + q;
                if (yy < H) {
                    const T *row = src + yy * W + x;
                    T v[2 * R + 1];
#pragma unroll
                    for (int c = 0; c < 2 * R + 1; ++c) v[c] = row[c - R];
#pragma unroll
                    for (int j = 0; j < kBandV; ++j) {
                        const int oy = q - R - j;
                        if (oy >= -R && oy <= R) {
#pragma unroll
                            for (int ox = -R; ox <= R; ++ox) {
                                const int k = cu::tap_index<SHAPE, 2, R>(0, oy, ox);
                                if (k >= 0) acc[j] = fma(wt.w[k], v[ox + R], acc[j]);
                            }
                        }
                    }
                }
            }
            const int64_t gx = X0 + x;
            const bool colint = gx >= R && gx < Ex - R;
#pragma unroll
            for (int j = 0; j < kBandV; ++j) {
                const int y = y0 + j;
                if (y < hiY) {
                    const int64_t gy = Y0 + y;
                    const bool interior = colint && gy >= R && gy < Ey - R;
                    if (last) {
                        if (interior) out[gy * Ex + gx] = acc[j];
                    } else {
                        dst[y * W + x] = interior ? acc[j] : src[y * W + x];
                    }
                }
            }
        }
        __syncthreads();
        // the staged input is not needed after the first sub-step
        T *tmp = src;
        src = dst;
        dst = tmp;
    }
    // not at the start: the next sweep's blocks, placed among these, ran it 5 % slower
    // (f16 on 16384^2, 994 -> 1035 us for 8 steps; 979 us from here)
    cu::chain_next();
}

template <typename T, int SHAPE, int R>
stencil_status launch_band_n(const Plan &p, const void *in, void *out, int t, int band, cudaStream_t st)
{
    using Wt = cu::Weights<T, cu::Taps<SHAPE, 2, R>::K>;
    Wt wt;
    for (int k = 0; k < cu::Taps<SHAPE, 2, R>::K; k++) wt.w[k] = (T)p.w[k];
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    BandGeom g{p.dims[1], p.dims[2], band_length(p.dims[1], p.dims[2], band, std::max(1, sms)), {}};
    g.p = band_pieces(g.ny, g.nx, band, g.len);
    const size_t smem = (size_t)(band + 2 * t * R) * (g.len + 2 * t * R) * sizeof(T) * 2;
    if (smem > 227 * 1024) return fail(STENCIL_ERR_UNSUPPORTED, "CUDA-core band does not fit in shared memory");
    auto kern = cu2d_band<T, SHAPE, R>;
    stencil_status s = ensure_smem((const void *)kern, smem);
    if (s != STENCIL_OK) return s;
    const cudaError_t e = launch_chained(kern, (unsigned)(g.p.n_h + g.p.n_v), kBandThreads, smem, st, (const T *)in,
                                         (T *)out, wt, p.ext[2], t, g);
    if (e == cudaSuccess) note_launch();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "cu2d_band launch");
}

template <typename T, int SHAPE>
stencil_status launch_band_r(const Plan &p, const void *in, void *out, int t, int band, cudaStream_t st)
{
    switch (p.pat.r) {  // t > 1 and t r <= 12
    case 1: return launch_band_n<T, SHAPE, 1>(p, in, out, t, band, st);
    case 2: return launch_band_n<T, SHAPE, 2>(p, in, out, t, band, st);
    case 3: return launch_band_n<T, SHAPE, 3>(p, in, out, t, band, st);
    case 4: return launch_band_n<T, SHAPE, 4>(p, in, out, t, band, st);
    case 5: return launch_band_n<T, SHAPE, 5>(p, in, out, t, band, st);
    case 6: return launch_band_n<T, SHAPE, 6>(p, in, out, t, band, st);
    }
    return fail(STENCIL_ERR_UNSUPPORTED, "band sweep: no kernel for this radius");
}

}  // namespace

stencil_status launch_cu_band(const Plan &p, const void *in, void *out, int t, int band, cudaStream_t st)
{
    if (p.pat.d != 2) return fail(STENCIL_ERR_UNSUPPORTED, "band sweep: 2-D only");
    if (p.dtype == STENCIL_F64)
        return p.pat.shape == STENCIL_BOX ? launch_band_r<double, 0>(p, in, out, t, band, st)
                                          : launch_band_r<double, 1>(p, in, out, t, band, st);
    return p.pat.shape == STENCIL_BOX ? launch_band_r<float, 0>(p, in, out, t, band, st)
                                      : launch_band_r<float, 1>(p, in, out, t, band, st);
}

}  // namespace gbs
