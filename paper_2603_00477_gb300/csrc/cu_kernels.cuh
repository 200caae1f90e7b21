// cu_kernels.cuh -- CUDA-core stencil sweeps with temporal blocking.
//
// Paper Sec. 3.2.2 (CUDA cores with temporal fusion): t steps are fused in
// one pass over the grid; the intermediate steps never leave the SM, so the
// HBM traffic per point stays one read and one write (M = 2D) while the
// arithmetic grows to t * 2K (Eq. 8).
//
// One CTA owns an output tile.  It stages the tile grown by t*r on every
// side (the dependency region of t steps) from global memory into shared
// memory, then runs the t sub-steps in shared memory (ping-pong between two
// buffers); sub-step s computes the region grown by (t - s) r.  Points that
// are not interior (the fixed halo, or outside the stored array) keep their
// value, which re-imposes the Dirichlet boundary after every sub-step.  The
// last sub-step writes straight to global memory.  FP64 (and 3-D): each
// thread computes a strip of V outputs along the slowest tile axis and reuses
// every loaded input row/plane across the strip from registers.  FP32 2-D:
// each thread walks a strip of rows for four adjacent columns and rotates
// the partial sums of the 2r+1 output rows an input row touches through
// registers (f32_substep4).
//
// Weights are kernel parameters (constant bank; FP64 kernels copy them to
// shared memory), K values in the library's lexicographic offset order.
#pragma once

#include <cstdint>
#include <type_traits>
#include <utility>

#include <cuda_runtime.h>

namespace gbs {
namespace cu {

constexpr int kThreads = 256;

template <int SHAPE, int D, int R>
struct Taps {
    static constexpr int side = 2 * R + 1;
    static constexpr int K = SHAPE == 0 ? (D == 2 ? side * side : side * side * side) : 2 * D * R + 1;
};

// Index of offset (oz, oy, ox) in the lexicographic offset list, -1 if the
// offset is not part of the pattern.  D == 2 ignores oz.
template <int SHAPE, int D, int R>
__host__ __device__ constexpr int tap_index(int oz, int oy, int ox)
{
    if (SHAPE == 0) {
        return D == 2 ? (oy + R) * (2 * R + 1) + (ox + R)
                      : ((oz + R) * (2 * R + 1) + (oy + R)) * (2 * R + 1) + (ox + R);
    }
    const int nz = (D == 3 && oz != 0) + (oy != 0) + (ox != 0);
    if (nz > 1) return -1;
    if (D == 2) {
        if (oy < 0) return oy + R;
        if (oy == 0) return 2 * R + ox;
        return 3 * R + oy;
    }
    if (oz < 0) return oz + R;
    if (oz == 0) {
        if (oy < 0) return R + oy + R;
        if (oy == 0) return 3 * R + ox;
        return 4 * R + oy;
    }
    return 5 * R + oz;
}

template <typename T, int K>
struct Weights {
    T w[K];
};

// ---------------------------------------------------------------------------
// 2-D: tile BY x BX, strips of V rows.
// ---------------------------------------------------------------------------
struct Tiles {
    int ntx;         // tiles along x (row-major tile order)
    int xshift;      // FP32: the tile grid starts xshift columns further left so that every
                     // staged window begins on a 16-byte boundary (then vec16 = 1)
    int vec16;       // stage interior tiles with 16-byte copies
    int next_early;  // chain_next at the start (next_sweep_early)
};

// Asynchronous global -> shared copy of one element (cp.async, L1-allocating);
// src_bytes = 0 writes zeros without reading global memory.
template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void *smem_dst, const void *gmem_src, bool valid)
{
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
    const int n = valid ? BYTES : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(gmem_src), "n"(BYTES), "r"(n)
                 : "memory");
}

// Sweeps of a run follow each other on one stream, each reading what the last
// wrote (launch_chained).  A sweep touches no global memory before the one in front
// of it is complete and its writes are visible (chain_wait); it lets the next one's
// blocks take their places (chain_next) as soon as its own have all started, or,
// where a sweep is bound by the FMA pipes, when their work is done: blocks placed
// earlier pile up on the SMs that finish first.  (FP64 Box-2D3R on 600 x 500, ten
// sweeps: 296 us unchained, 403 us with chain_next at the start.)  The tiled 2-D kernel
// has either (next_sweep_early).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// f(integral_constant<int, 0>), f(<1>), ... f(<N-1>) while f returns true:
// a loop whose index is a compile-time constant in the body.
template <typename F, int... I>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, I...>)
{
    (void)(f(std::integral_constant<int, I>{}) && ...);
}
template <int N, typename F>
__device__ __forceinline__ void static_for(F &&f)
{
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// FP32 sub-step, register-rotation form.  A work item is a pair of adjacent
// columns (x, x+1) and a strip of S output rows.  The thread walks down the
// strip's input rows once; each row window is read with 8-byte shared loads
// (D = parity of the window start) and added to the 2R+1 output rows it
// touches, whose partial sums rotate through 2R+1 register slots.  The row
// loop is unrolled by 2R+1, so every slot index and weight index is a
// compile-time constant and no FMA carries a condition; output row jj is
// complete after input row jj + 2R and is stored from its slot.  `fast`: the
// whole region is interior and the stores skip the boundary tests.
template <int SHAPE, int R, int D, typename WT>
__device__ __forceinline__ void f32_substep(const float *__restrict__ src, float *__restrict__ dst,
                                            float *__restrict__ out, const WT &wt, int W, int H, int lo, int hiY,
                                            int hiX, int64_t Y0, int64_t X0, int64_t Ey, int64_t Ex, bool last,
                                            bool fast)
{
    constexpr int NS = 2 * R + 1;      // rotating slots
    constexpr int NV = 2 * R + 2 + D;  // window values per row
    constexpr int NL = (NV + 1) / 2;   // float2 loads per row
    const int cw = hiX - lo, ch = hiY - lo;
    const int npairs = (cw + 1) / 2;
    // strips of ~16 rows (the 2R extra input rows per strip are the only
    // redundant work), enough of them to give every thread work
    const int nstrips = max(1, min((ch + 15) / 16, (int)((blockDim.x + npairs - 1) / npairs)));
    const int S = (ch + nstrips - 1) / nstrips;
    auto store = [&](int y, int x, float v0, float v1, bool second) {
        if (fast) {
            if (last) {
                float *o = out + (Y0 + y) * Ex + (X0 + x);
                if (second && ((reinterpret_cast<uintptr_t>(o) & 7) == 0)) {
                    *reinterpret_cast<float2 *>(o) = make_float2(v0, v1);
                } else {
                    o[0] = v0;
                    if (second) o[1] = v1;
                }
            } else {
                // W is even, so dst + y*W + x is 8-byte aligned exactly when x is
                // even (x has the parity of s*R: uniform over the sub-step)
                float *o = dst + y * W + x;
                if (second && (x & 1) == 0) {
                    *reinterpret_cast<float2 *>(o) = make_float2(v0, v1);
                } else {
                    o[0] = v0;
                    if (second) o[1] = v1;
                }
            }
            return;
        }
        const int64_t gy = Y0 + y, gx = X0 + x;
        const bool rowint = gy >= R && gy < Ey - R;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && !second) break;
            const int64_t gxh = gx + h;
            const bool interior = rowint && gxh >= R && gxh < Ex - R;
            const float val = h ? v1 : v0;
            if (last) {
                if (interior) out[gy * Ex + gxh] = val;
            } else {
                dst[y * W + x + h] = interior ? val : src[y * W + x + h];
            }
        }
    };

    for (int item = threadIdx.x; item < nstrips * npairs; item += blockDim.x) {
        const int sy = item / npairs, px = item - sy * npairs;
        const int y0 = lo + sy * S;
        const int yend = min(y0 + S, hiY);  // outputs y0 .. yend-1
        if (y0 >= yend) continue;
        const int x = lo + 2 * px;
        const bool second = x + 1 < hiX;
        const int nrows = (yend - y0) + 2 * R;  // input rows y0-R .. yend-1+R
        float a0[NS], a1[NS];
#pragma unroll
        for (int m = 0; m < NS; ++m) a0[m] = a1[m] = 0.0f;
        const float *col = src + x - R - D;
        for (int base = 0; base < nrows; base += NS) {
#pragma unroll
            for (int u = 0; u < NS; ++u) {
                const int qq = base + u;  // relative input row; absolute row y0 - R + qq
                if (qq < nrows) {
                    const float2 *row = reinterpret_cast<const float2 *>(col + (y0 - R + qq) * W);
                    float v[2 * NL];
#pragma unroll
                    for (int c = 0; c < NL; ++c) {
                        const float2 t2 = row[c];
                        v[2 * c] = t2.x;
                        v[2 * c + 1] = t2.y;
                    }
                    // output jj = qq - e (e = 0..2R) takes this row with oy = e - R
#pragma unroll
                    for (int e = 0; e < NS; ++e) {
                        const int slot = ((u - e) % NS + NS) % NS;
#pragma unroll
                        for (int ox = -R; ox <= R; ++ox) {
                            const int k = tap_index<SHAPE, 2, R>(0, e - R, ox);
                            if (k >= 0) {
                                a0[slot] = fmaf(wt.w[k], v[D + R + ox], a0[slot]);
                                a1[slot] = fmaf(wt.w[k], v[D + R + ox + 1], a1[slot]);
                            }
                        }
                    }
                    // output jj = qq - 2R is complete (slot (u - 2R) mod NS = (u + 1) mod NS)
                    constexpr int dummy = 0;
                    (void)dummy;
                    const int jj = qq - 2 * R;
                    const int done = (u + 1) % NS;
                    if (jj >= 0) store(y0 + jj, x, a0[done], a1[done], second);
                    a0[done] = 0.0f;
                    a1[done] = 0.0f;
                }
            }
        }
    }
}

// Row pitch of a staged tile row of width W and the elements of one staging
// buffer of H rows: FP32 rows are padded to 16-byte multiples (the 4-column
// sub-step reads them with 16-byte loads) and each buffer has 8 elements of
// slack at its end (the last window of the last row reads past column W).
template <typename T>
__host__ __device__ constexpr int row_pitch(int W)
{
    return sizeof(T) == 4 ? (W + 3) & ~3 : W;
}
template <typename T>
__host__ __device__ constexpr size_t buf_elems(int H, int W)
{
    return (size_t)H * row_pitch<T>(W) + (sizeof(T) == 4 ? 8 : 0);
}

// FP32 sub-step, 4-column register-rotation form.  A work item is a quad of
// adjacent columns (x .. x+3) and a strip of S output rows.  The thread walks
// down the strip's input rows once; each row window (columns x-R-D ..,
// D = (lo-R) mod 4 so the window starts on a 16-byte boundary) is read with
// 16-byte shared loads and added to the 2R+1 output rows it touches, whose
// partial sums rotate through 2R+1 register slots.  The first 2R+1 input rows
// are peeled so that no FMA goes into an output above the strip; the row loop
// is unrolled by 2R+1, so every slot and weight index is a compile-time
// constant.  Output row jj is complete after input row jj + 2R and is stored
// (as two 8-byte or four 4-byte stores, by alignment) from its slot.  P is
// the row pitch of src and dst (a multiple of 4).
template <int SHAPE, int R, int D, typename WT>
__device__ __forceinline__ void f32_substep4(const float *__restrict__ src, float *__restrict__ dst,
                                             float *__restrict__ out, const WT &wt, int P, int lo, int hiY, int hiX,
                                             int64_t Y0, int64_t X0, int64_t Ey, int64_t Ex, bool last,
                                             bool all_interior)
{
    constexpr int NS = 2 * R + 1;          // rotating slots
    constexpr int NV = 2 * R + 4 + D;      // window values per row
    constexpr int NL = (NV + 3) / 4;       // 16-byte loads per row
    const int cw = hiX - lo, ch = hiY - lo;
    const int nquads = (cw + 3) / 4;
    // enough strips to give every thread a work item, each of >= 4 rows
    const int nstrips = max(1, min(max(1, ch / 4), (int)((blockDim.x + nquads - 1) / nquads)));
    const int S = (ch + nstrips - 1) / nstrips;
    const bool fast = all_interior;

    for (int item = threadIdx.x; item < nstrips * nquads; item += blockDim.x) {
        const int sy = item / nquads, qx = item - sy * nquads;
        const int y0 = lo + sy * S;
        const int yend = min(y0 + S, hiY);  // outputs y0 .. yend-1
        if (y0 >= yend) continue;
        const int x = lo + 4 * qx;
        const int nval = min(4, hiX - x);
        const int nrows = (yend - y0) + 2 * R;  // input rows y0-R .. yend-1+R
        const float *col = src + x - R - D;
        // output store of row y (4 values), by alignment and boundary
        auto store = [&](int y, const float (&a)[4]) {
            if (fast && nval == 4) {
                float *o = last ? out + (Y0 + y) * Ex + (X0 + x) : dst + y * P + x;
                const uintptr_t al = reinterpret_cast<uintptr_t>(o) & 15;
                if (al == 0) {
                    *reinterpret_cast<float4 *>(o) = make_float4(a[0], a[1], a[2], a[3]);
                } else if ((al & 7) == 0) {
                    reinterpret_cast<float2 *>(o)[0] = make_float2(a[0], a[1]);
                    reinterpret_cast<float2 *>(o)[1] = make_float2(a[2], a[3]);
                } else {
                    o[0] = a[0];
                    o[1] = a[1];
                    o[2] = a[2];
                    o[3] = a[3];
                }
                return;
            }
            const int64_t gy = Y0 + y;
            const bool rowint = gy >= R && gy < Ey - R;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                if (h >= nval) break;
                const int64_t gx = X0 + x + h;
                const bool interior = rowint && gx >= R && gx < Ex - R;
                if (last) {
                    if (interior) out[gy * Ex + gx] = a[h];
                } else {
                    dst[y * P + x + h] = interior ? a[h] : src[y * P + x + h];
                }
            }
        };
        float acc[NS][4];
#pragma unroll
        for (int m = 0; m < NS; ++m) acc[m][0] = acc[m][1] = acc[m][2] = acc[m][3] = 0.0f;
        // one input row (relative row qq, unrolled position u) into the slots
        // of outputs qq - e for e in [0, e_hi]
        auto row = [&](int qq, int u, int e_hi) {
            const float4 *rp = reinterpret_cast<const float4 *>(col + (y0 - R + qq) * P);
            float v[4 * NL];
#pragma unroll
            for (int c = 0; c < NL; ++c) {
                const float4 t4 = rp[c];
                v[4 * c] = t4.x;
                v[4 * c + 1] = t4.y;
                v[4 * c + 2] = t4.z;
                v[4 * c + 3] = t4.w;
            }
#pragma unroll
            for (int e = 0; e < NS; ++e) {
                if (e > e_hi) continue;
                const int slot = ((u - e) % NS + NS) % NS;
#pragma unroll
                for (int ox = -R; ox <= R; ++ox) {
                    const int k = tap_index<SHAPE, 2, R>(0, e - R, ox);
                    if (k >= 0) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[slot][c] = fmaf(wt.w[k], v[D + R + ox + c], acc[slot][c]);
                    }
                }
            }
        };
        // head: input row u (u <= 2R) feeds only outputs u - e >= 0
#pragma unroll
        for (int u = 0; u < NS; ++u)
            if (u < nrows) row(u, u, u);
        if (2 * R < nrows) {  // output 0 is complete after row 2R (slot 0)
            store(y0, acc[0]);
            acc[0][0] = acc[0][1] = acc[0][2] = acc[0][3] = 0.0f;
        }
        for (int base = NS; base < nrows; base += NS) {
#pragma unroll
            for (int u = 0; u < NS; ++u) {
                const int qq = base + u;
                if (qq < nrows) {
                    row(qq, u, 2 * R);
                    const int jj = qq - 2 * R;  // complete output
                    const int done = (u + 1) % NS;
                    store(y0 + jj, acc[done]);
                    acc[done][0] = acc[done][1] = acc[done][2] = acc[done][3] = 0.0f;
                }
            }
        }
    }
}

// FP32 sub-step, fixed-strip form: the fast case of f32_substep4 (every point
// of the region interior, no band, whole quads: cw a multiple of 4,
// ch >= S).  A work item is a quad of columns and S output rows, S a
// compile-time constant: the S + 2R input rows are unrolled completely, so
// each input row goes exactly into the outputs it touches (no partial sums
// of rows outside the strip, no slot rotation) and every index is a
// constant.  When ch is not a multiple of S the last strip of a column
// starts at hiY - S and overlaps the one above; the overlapping outputs are
// computed twice with identical values.  Stores are 16- or 8-byte vectors
// (the alignment of x0 + x is the same for every item of the sub-step).
template <int SHAPE, int R, int D, int S, typename WT>
__device__ __forceinline__ void f32_substep4_fixed(const float *__restrict__ src, float *__restrict__ dst,
                                                   float *__restrict__ out, const WT &wt, int P, int lo, int hiY,
                                                   int hiX, int64_t Y0, int64_t X0, int64_t Ex, bool last)
{
    constexpr int NV = 2 * R + 4 + D;  // window values per row
    constexpr int NL = (NV + 3) / 4;   // 16-byte loads per row
    constexpr int NR = S + 2 * R;      // input rows per strip
    const int nquads = (hiX - lo) >> 2;
    const int nstrips = (hiY - lo + S - 1) / S;
    const int nitems = nquads * nstrips;
    // outputs: (row y, column x) of the region is obase[off0 + y * pitch + x]
    float *const obase = last ? out : dst;
    const int64_t off0 = last ? Y0 * Ex + X0 : 0;
    const int64_t pitch = last ? Ex : P;
    // element offset of the first output within its 16-byte chunk: the same
    // for every item when the pitch is a multiple of 4 (else scalar stores)
    const int phase = (pitch & 3) ? 1
                                  : (int)(((reinterpret_cast<uintptr_t>(obase) >> 2) +
                                           (uint64_t)(off0 + (int64_t)lo * pitch + lo)) & 3);
    for (int item = threadIdx.x; item < nitems; item += blockDim.x) {
        const int sy = item / nquads, qx = item - sy * nquads;
        const int y0 = min(lo + sy * S, hiY - S);
        const int x = lo + 4 * qx;
        const float4 *rp = reinterpret_cast<const float4 *>(src + (y0 - R) * P + x - R - D);
        const int p4 = P >> 2;
        float acc[S][4];
#pragma unroll
        for (int j = 0; j < S; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            float v[4 * NL];
#pragma unroll
            for (int c = 0; c < NL; ++c) {
                const float4 t4 = rp[q * p4 + c];
                v[4 * c] = t4.x;
                v[4 * c + 1] = t4.y;
                v[4 * c + 2] = t4.z;
                v[4 * c + 3] = t4.w;
            }
            // input row q (row y0 - R + q) feeds outputs j = q - R - oy, oy in [-R, R]
#pragma unroll
            for (int j = 0; j < S; ++j) {
                const int oy = q - R - j;
                if (oy < -R || oy > R) continue;
#pragma unroll
                for (int ox = -R; ox <= R; ++ox) {
                    const int k = tap_index<SHAPE, 2, R>(0, oy, ox);
                    if (k >= 0) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[j][c] = fmaf(wt.w[k], v[D + R + ox + c], acc[j][c]);
                    }
                }
            }
        }
        float *o = obase + (off0 + (int64_t)y0 * pitch + x);
        if (phase == 0) {
#pragma unroll
            for (int j = 0; j < S; ++j)
                *reinterpret_cast<float4 *>(o + j * pitch) = make_float4(acc[j][0], acc[j][1], acc[j][2], acc[j][3]);
        } else if (phase == 2) {
#pragma unroll
            for (int j = 0; j < S; ++j) {
                float2 *o2 = reinterpret_cast<float2 *>(o + j * pitch);
                o2[0] = make_float2(acc[j][0], acc[j][1]);
                o2[1] = make_float2(acc[j][2], acc[j][3]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < S; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) o[j * pitch + c] = acc[j][c];
        }
    }
}

// Selects the window phase D = (lo - R) mod 4 and the strip height (4 or 8)
// of f32_substep4_fixed.
template <int SHAPE, int R, typename WT>
__device__ __forceinline__ void f32_fixed_dispatch(int D, bool s4, const float *__restrict__ src,
                                                   float *__restrict__ dst, float *__restrict__ out, const WT &wt,
                                                   int P, int lo, int hiY, int hiX, int64_t Y0, int64_t X0,
                                                   int64_t Ex, bool last)
{
#define GBS_FIXED(DD)                                                                                          \
    if (s4)                                                                                                    \
        f32_substep4_fixed<SHAPE, R, DD, 4>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last);             \
    else                                                                                                       \
        f32_substep4_fixed<SHAPE, R, DD, 8>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last);
    switch (D) {
    case 0: GBS_FIXED(0) break;
    case 1: GBS_FIXED(1) break;
    case 2: GBS_FIXED(2) break;
    default: GBS_FIXED(3) break;
    }
#undef GBS_FIXED
}

// f32_substep4_fixed with strips of 2 rows (radii 3 and more).
template <int SHAPE, int R, typename WT>
__device__ __forceinline__ void f32_fixed_dispatch2(int D, const float *__restrict__ src, float *__restrict__ dst,
                                                    float *__restrict__ out, const WT &wt, int P, int lo, int hiY,
                                                    int hiX, int64_t Y0, int64_t X0, int64_t Ex, bool last)
{
    switch (D) {
    case 0: f32_substep4_fixed<SHAPE, R, 0, 2>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last); break;
    case 1: f32_substep4_fixed<SHAPE, R, 1, 2>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last); break;
    case 2: f32_substep4_fixed<SHAPE, R, 2, 2>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last); break;
    default: f32_substep4_fixed<SHAPE, R, 3, 2>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex, last); break;
    }
}

// Persistent form: CTA b processes tiles b, b + gridDim.x, ...; while it
// computes one tile it prefetches the next into the other staging buffer
// with cp.async, so the FMA pipe never waits for a synchronous load phase.
// Shared memory: two staging buffers (H x W) and, for t > 1, a work buffer
// for the intermediate sub-steps.
// FP64 kernels read their weights from shared memory (one LDS per FMA is
// free next to the FP64 pipe, and keeping K doubles in registers across the
// persistent loop would spill); FP32 kernels read them from the constant bank.
template <typename T, int K>
__host__ __device__ constexpr int weight_smem_bytes()
{
    return sizeof(T) == 8 ? (int)((K * sizeof(T) + 15) / 16 * 16) : 0;
}

template <typename T, int SHAPE, int R, int V>
__global__ void __launch_bounds__(kThreads, (sizeof(T) == 4 && R <= 3) ? 3 : 2)
    cu2d_sweep(const T *__restrict__ in, T *__restrict__ out,
               const __grid_constant__ Weights<T, Taps<SHAPE, 2, R>::K> wt, int64_t Ey, int64_t Ex, int BY, int BX,
               int t, const Tiles tiles, int ntiles)
{
    if (tiles.next_early) chain_next();
    chain_wait();
    constexpr int KT = Taps<SHAPE, 2, R>::K;
    constexpr bool kSmemW = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *wsm = reinterpret_cast<T *>(smem_raw);
    if (kSmemW) {
        for (int k = threadIdx.x; k < KT; k += blockDim.x) wsm[k] = wt.w[k];
    }
    unsigned char *base = smem_raw + weight_smem_bytes<T, KT>();
    const int H = BY + 2 * t * R, W = BX + 2 * t * R, P = row_pitch<T>(W);
    const size_t buf = buf_elems<T>(H, W);
    T *const stage0 = reinterpret_cast<T *>(base), *const stage1 = stage0 + buf;
    T *work = reinterpret_cast<T *>(base) + 2 * buf;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

    auto origin = [&](int id, int64_t *Y0, int64_t *X0) {
        int by, bx;
        by = id / tiles.ntx;
        bx = id % tiles.ntx;
        *Y0 = R + (int64_t)by * BY - (int64_t)t * R;
        *X0 = R + (int64_t)bx * BX - (int64_t)t * R - tiles.xshift;
    };
    // Stage the dependency region of a tile; cells outside the stored array
    // are zero-filled and never used by an interior point.
    auto prefetch = [&](int id, T *dst) {
        int64_t Y0, X0;
        origin(id, &Y0, &X0);
        if (sizeof(T) == 4 && tiles.vec16 && Y0 >= 0 && X0 >= 0 && Y0 + H <= Ey && X0 + P <= Ex) {
            // 16-byte copies: X0, the row length and the input are 16-byte aligned
            const T *g = in + Y0 * Ex + X0;
            for (int y = warp; y < H; y += nwarps) {
                const T *grow = g + y * Ex;
                T *srow = dst + y * P;
                for (int c = lane; 4 * c < W; c += 32) cp_async_elem<16>(srow + 4 * c, grow + 4 * c, true);
            }
            return;
        }
        if (Y0 >= 0 && X0 >= 0 && Y0 + H <= Ey && X0 + W <= Ex) {
            // the whole region lies in the stored array: no per-element tests
            const T *g = in + Y0 * Ex + X0;
            for (int y = warp; y < H; y += nwarps) {
                const T *grow = g + y * Ex;
                T *srow = dst + y * P;
                for (int x = lane; x < W; x += 32) cp_async_elem<sizeof(T)>(srow + x, grow + x, true);
            }
            return;
        }
        for (int y = warp; y < H; y += nwarps) {
            const int64_t gy = Y0 + y;
            const bool rowok = gy >= 0 && gy < Ey;
            for (int x = lane; x < W; x += 32) {
                const int64_t gx = X0 + x;
                const bool ok = rowok && gx >= 0 && gx < Ex;
                cp_async_elem<sizeof(T)>(dst + y * P + x, ok ? in + gy * Ex + gx : in, ok);
            }
        }
    };

    int cur = 0;
    if ((int)blockIdx.x < ntiles) prefetch(blockIdx.x, stage0);
    cp_async_commit();
    for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
        const int nid = id + gridDim.x;
        if (nid < ntiles) prefetch(nid, cur ? stage0 : stage1);
        cp_async_commit();
        cp_async_wait_group<1>();  // this tile's copies (all but the newest group) have landed
        __syncthreads();
        int64_t Y0, X0;
        origin(id, &Y0, &X0);

        T *src = cur ? stage1 : stage0, *dst = work;
        for (int s = 1; s <= t; ++s) {
            const int lo = s * R;
            const int hiY = H - s * R, hiX = W - s * R;
            const int cw = hiX - lo, ch = hiY - lo;
            const int strips = (ch + V - 1) / V;
            const bool last = s == t;
            if constexpr (sizeof(T) == 4) {
                const bool all_int = Y0 + lo >= R && Y0 + hiY <= Ey - R && X0 + lo >= R && X0 + hiX <= Ex - R;
                if constexpr (R <= 2) {
                    if (all_int && (cw & 3) == 0 && ch >= 8) {
                        // strips of 8 rows, or of 4 when that tiles the region exactly
                        const bool s4 = (ch & 7) != 0 && (ch & 3) == 0;
                        f32_fixed_dispatch<SHAPE, R>((lo - R) & 3, s4, src, dst, out, wt, P, lo, hiY, hiX, Y0, X0,
                                                     Ex, last);
                        __syncthreads();
                        T *tmp = src;
                        src = dst;
                        dst = tmp;
                        continue;
                    }
                } else {
                    // larger radii: strips of 2 rows (each item reads 2 + 2R rows
                    // for 8 outputs: loads stay a few % of the (2R+1)^2 taps, and
                    // the unrolled code stays a few thousand FMAs)
                    if (all_int && (cw & 3) == 0 && ch >= 2) {
                        f32_fixed_dispatch2<SHAPE, R>((lo - R) & 3, src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ex,
                                                      last);
                        __syncthreads();
                        T *tmp = src;
                        src = dst;
                        dst = tmp;
                        continue;
                    }
                }
                switch ((lo - R) & 3) {  // offset of the first window within its 16-byte chunk
                case 0:
                    f32_substep4<SHAPE, R, 0>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ey, Ex, last, all_int);
                    break;
                case 1:
                    f32_substep4<SHAPE, R, 1>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ey, Ex, last, all_int);
                    break;
                case 2:
                    f32_substep4<SHAPE, R, 2>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ey, Ex, last, all_int);
                    break;
                default:
                    f32_substep4<SHAPE, R, 3>(src, dst, out, wt, P, lo, hiY, hiX, Y0, X0, Ey, Ex, last, all_int);
                    break;
                }
                __syncthreads();
                T *tmp = src;
                src = dst;
                dst = tmp;
                continue;
            }
            for (int item = threadIdx.x; item < cw * strips; item += blockDim.x) {
                const int x = lo + item % cw;
                const int y0 = lo + (item / cw) * V;
                T acc[V];
#pragma unroll
                for (int j = 0; j < V; ++j) acc[j] = T(0);
#pragma unroll
                for (int q = 0; q < V + 2 * R; ++q) {
                    const int yy = y0 - R + q;
                    if (yy < H) {
                        const T *row = src + yy * P + x;
                        T v[2 * R + 1];
#pragma unroll
                        for (int c = 0; c < 2 * R + 1; ++c) v[c] = row[c - R];
#pragma unroll
                        for (int j = 0; j < V; ++j) {
                            const int oy = q - R - j;
                            if (oy >= -R && oy <= R) {
#pragma unroll
                                for (int ox = -R; ox <= R; ++ox) {
                                    const int k = tap_index<SHAPE, 2, R>(0, oy, ox);
                                    if (k >= 0) acc[j] = fma(kSmemW ? wsm[k] : wt.w[k], v[ox + R], acc[j]);
                                }
                            }
                        }
                    }
                }
                const int64_t gx = X0 + x;
                const bool colint = gx >= R && gx < Ex - R;
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const int y = y0 + j;
                    if (y < hiY) {
                        const int64_t gy = Y0 + y;
                        const bool interior = colint && gy >= R && gy < Ey - R;
                        if (last) {
                            if (interior) out[gy * Ex + gx] = acc[j];
                        } else {
                            dst[y * P + x] = interior ? acc[j] : src[y * P + x];
                        }
                    }
                }
            }
            __syncthreads();
            // next sub-step reads what this one wrote; the staged input is no
            // longer needed after the first sub-step, so it becomes the target
            T *tmp = src;
            src = dst;
            dst = tmp;
        }
        cur ^= 1;
    }
    cp_async_wait_group<0>();
    if (!tiles.next_early) chain_next();
}

// ---------------------------------------------------------------------------
// 2-D FP32, t = 1 or 2, radius <= 3: a warp marches down a strip of columns.
// ---------------------------------------------------------------------------
// A work item is one warp's: 128 columns (one 16-byte quad per lane) and a
// segment of output rows.  Each input row is read once, kMarchDepth - 1 rows
// ahead, by cp.async into a ring of the warp's own; a lane reads its own quad
// back, gets the R columns left and right of it from the neighbouring lanes by
// shuffles, and adds the row into the 2R + 1 output rows it touches, whose
// partial sums rotate through registers (the row loop is unrolled, so every slot
// and weight index is a constant).  A completed row of a fused step is the next
// step's input row.  There is no barrier and no phase: every warp always has
// loads in flight, which is what a stencil bound by HBM needs.  (Loads ahead
// into registers do not do: a warp has six scoreboards, a wait on the oldest
// load then waits for the newest that shares its scoreboard, and the same
// kernel with five rows ahead in registers ran at 551 us where this runs at
// 380 us.)  The price is the edge lanes: a step makes one lane at each end
// invalid, so a warp yields 4 (32 - 2t) columns of its 128.
// Bound by HBM.  Measured, one sweep (tiled kernel below before): Box-2D2R t = 1
// on 16384^2 548 -> 380 us (HBM floor 317, a tiled copy 338); Star-2D2R t = 2 on
// 1021 x 1531 (words, in L2) 18.8 -> 9.8 us.
// Rows that are not 16-byte multiples are copied and stored as four coalesced
// 4-byte words per lane; the shared-memory rows turn them into quads and back.
constexpr int kMarchThreads = 256;

constexpr int kMarchDepth = 8;  // ring rows per warp (a power of two)

// The (shape, radius, depth) triples built: depth 2 where the partial sums and
// weights of two steps fit in registers.
template <int SHAPE, int R, int T>
__host__ __device__ constexpr bool march_has()
{
    return R <= 3 && (T == 1 || (T == 2 && (R <= 2 || SHAPE == 1)));
}

// Columns a warp yields.
template <int R, int T>
__host__ __device__ constexpr int march_cols()
{
    return 4 * (32 - 2 * T);  // R <= 4: one lane per side and step
}

// Resident CTAs per SM the register budget is set for.
template <int SHAPE, int R, int T>
__host__ __device__ constexpr int march_ctas()
{
    return T == 1 ? (R <= 2 ? 3 : 2) : 2;  // K weights and 4 T (2R + 1) partial sums in registers
}

// Floats of shared memory per warp: the ring of input rows and (words only) a
// row on its way out.
template <bool VEC>
__host__ __device__ constexpr int march_warp_floats()
{
    return 128 * (kMarchDepth + (VEC ? 0 : 1));
}

// Whether the products of column pairs run as packed FMAs (fma.rn.f32x2: the same
// two roundings from one issue slot).  They take no constant-bank operand, so
// they pay where the weights are in registers anyway (the batched kernel) or
// where a weight is used often between loads: Box-2D2R at t = 2, 746 us a sweep
// of 16384^2 where the tiled kernel took 1097.  In the other kernels here, which
// read weights from the constant bank, they ran 0 to 10 % slower.
template <int SHAPE, int R, int T>
__host__ __device__ constexpr bool march_packs()
{
    return SHAPE == 0 && R == 2 && T == 2;
}

// One work item of a warp: output rows [y0, y1), the cw <= march_cols columns
// from w0 + 4T on (w0: first column of the 128-column window, a multiple of 4 where VEC).
template <int SHAPE, int R, int T, bool VEC, bool PACK, typename WT>
__device__ __forceinline__ void march_strip(const float *__restrict__ in, float *__restrict__ out, const WT &wt,
                                            int64_t Ey, int64_t Ex, int64_t w0, int64_t y0, int64_t y1, int cw,
                                            float *ring)
{
    constexpr int NS = 2 * R + 1, U = NS, D = kMarchDepth;
    static_assert(R >= 1 && R <= 4, "one quad of halo columns per side and step");
    float *const turn_out = ring + 128 * D;
    const int lane = threadIdx.x & 31;
    const int64_t x = w0 + 4 * lane;  // this lane's columns x .. x + 3
    const int64_t ys = y0 - R * T;  // first input row
    const int nrows = (int)(y1 - y0) + 2 * R * T;
    // interior columns of the quad, and columns this lane stores
    unsigned cint = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) cint |= (x + c >= R && x + c < Ex - R) ? 1u << c : 0u;
    const bool store_lane = lane >= T && lane < T + cw / 4;
    const bool xok = x >= 0 && x < Ex;  // VEC: a quad lies wholly inside or outside a row
    // rows i that exist and are wanted: [i_lo, i_hi)
    const int i_lo = ys < 0 ? (int)-ys : 0, i_hi = (int)min((int64_t)nrows, Ey - ys);
    float *o = out + (ys - R * T) * Ex + (VEC ? x : w0 + lane);  // the row completed after input row i
    const float *src = in + ys * Ex + (VEC ? x : w0 + lane);
    // copy input row ys + i to its ring row (rows and columns outside the stored array become zero)
    auto load = [&](int i) {
        const bool rok = i >= i_lo && i < i_hi;
        float *d = ring + (i & (D - 1)) * 128 + (VEC ? 4 * lane : lane);
        if constexpr (VEC) {
            const bool ok = rok && xok;
            cp_async_elem<16>(d, ok ? src : in, ok);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t gx = w0 + lane + 32 * j;
                const bool ok = rok && gx >= 0 && gx < Ex;
                cp_async_elem<4>(d + 32 * j, ok ? src + 32 * j : in, ok);
            }
        }
        cp_async_commit();
        src += Ex;
    };
    cp_async_wait_group<0>();  // the previous item's rows have landed and are read
    __syncwarp();
    for (int i = 0; i < D - 1; ++i) load(i);
    float2 acc[T][NS][2];
#pragma unroll
    for (int s = 0; s < T; ++s)
#pragma unroll
        for (int m = 0; m < NS; ++m) acc[s][m][0] = acc[s][m][1] = make_float2(0.0f, 0.0f);
    // values of the rows R back, which the fixed boundary keeps (t > 1)
    float hist[T > 1 ? T - 1 : 1][NS][4];
    for (int base = 0; base < nrows; base += U) {
        static_for<U>([&](auto UC) -> bool {
            constexpr int u = decltype(UC)::value;
            const int i = base + u;
            if (i >= nrows) return false;
            cp_async_wait_group<D - 2>();  // row i has landed
            if constexpr (!VEC) __syncwarp();
            float q[4];
            {
                const float4 t4 = *reinterpret_cast<const float4 *>(ring + (i & (D - 1)) * 128 + 4 * lane);
                q[0] = t4.x;
                q[1] = t4.y;
                q[2] = t4.z;
                q[3] = t4.w;
            }
            // row i + D - 1 takes the ring row of row i - 1, whose quads every lane has read
            load(i + D - 1);
            static_for<T>([&](auto SC) -> bool {
                constexpr int s = decltype(SC)::value;   // fused step s + 1; its input row is ys + i - s R
                constexpr int us = ((u - 2 * R * s) % NS + NS) % NS;  // that row's slot phase
                if (s > 0 && i < 2 * R * s) return false;  // no complete row of step s yet
                float v[4 + 2 * R];
#pragma unroll
                for (int c = 0; c < R; ++c) {
                    v[c] = __shfl_up_sync(0xffffffffu, q[c + 4 - R], 1);
                    v[R + 4 + c] = __shfl_down_sync(0xffffffffu, q[c], 1);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) v[R + c] = q[c];
                if constexpr (s < T - 1) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) hist[s][us][c] = q[c];
                }
                // row j (relative) adds into outputs j - e, e = 0 .. 2R, with oy = e - R
#pragma unroll
                for (int e = 0; e < NS; ++e) {
                    const int slot = ((us - e) % NS + NS) % NS;
#pragma unroll
                    for (int ox = -R; ox <= R; ++ox) {
                        const int k = tap_index<SHAPE, 2, R>(0, e - R, ox);
                        if (k >= 0) {
#pragma unroll
                            for (int c = 0; c < 2; ++c) {
                                float2 &a = acc[s][slot][c];
                                const float2 x = make_float2(v[R + ox + 2 * c], v[R + ox + 2 * c + 1]);
                                if constexpr (PACK)
                                    a = __ffma2_rn(make_float2(wt.w[k], wt.w[k]), x, a);
                                else
                                    a = make_float2(fmaf(wt.w[k], x.x, a.x), fmaf(wt.w[k], x.y, a.y));
                            }
                        }
                    }
                }
                // output j - 2R is complete: slot (us + 1) mod NS
                constexpr int done = (us + 1) % NS;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    q[2 * c] = acc[s][done][c].x;
                    q[2 * c + 1] = acc[s][done][c].y;
                    acc[s][done][c] = make_float2(0.0f, 0.0f);
                }
                if constexpr (s < T - 1) {
                    // the halo keeps its value between the fused steps
                    const int64_t y = ys + i - (int64_t)R * (s + 1);  // the completed row
                    const bool rint = y >= R && y < Ey - R;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (!(rint && ((cint >> c) & 1u))) q[c] = hist[s][((us - R) % NS + NS) % NS][c];
                } else if (i >= 2 * R * T) {
                    if constexpr (VEC) {
                        if (store_lane) {
                            if (cint == 0xfu) {
                                *reinterpret_cast<float4 *>(o) = make_float4(q[0], q[1], q[2], q[3]);
                            } else {
#pragma unroll
                                for (int c = 0; c < 4; ++c)
                                    if ((cint >> c) & 1u) o[c] = q[c];
                            }
                        }
                    } else {
                        *reinterpret_cast<float4 *>(turn_out + 4 * lane) = make_float4(q[0], q[1], q[2], q[3]);
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int col = 32 * j + lane;
                            const int64_t gx = w0 + col;
                            if (col >= 4 * T && col < 4 * T + cw && gx >= R && gx < Ex - R)
                                o[32 * j] = turn_out[col];
                        }
                        __syncwarp();
                    }
                }
                return true;
            });
            o += Ex;
            return true;
        });
    }
}

template <int SHAPE, int R, int T, bool VEC>
__global__ void __launch_bounds__(kMarchThreads, (march_ctas<SHAPE, R, T>()))
    cu2d_march(const float *__restrict__ in, float *__restrict__ out,
               const __grid_constant__ Weights<float, Taps<SHAPE, 2, R>::K> wt, int64_t Ey, int64_t Ex, int ncb,
               int seg, int nitems, int xb)
{
    chain_next();
    chain_wait();
    constexpr int CW = march_cols<R, T>();
    __shared__ __align__(16) float smem[(kMarchThreads / 32) * march_warp_floats<VEC>()];
    float *const ring = smem + (threadIdx.x >> 5) * march_warp_floats<VEC>();
    const int nwarps = (int)(gridDim.x * (kMarchThreads / 32));
    for (int item = (int)(blockIdx.x * (kMarchThreads / 32) + (threadIdx.x >> 5)); item < nitems; item += nwarps) {
        const int64_t y0 = R + (int64_t)(item / ncb) * seg;
        march_strip<SHAPE, R, T, VEC, march_packs<SHAPE, R, T>()>(in, out, wt, Ey, Ex, xb + (int64_t)(item % ncb) * CW - 4 * T, y0,
                                      min(y0 + seg, Ey - R), CW, ring);
    }
    cp_async_wait_group<0>();
}

// ---------------------------------------------------------------------------
// 3-D: tile BZ x BY x BX, strips of V planes.
// ---------------------------------------------------------------------------
template <typename T, int SHAPE, int R, int V>
__global__ void __launch_bounds__(kThreads, 2)
    cu3d_sweep(const T *__restrict__ in, T *__restrict__ out,
               const __grid_constant__ Weights<T, Taps<SHAPE, 3, R>::K> wt, int64_t Ez, int64_t Ey, int64_t Ex,
               int BZ, int BY, int BX, int t, int tiles_x, int tiles_y, int ntiles)
{
    chain_wait();
    constexpr int KT = Taps<SHAPE, 3, R>::K;
    constexpr bool kSmemW = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *wsm = reinterpret_cast<T *>(smem_raw);
    if (kSmemW) {
        for (int k = threadIdx.x; k < KT; k += blockDim.x) wsm[k] = wt.w[k];
    }
    unsigned char *base = smem_raw + weight_smem_bytes<T, KT>();
    const int Z = BZ + 2 * t * R, H = BY + 2 * t * R, W = BX + 2 * t * R;
    const int plane = H * W;
    const size_t buf = (size_t)Z * plane;
    T *stage[2] = {reinterpret_cast<T *>(base), reinterpret_cast<T *>(base) + buf};
    T *work = reinterpret_cast<T *>(base) + 2 * buf;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;

    auto origin = [&](int id, int64_t *Z0, int64_t *Y0, int64_t *X0) {
        const int bx = id % tiles_x, by = (id / tiles_x) % tiles_y, bz = id / (tiles_x * tiles_y);
        *Z0 = R + (int64_t)bz * BZ - (int64_t)t * R;
        *Y0 = R + (int64_t)by * BY - (int64_t)t * R;
        *X0 = R + (int64_t)bx * BX - (int64_t)t * R;
    };
    auto prefetch = [&](int id, T *dst) {
        int64_t Z0, Y0, X0;
        origin(id, &Z0, &Y0, &X0);
        for (int zy = warp; zy < Z * H; zy += nwarps) {
            const int z = zy / H, y = zy % H;
            const int64_t gz = Z0 + z, gy = Y0 + y;
            const bool ok = gz >= 0 && gz < Ez && gy >= 0 && gy < Ey;
            const T *row = in + (gz * Ey + gy) * Ex;
            for (int x = lane; x < W; x += 32) {
                const int64_t gx = X0 + x;
                const bool v = ok && gx >= 0 && gx < Ex;
                cp_async_elem<sizeof(T)>(dst + z * plane + y * W + x, v ? row + gx : in, v);
            }
        }
    };

    int cur = 0;
    if ((int)blockIdx.x < ntiles) prefetch(blockIdx.x, stage[0]);
    cp_async_commit();
    for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
        const int nid = id + gridDim.x;
        if (nid < ntiles) prefetch(nid, stage[cur ^ 1]);
        cp_async_commit();
        cp_async_wait_group<1>();
        __syncthreads();
        int64_t Z0, Y0, X0;
        origin(id, &Z0, &Y0, &X0);

        T *src = stage[cur], *dst = work;
        for (int s = 1; s <= t; ++s) {
            const int lo = s * R;
            const int hiZ = Z - s * R, hiY = H - s * R, hiX = W - s * R;
            const int cw = hiX - lo, ch = hiY - lo, cz = hiZ - lo;
            const int strips = (cz + V - 1) / V;
            const bool last = s == t;
            for (int item = threadIdx.x; item < cw * ch * strips; item += blockDim.x) {
                const int x = lo + item % cw;
                const int y = lo + (item / cw) % ch;
                const int z0 = lo + (item / (cw * ch)) * V;
                T acc[V];
#pragma unroll
                for (int j = 0; j < V; ++j) acc[j] = T(0);
#pragma unroll
                for (int q = 0; q < V + 2 * R; ++q) {
                    const int zz = z0 - R + q;
                    if (zz < Z) {
                        const T *pl = src + zz * plane + y * W + x;
#pragma unroll
                        for (int j = 0; j < V; ++j) {
                            const int oz = q - R - j;
                            if (oz >= -R && oz <= R) {
#pragma unroll
                                for (int oy = -R; oy <= R; ++oy) {
#pragma unroll
                                    for (int ox = -R; ox <= R; ++ox) {
                                        const int k = tap_index<SHAPE, 3, R>(oz, oy, ox);
                                        if (k >= 0)
                                            acc[j] = fma(kSmemW ? wsm[k] : wt.w[k], pl[oy * W + ox], acc[j]);
                                    }
                                }
                            }
                        }
                    }
                }
                const int64_t gx = X0 + x, gy = Y0 + y;
                const bool lineint = gx >= R && gx < Ex - R && gy >= R && gy < Ey - R;
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const int z = z0 + j;
                    if (z < hiZ) {
                        const int64_t gz = Z0 + z;
                        const bool interior = lineint && gz >= R && gz < Ez - R;
                        if (last) {
                            if (interior) out[(gz * Ey + gy) * Ex + gx] = acc[j];
                        } else {
                            const int o = z * plane + y * W + x;
                            dst[o] = interior ? acc[j] : src[o];
                        }
                    }
                }
            }
            __syncthreads();
            T *tmp = src;
            src = dst;
            dst = tmp;
        }
        cur ^= 1;
    }
    cp_async_wait_group<0>();
    chain_next();
}

// ---------------------------------------------------------------------------
// 3-D, one step per sweep (t = 1), 2.5-D streaming: a work item is a
// (BY x BX) tile of one z chunk of cz planes.  The CTA marches along z with a
// ring of NP = 2R + 1 + PF input planes (each the tile grown by R in y and x)
// in shared memory: while plane z is computed, planes z + R + 1 ..
// z + R + PF are in flight (cp.async, 16-byte copies where the stored rows
// allow), so every input plane is read once per tile and the only re-reads
// are the y/x halo.  256 threads: thread (ty, tx) = (tid / 16, tid % 16)
// computes outputs (y, x0 .. x0 + 3) for x0 = 4 tx and the RPT rows
// y = ty + 16 i; each (oz, oy) row segment of 4 + 2R values is read with
// 16-byte shared loads (rows padded to 16 bytes) and used for the 4 outputs.
// ---------------------------------------------------------------------------
template <typename T>
__host__ __device__ constexpr int stream_rows_per_thread()
{
    return sizeof(T) == 4 ? 2 : 1;  // BY = 16 * RPT: 32 (FP32), 16 (FP64)
}

// Staged row pitch: BX = 64 plus the x halo, padded to 16 bytes.
template <typename T, int R>
__host__ __device__ constexpr int stream_pitch()
{
    return (64 + 2 * R + (int)(16 / sizeof(T)) - 1) / (int)(16 / sizeof(T)) * (int)(16 / sizeof(T));
}

template <typename T, int R>
__host__ __device__ constexpr int stream_plane_elems()
{
    return (16 * stream_rows_per_thread<T>() + 2 * R) * stream_pitch<T, R>();
}

// Planes in flight ahead of the computed one: as many as fit (up to 4) in
// ~110 KB of ring, so that two CTAs share an SM.
template <typename T, int R>
__host__ __device__ constexpr int stream_prefetch()
{
    return (110 * 1024 / (stream_plane_elems<T, R>() * (int)sizeof(T)) - (2 * R + 1)) > 4
               ? 4
               : ((110 * 1024 / (stream_plane_elems<T, R>() * (int)sizeof(T)) - (2 * R + 1)) < 1
                      ? 1
                      : (110 * 1024 / (stream_plane_elems<T, R>() * (int)sizeof(T)) - (2 * R + 1)));
}

template <typename T, int R>
__host__ __device__ constexpr size_t stream_smem_bytes(int K)
{
    return (sizeof(T) == 8 ? (size_t)((K * sizeof(T) + 15) / 16 * 16) : 0) +
           (size_t)(2 * R + 1 + stream_prefetch<T, R>()) * stream_plane_elems<T, R>() * sizeof(T);
}

// Columns [lo, hi] of a thread's row segment (of 4 + 2R values) that the
// taps of plane offset oz, row offset oy touch: x0 + R + ox + c for the ox
// with a tap and c = 0..3 (lo > hi: no tap in this row).
template <int SHAPE, int R>
__host__ __device__ constexpr int seg_lo(int oz, int oy)
{
    int lo = 1 << 20;
    for (int ox = -R; ox <= R; ++ox)
        if (tap_index<SHAPE, 3, R>(oz, oy, ox) >= 0 && R + ox < lo) lo = R + ox;
    return lo;
}
template <int SHAPE, int R>
__host__ __device__ constexpr int seg_hi(int oz, int oy)
{
    int hi = -1;
    for (int ox = -R; ox <= R; ++ox)
        if (tap_index<SHAPE, 3, R>(oz, oy, ox) >= 0 && R + ox + 3 > hi) hi = R + ox + 3;
    return hi;
}

// v[i] = rowp[i] for i in [lo, hi] with the widest shared loads their
// alignment allows (rowp is 16-byte aligned): 16-byte, then 8-byte (FP32),
// then single loads.  lo and hi are constants once the callers' loops over
// the tap offsets are unrolled, so every branch folds away.
template <typename T, int NV>
__device__ __forceinline__ void load_seg(const T *__restrict__ rowp, T *v, int lo, int hi)
{
    constexpr int VE = 16 / (int)sizeof(T);
    auto s16 = [&](int j) { return j >= 0 && j % VE == 0 && j >= lo && j + VE - 1 <= hi; };
    auto s8 = [&](int j) {
        return sizeof(T) == 4 && j >= 0 && j % 2 == 0 && j >= lo && j + 1 <= hi && !s16(j - j % VE);
    };
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if (i < lo || i > hi) continue;
        if (s16(i)) {
            if constexpr (sizeof(T) == 4) {
                const float4 q = *reinterpret_cast<const float4 *>(rowp + i);
                v[i] = q.x;
                v[i + 1] = q.y;
                v[i + 2] = q.z;
                v[i + 3] = q.w;
            } else {
                const double2 q = *reinterpret_cast<const double2 *>(rowp + i);
                v[i] = q.x;
                v[i + 1] = q.y;
            }
        } else if (s16(i - i % VE)) {
            // loaded with its 16-byte group
        } else if (s8(i)) {
            const float2 q = *reinterpret_cast<const float2 *>(reinterpret_cast<const float *>(rowp) + i);
            v[i] = (T)q.x;
            v[i + 1] = (T)q.y;
        } else if (s8(i - i % 2)) {
            // loaded with its 8-byte pair
        } else {
            v[i] = rowp[i];
        }
    }
}

template <typename T, int SHAPE, int R>
__global__ void __launch_bounds__(kThreads, 2)
    cu3d_stream(const T *__restrict__ in, T *__restrict__ out,
                const __grid_constant__ Weights<T, Taps<SHAPE, 3, R>::K> wt, int64_t Ez, int64_t Ey, int64_t Ex,
                int tiles_x, int tiles_y, int cz, int nitems)
{
    chain_wait();
    constexpr int KT = Taps<SHAPE, 3, R>::K;
    constexpr bool kSmemW = sizeof(T) == 8;
    constexpr int RPT = stream_rows_per_thread<T>(), BY = 16 * RPT, BX = 64;
    constexpr int PW = stream_pitch<T, R>(), PH = BY + 2 * R, PE = stream_plane_elems<T, R>();
    constexpr int PF = stream_prefetch<T, R>();
    constexpr int NP = 2 * R + 1 + PF;
    constexpr int VE = 16 / (int)sizeof(T);  // elements per 16 bytes
    constexpr int NV = 4 + 2 * R;            // row segment of a thread
    constexpr int NL = (NV + VE - 1) / VE;   // 16-byte loads per row segment
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *wsm = reinterpret_cast<T *>(smem_raw);
    if (kSmemW) {
        for (int k = threadIdx.x; k < KT; k += blockDim.x) wsm[k] = wt.w[k];
    }
    T *ring = reinterpret_cast<T *>(smem_raw + (kSmemW ? (KT * sizeof(T) + 15) / 16 * 16 : 0));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ty = tid >> 4, tx = tid & 15, x0 = 4 * tx;
    const int64_t nz = Ez - 2 * R, ny = Ey - 2 * R, nx = Ex - 2 * R;
    // rows start on 16-byte boundaries in global memory when the stored row
    // length is a 16-byte multiple and `in` is aligned (the staged window of
    // every tile starts at column 64 bx, a 16-byte multiple)
    const bool vec = (Ex * (int64_t)sizeof(T)) % 16 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;

    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        const int bx = item % tiles_x, by = (item / tiles_x) % tiles_y, bz = item / (tiles_x * tiles_y);
        // stored coordinates of the first output of the item
        const int64_t Z0 = R + (int64_t)bz * cz, Y0 = R + (int64_t)by * BY, X0 = R + (int64_t)bx * BX;
        const int64_t rem = nz - (Z0 - R);
        const int nzo = (int)(rem < cz ? rem : cz);  // output planes of this item
        const int64_t zfirst = Z0 - R;                                // first input plane
        const int nin = nzo + 2 * R;                                  // input planes of the item
        // copy input plane gz (rows Y0-R.., columns X0-R.., zero outside the
        // stored grid) into its ring slot
        auto load_plane = [&](int64_t gz) {
            T *dst = ring + (size_t)((gz - zfirst) % NP) * PE;
            const bool zok = gz >= 0 && gz < Ez;
            for (int row = warp; row < PH; row += kThreads / 32) {
                const int64_t gy = Y0 - R + row;
                const bool rok = zok && gy >= 0 && gy < Ey;
                const T *src = in + ((rok ? gz : 0) * Ey + (rok ? gy : 0)) * Ex;
                for (int c = lane * VE; c < PW; c += 32 * VE) {
                    const int64_t gx = X0 - R + c;
                    if (vec && rok && gx + VE <= Ex) {
                        cp_async_elem<16>(dst + row * PW + c, src + gx, true);
                    } else {
#pragma unroll
                        for (int e = 0; e < VE; ++e) {
                            const bool ok = rok && gx + e < Ex;
                            cp_async_elem<sizeof(T)>(dst + row * PW + c + e, ok ? src + gx + e : in, ok);
                        }
                    }
                }
            }
        };
        __syncthreads();  // the previous item's reads of the ring are done
        // planes 0 .. 2R (the first output's) and the PF planes after them
        for (int k = 0; k < 2 * R + 1; ++k) load_plane(zfirst + k);
        cp_async_commit();
#pragma unroll
        for (int f = 0; f < PF; ++f) {
            if (2 * R + 1 + f < nin) load_plane(zfirst + 2 * R + 1 + f);
            cp_async_commit();
        }
        for (int zo = 0; zo < nzo; ++zo) {
            // planes zo .. zo + 2R are needed: all but the PF newest groups
            cp_async_wait_group<PF>();
            __syncthreads();
            T acc[RPT][4];
#pragma unroll
            for (int i = 0; i < RPT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = T(0);
#pragma unroll
            for (int oz = -R; oz <= R; ++oz) {
                const T *pl = ring + (size_t)((zo + R + oz) % NP) * PE;
#pragma unroll
                for (int oy = -R; oy <= R; ++oy) {
                    bool any = false;
#pragma unroll
                    for (int ox = -R; ox <= R; ++ox) any = any || tap_index<SHAPE, 3, R>(oz, oy, ox) >= 0;
                    if (!any) continue;
#pragma unroll
                    for (int i = 0; i < RPT; ++i) {
                        const T *rowp = pl + (ty + 16 * i + R + oy) * PW + x0;
                        T v[NL * VE];
                        load_seg<T, NL * VE>(rowp, v, seg_lo<SHAPE, R>(oz, oy), seg_hi<SHAPE, R>(oz, oy));
#pragma unroll
                        for (int ox = -R; ox <= R; ++ox) {
                            const int k = tap_index<SHAPE, 3, R>(oz, oy, ox);
                            if (k >= 0) {
                                const T wk = kSmemW ? wsm[k] : wt.w[k];
#pragma unroll
                                for (int c = 0; c < 4; ++c) acc[i][c] = fma(wk, v[c + R + ox], acc[i][c]);
                            }
                        }
                    }
                }
            }
            const int64_t gz = Z0 + zo;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int64_t gy = Y0 + ty + 16 * i;
                if (gy - R >= ny) continue;
                T *orow = out + (gz * Ey + gy) * Ex;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int64_t gx = X0 + x0 + c;
                    if (gx - R < nx) orow[gx] = acc[i][c];
                }
            }
            __syncthreads();  // plane zo is no longer read: its slot takes plane zo + 2R + 1 + PF
            if (zo + 2 * R + 1 + PF < nin) load_plane(zfirst + zo + 2 * R + 1 + PF);
            cp_async_commit();
        }
    }
    cp_async_wait_group<0>();
    chain_next();
}


// ---------------------------------------------------------------------------
// 3-D, t = 1, FP32: z-marching with rotating partial sums.
// ---------------------------------------------------------------------------
// A work item is a tile of nq quads (16 bytes) x ns TY rows and a run of cz
// output planes; thread (strip, quad) = (tid / nq, tid mod nq) owns TY rows of
// four columns.  nq and ns are chosen per grid so that whole tiles cover it with
// few idle threads (rot_tile).  The CTA stages one input plane at a time (a ring
// of kRotNPL planes keeps the next ones in flight with cp.async) and adds it,
// once, into every output plane it touches: input plane ip contributes its 2-D
// slice w(oz, ., .) to output plane ip - R - oz for oz in [-R, R], so each
// thread keeps partial sums of its outputs for 2R+1 output planes in registers
// (slots rotate with the plane index; the plane loop is unrolled by 2R+1, so
// every slot and weight index is a compile-time constant).  Output plane oq
// is complete after input plane oq + 2R and is stored from its slot.  Input
// planes of the first and last 2R of a run also add into slots of outputs
// outside the run; those slots are cleared, never stored.
// Staged planes hold quads -1 .. nq of the tile's rows -R .. ns TY + R - 1 (tiles
// start at a stored column that is a multiple of 4): a thread's taps need the
// quads qx, qx+1, qx+2 of a staged row; rows that only the centre column touches
// (star stencils) need quad qx+1 alone.  The quads a thread copies sit at the
// same place of every plane, so their offsets and masks are found once per
// item: a copy is one address add and one cp.async (four words where stored
// rows are not 16-byte multiples).  One barrier per plane.  Word rows are stored
// through shared memory as coalesced words.
// Measured, one sweep (64 x 32 tiles, per-copy index arithmetic, two barriers per
// plane before): Star-3D2R 512^3 305 -> 230 us (HBM floor 159), Box-3D1R
// 301 x 417 x 533 (words) 240 -> 179 us (floor 80); bound by issue: 27 FMAs of
// ~40 instructions per output for the box.
constexpr int kRotNPL = 4;   // ring planes: the one computed and three in flight
constexpr int kRotCopies = 6;  // quads of a staged plane a thread copies, at most

template <int SHAPE, int R>
__host__ __device__ constexpr int rot_rows_per_thread()
{
    return R == 1 ? 4 : 2;
}

// Does staged row j (0 .. RPT + 2R - 1) of a thread need more than the
// centre quad?  (Yes if some output row i takes it as its own row, oy = 0,
// or the stencil is a box.)
template <int SHAPE, int R, int RPT>
__host__ __device__ constexpr bool rot_full_row(int j)
{
    return SHAPE == 0 || (j >= R && j < R + RPT);
}

struct RotTile {
    int nq = 0, ns = 0;            // quads per row, strips of TY rows
    int tiles_x = 0, tiles_y = 0;
    size_t smem = 0;
};

// The tile of a grid with ny x nx interior points per plane (columns xb .. from
// the first quad on): the fewest thread-planes, with the staged halo's extra
// reads weighted by half.
template <int R, int TY>
inline RotTile rot_tile(int64_t ny, int64_t span, bool vec)
{
    RotTile best;
    double best_cost = 0;
    for (int nq = 8; nq <= 64; nq++) {
        RotTile t;
        t.nq = nq;
        t.ns = kThreads / nq;
        const int ph = t.ns * TY + 2 * R, quads = ph * (nq + 2);
        if (quads > kRotCopies * kThreads) continue;
        const int64_t tx = (span + 4 * nq - 1) / (4 * nq), ty = (ny + t.ns * TY - 1) / (t.ns * TY);
        const double halo = (double)quads / (t.ns * TY * nq);
        const double cost = (double)tx * ty * (1.0 + 0.5 * (halo - 1.0));
        if (best.nq == 0 || cost < best_cost) {
            t.tiles_x = (int)tx;
            t.tiles_y = (int)ty;
            t.smem = (size_t)kRotNPL * quads * 16 + (vec ? 0 : kThreads * 16);
            best = t;
            best_cost = cost;
        }
    }
    return best;
}

template <int SHAPE, int R, bool VEC>
__global__ void __launch_bounds__(kThreads, 2)
    cu3d_rot(const float *__restrict__ in, float *__restrict__ out,
             const __grid_constant__ Weights<float, Taps<SHAPE, 3, R>::K> wt, int64_t Ez, int64_t Ey, int64_t Ex,
             int nq, int ns, int tiles_x, int tiles_y, int nitems, int cz, int xb)
{
    chain_wait();
    constexpr int TY = rot_rows_per_thread<SHAPE, R>(), NS = 2 * R + 1, NPL = kRotNPL;
    static_assert(R <= 3, "one quad of halo columns per side");
    extern __shared__ __align__(16) float ring[];
    const int tid = threadIdx.x, strip = tid / nq, qx = tid - strip * nq;
    const bool active = strip < ns;
    const int PH = ns * TY + 2 * R, PQ = nq + 2, PW = 4 * PQ, quads = PH * PQ, PE = 4 * quads;
    float *const turn = ring + (size_t)NPL * PE + (tid >> 5) * 128;  // word rows: a warp's 32 quads
    const int64_t nz = Ez - 2 * R, ny = Ey - 2 * R, nx = Ex - 2 * R, plane = Ey * Ex;
    const int ex32 = (int)Ex;  // a stored plane holds < 2^31 values (rot3d_plane_fits)

    for (int item = blockIdx.x; item < nitems; item += gridDim.x) {
        const int bx = item % tiles_x, by = (item / tiles_x) % tiles_y, bz = item / (tiles_x * tiles_y);
        // stored coordinates of the item's first output (column X0 may lie in the halo)
        const int64_t Z0 = R + (int64_t)bz * cz, Y0 = R + (int64_t)by * (ns * TY), X0 = xb + (int64_t)bx * (4 * nq);
        const int64_t rem = nz - (Z0 - R);
        const int nzo = (int)(rem < cz ? rem : cz);
        const int nin = nzo + 2 * R;
        // this thread's copies: offset within a plane, and which values exist
        int goff[kRotCopies];
        unsigned have = 0;  // VEC: bit m; words: bits 4m .. 4m + 3
#pragma unroll
        for (int m = 0; m < kRotCopies; ++m) {
            const int e = tid + m * kThreads, row = e / PQ, ch = e - row * PQ;
            const int64_t gy = Y0 - R + row, gx = X0 - 4 + 4 * ch;
            const bool rok = e < quads && gy >= 0 && gy < Ey;
            goff[m] = rok ? (int)(gy * Ex + gx) : 0;
            if constexpr (VEC) {
                have |= (rok && gx >= 0 && gx < Ex) ? 1u << m : 0u;
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) have |= (rok && gx + c >= 0 && gx + c < Ex) ? 1u << (4 * m + c) : 0u;
            }
        }
        const float *src = in + (Z0 - R) * plane;  // the next plane to copy
        auto load_plane = [&](int ip) {
            float *dst = ring + (size_t)(ip & (NPL - 1)) * PE + 4 * tid;
#pragma unroll
            for (int m = 0; m < kRotCopies; ++m) {
                if (tid + m * kThreads >= quads) break;
                float *d = dst + 4 * m * kThreads;
                if constexpr (VEC) {
                    const bool ok = (have >> m) & 1u;
                    cp_async_elem<16>(d, ok ? src + goff[m] : in, ok);
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const bool ok = (have >> (4 * m + c)) & 1u;
                        cp_async_elem<4>(d + c, ok ? src + goff[m] + c : in, ok);
                    }
                }
            }
            src += plane;
        };
        __syncthreads();  // the previous item's reads of the ring are done
#pragma unroll
        for (int k = 0; k < NPL - 1; ++k) {
            if (k < nin) load_plane(k);
            cp_async_commit();
        }
        float acc[NS][TY][4];
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int i = 0; i < TY; ++i) acc[s][i][0] = acc[s][i][1] = acc[s][i][2] = acc[s][i][3] = 0.0f;
        // stores.  VEC: the thread's own quads; words: value j of the warp's 128 is
        // component lane % 4 of the quad of lane 8 j + lane / 4
        const int64_t gy0 = Y0 + strip * TY, gx0 = X0 + 4 * qx;
        const int nrow_ok = active ? (int)min((int64_t)TY, ny + R - gy0) : 0;  // rows of the thread inside the interior
        unsigned cmask = 0;  // interior columns of the quad
#pragma unroll
        for (int c = 0; c < 4; ++c) cmask |= (gx0 + c >= R && gx0 + c - R < nx) ? (1u << c) : 0u;
        float *dst = out + Z0 * plane + gy0 * Ex + gx0;  // the next output plane
        int woff[VEC ? 1 : 4];   // words: offset of value j from `out`'s plane, rows it is stored in
        int wrow = 0;  // four bits per j
        if constexpr (!VEC) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int t2 = (tid & ~31) + 8 * j + ((tid & 31) >> 2), s2 = t2 / nq, q2 = t2 - s2 * nq;
                const int64_t y2 = Y0 + s2 * TY, x2 = X0 + 4 * q2 + (tid & 3);
                woff[j] = (int)(y2 * Ex + x2);
                wrow |= (s2 < ns && x2 >= R && x2 - R < nx ? (int)max((int64_t)0, min((int64_t)TY, ny + R - y2)) : 0)
                        << (4 * j);
            }
            dst = out + Z0 * plane;
        }
        const int col = (strip * TY) * PW + 4 * qx;
        for (int base = 0; base < nin; base += NS) {
            // the NS planes of this round; u is a compile-time constant, so every
            // accumulator slot index below is one too (no run-time selects)
            static_for<NS>([&](auto UC) -> bool {
                constexpr int u = decltype(UC)::value;
                const int ip = base + u;
                if (ip >= nin) return false;
                cp_async_wait_group<NPL - 2>();  // this thread's copies of plane ip have landed
                __syncthreads();                 // everyone's have, and plane ip - 1 is read
                if (ip + NPL - 1 < nin) load_plane(ip + NPL - 1);
                cp_async_commit();
                if (active) {
                    const float *pl = ring + (size_t)(ip & (NPL - 1)) * PE + col;
#pragma unroll
                    for (int j = 0; j < TY + 2 * R; ++j) {
                        const float *rowp = pl + j * PW;
                        float v[12];
                        const float4 c1 = *reinterpret_cast<const float4 *>(rowp + 4);
                        v[4] = c1.x;
                        v[5] = c1.y;
                        v[6] = c1.z;
                        v[7] = c1.w;
                        if (rot_full_row<SHAPE, R, TY>(j)) {
                            const float4 c0 = *reinterpret_cast<const float4 *>(rowp);
                            const float4 c2 = *reinterpret_cast<const float4 *>(rowp + 8);
                            v[0] = c0.x;
                            v[1] = c0.y;
                            v[2] = c0.z;
                            v[3] = c0.w;
                            v[8] = c2.x;
                            v[9] = c2.y;
                            v[10] = c2.z;
                            v[11] = c2.w;
                        }
#pragma unroll
                        for (int i = 0; i < TY; ++i) {
                            const int oy = j - i - R;
                            if (oy < -R || oy > R) continue;
#pragma unroll
                            for (int oz = -R; oz <= R; ++oz) {
                                const int slot = ((u - R - oz) % NS + 2 * NS) % NS;
#pragma unroll
                                for (int ox = -R; ox <= R; ++ox) {
                                    const int k = tap_index<SHAPE, 3, R>(oz, oy, ox);
                                    if (k >= 0) {
#pragma unroll
                                        for (int c = 0; c < 4; ++c)
                                            acc[slot][i][c] = fmaf(wt.w[k], v[4 + c + ox], acc[slot][i][c]);
                                    }
                                }
                            }
                        }
                    }
                }
                // output plane ip - 2R is complete (slot (u + 1) mod NS)
                constexpr int sd = (u + 1) % NS;
                if (ip >= 2 * R) {
#pragma unroll
                    for (int i = 0; i < TY; ++i) {
                        if constexpr (VEC) {
                            if (i < nrow_ok) {
                                float *o = dst + i * ex32;
                                if (cmask == 0xfu) {
                                    *reinterpret_cast<float4 *>(o) =
                                        make_float4(acc[sd][i][0], acc[sd][i][1], acc[sd][i][2], acc[sd][i][3]);
                                } else {
#pragma unroll
                                    for (int c = 0; c < 4; ++c)
                                        if ((cmask >> c) & 1u) o[c] = acc[sd][i][c];
                                }
                            }
                        } else {
                            __syncwarp();
                            *reinterpret_cast<float4 *>(turn + 4 * (tid & 31)) =
                                make_float4(acc[sd][i][0], acc[sd][i][1], acc[sd][i][2], acc[sd][i][3]);
                            __syncwarp();
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const float w = turn[32 * j + (tid & 31)];
                                if (i < ((wrow >> (4 * j)) & 15)) dst[woff[j] + i * ex32] = w;
                            }
                        }
                    }
                    dst += plane;
                }
#pragma unroll
                for (int i = 0; i < TY; ++i) acc[sd][i][0] = acc[sd][i][1] = acc[sd][i][2] = acc[sd][i][3] = 0.0f;
                return true;
            });
        }
        cp_async_wait_group<0>();
    }
    chain_next();
}

}  // namespace cu
}  // namespace gbs
