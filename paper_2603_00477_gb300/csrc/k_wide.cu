// k_wide.cu -- 2-D FP32 grids on the tcgen05 tensor cores (kernels tc2d_wide:
// precisions f16, f16x3, bf16x3; tc2d_ws: tf32, tf32x3): the Toeplitz
// (kernel-fusion) formulation of the paper's Sec. 2.2 with the weights as the
// A operand over two-dimensional blocks of outputs.
//
// One MMA row block is a block of 16 x 8 outputs (M = 128), one MMA column a
// block position, so the A operand holds the composite weights w^(t) of every
// (output of the block, input of its 16 + 2R by 8 + 2R neighbourhood) pair.  A
// line of 128 outputs (M = 128 columns of one row) would need a
// 128 + 2R window for each of the 2R + 1 lines: (2R+1)(128+2R) products per
// output, of which (2R+1)^2 are useful.  A 16 x 8 block needs
// (16+2R)(8+2R): for R = 8, 768 instead of 2448 (9 x 17 = 153 MMAs of K = 16
// per 128 x N outputs against 48), for R = 7 in TF32 (K = 8) 90 against
// 15 x 6 = 90 MMAs of a quarter of the width.  The MMAs stop being the bound
// (48 x 128 cycles per 32768 outputs at R = 8 against ~12,200 cycles of HBM
// traffic for the same outputs).
//
// A operand.  Output (my, mx) of a block sits at row m = 8 (15 - my) + 7 - mx;
// K runs over 16-byte chunks c of an input row ky of the neighbourhood.  The
// core matrix (8 rows x 16 bytes) of row group g and K chunk (ky, c) holds
// w[ky + g - 15][CE c + j + i - 7] (row i, column j; CE values per chunk): it
// depends on (ky + g, c) only.  So one strip of (31 + 2R) x NC core matrices
// (NC = chunks of a neighbourhood row), zero outside lines 15 .. 15 + 2R,
// serves every MMA: start (ky NC + c) 128 bytes, SBO = NC x 128, LBO = 128 to
// the next chunk, or NC x 128 to the same chunk of the next row (the odd
// chunk of NC = 3, 5, 7 is paired over two rows).
//
// B operand.  The tile (16 GN + 2R rows x 64 + 2R columns, padded to whole
// chunks) is stored row by row.  Column n = 8 G + q of the MMA is the block at
// rows 16 G, columns 8 q, so the core matrix of (group G, chunk (ky, c)) is 8
// consecutive 16-byte units of row 16 G + ky: 16-bit operands, chunks
// q + c (8 values each); TF32, chunks 2 q + c (4 values each), for which even
// and odd chunks are kept in two planes.  SBO = 16 rows; LBO = one unit (16
// bit), the plane distance (TF32) or one row (the odd chunk).  No im2col copy.
//
// The 16-bit forms scale each tile by a power of two (FP16 has 5 exponent
// bits) and the weights likewise; the epilogue undoes both exactly.  A tile is
// read once: it is converted with the scale of the CTA's previous tile while
// its largest |x| is found, and converted again only if that scale would
// overflow or leave the largest value below 2^7 (the FP16 normal range starts
// at 2^-14, so values down to 2^-21 of the tile's largest keep 11 bits, and the
// lo parts of f16x3 stay exact to 2^-31 of it).  TF32 needs no scale.
//
// Persistent, warp specialised, one CTA per SM (672 threads): warps 0-11 load
// and convert the next tile into the other operand buffer, one thread of warp
// 20 issues the MMAs into the other TMEM accumulator, warps 12-19 read the
// previous accumulator back (tcgen05.ld), turn each 4 x 64 group of outputs
// through shared memory and store whole rows.  Every wait is bounded.  Only
// interior points farther than (t-1) r from the boundary are written; the
// CUDA-core band kernel computes the others.
//
// Measured against the line form this replaced (Box-2D2R, one fused sweep):
// f16 t = 4 on 16384^2 776 -> 572 us (HBM floor 317), f16x3 t = 4 on
// 7001 x 6007 (unaligned rows) 433 -> 214 us.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "launch.h"
#include "tc_layout.h"
#include "tc_ptx.cuh"

namespace gbs {

// Set when a bounded wait of this kernel runs out (each translation unit
// keeps its own error word; read_device_error reads them all).
__device__ int g_wide_error;

namespace wide {

using namespace tc;

enum Form { kF16 = 0, kF16x3, kBF16x3, kTF32, kTF32x3 };
__host__ __device__ constexpr bool is_split(int f) { return f == kF16x3 || f == kBF16x3 || f == kTF32x3; }
__host__ __device__ constexpr bool is_tf32(int f) { return f == kTF32 || f == kTF32x3; }

constexpr int kMaxR = kWideMaxR;
constexpr int kMaxLines = 2 * kMaxR + 1;
constexpr int kBY = 16;                       // rows of an output block (16 x 8: MMA M = 128)
constexpr int kTX = 64;                       // output columns per tile: 8 blocks
constexpr int kLoadWarps = 12;                // warps 0-11
constexpr int kLoaders = 32 * kLoadWarps;
constexpr int kEpiWarp = kLoadWarps;          // warps 12-19: TMEM lane quarter w % 4, half (w - 12) / 4
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kLoadWarps + kEpiWarps;  // warp 20
constexpr int kThreads = 32 * (kMmaWarp + 1);
constexpr int kBatch = 8;                     // independent 16-byte loads in flight per loader thread
constexpr int kBatchU = 4;                    // the same where a quad takes two (unaligned rows)
constexpr int kHeader = 1024;
constexpr int kStageRow = kTX + 8;             // epilogue staging: 4 rows of 64 outputs per warp, padded
constexpr int kStageBytes = kEpiWarps * 4 * kStageRow * 4;
constexpr unsigned long long kWaitCycles = 4ull << 30;       // ~2 s at 2 GHz
constexpr unsigned long long kDebugWaitCycles = 1ull << 22;  // ~2 ms: the test hook's limit

struct WideParams {
    double w[kMaxLines * kMaxLines];  // composite w^(t), (2R+1) x (2R+1), row-major
    int R, rh, band, ew;
    int gn;     // block rows per tile: 16 gn output rows, MMA N = 8 gn
    int nbuf;   // operand buffers (2, or 1 where two do not fit)
    int nc;     // 16-byte chunks of a neighbourhood row (8 + 2R columns)
    int pc;     // 8-column units of a staged row
    uint32_t plane;     // TF32: bytes between the even- and the odd-chunk plane
    uint32_t in_bytes;  // one operand buffer (hi or lo)
    int debug_unmet;  // test hook: wait once more on an mbarrier phase that never completes
    int vec16;        // stored rows are 16-byte multiples and `in` is aligned: tiles start aligned
    int xshift;       // tiles start xshift columns left of column 0
    int vst;          // widest output store (elements: 4, 2 or 1) whose alignment every tile row has
    int64_t Ey, Ex;
};

__device__ __forceinline__ float pow2f(int e)  // 2^e for -126 <= e <= 127
{
    return __int_as_float((e + 127) << 23);
}

// 16-bit operand types: FP16 (11 significant bits) or BF16 (8 significant
// bits, the range of FP32); packed conversions of two FP32 values and back.
template <bool BF>
struct Op;
template <>
struct Op<false> {
    using T2 = __half2;
    __device__ static T2 pack(float a, float b) { return __floats2half2_rn(a, b); }
    __device__ static float2 unpack(T2 v) { return __half22float2(v); }
    __device__ static uint16_t bits(double w)
    {
        const __half h = __double2half(w);
        return *reinterpret_cast<const uint16_t *>(&h);
    }
    __device__ static double value(uint16_t b)
    {
        return (double)__half2float(*reinterpret_cast<const __half *>(&b));
    }
};
template <>
struct Op<true> {
    using T2 = __nv_bfloat162;
    __device__ static T2 pack(float a, float b) { return __floats2bfloat162_rn(a, b); }
    __device__ static float2 unpack(T2 v) { return __bfloat1622float2(v); }
    __device__ static uint16_t bits(double w)
    {
        const __nv_bfloat16 h = __double2bfloat16(w);
        return *reinterpret_cast<const uint16_t *>(&h);
    }
    __device__ static double value(uint16_t b)
    {
        return (double)__bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(&b));
    }
};

// Largest |x| seen so far, as an unsigned integer (IEEE order).
__device__ __forceinline__ unsigned max_abs(unsigned m, const float4 &v)
{
    return max(m, max(max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu),
                      max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu)));
}

// Convert the four columns of item i (row i / (2 pc), columns 4 (i mod 2 pc) ..)
// and store them to the operand buffer: 8 bytes (16-bit forms) or one 16-byte
// chunk (TF32) at an offset that is linear in i.
template <int FORM>
__device__ __forceinline__ void put(unsigned char *hi, unsigned char *lo, int i, float4 v, float xs, uint32_t plane)
{
    if constexpr (is_tf32(FORM)) {
        const uint32_t off = (uint32_t)(i >> 1) * 16 + (i & 1) * plane;
        const float4 h = make_float4(to_tf32(v.x), to_tf32(v.y), to_tf32(v.z), to_tf32(v.w));
        *reinterpret_cast<float4 *>(hi + off) = h;
        if (is_split(FORM))
            *reinterpret_cast<float4 *>(lo + off) =
                make_float4(to_tf32(v.x - h.x), to_tf32(v.y - h.y), to_tf32(v.z - h.z), to_tf32(v.w - h.w));
    } else {
        using O = Op<FORM == kBF16x3>;
        const float x0 = v.x * xs, x1 = v.y * xs, x2 = v.z * xs, x3 = v.w * xs;
        const typename O::T2 h01 = O::pack(x0, x1), h23 = O::pack(x2, x3);
        uint2 hv;
        hv.x = *reinterpret_cast<const uint32_t *>(&h01);
        hv.y = *reinterpret_cast<const uint32_t *>(&h23);
        *reinterpret_cast<uint2 *>(hi + (uint32_t)i * 8) = hv;
        if (is_split(FORM)) {
            const float2 f01 = O::unpack(h01), f23 = O::unpack(h23);
            const typename O::T2 l01 = O::pack(x0 - f01.x, x1 - f01.y), l23 = O::pack(x2 - f23.x, x3 - f23.y);
            uint2 lv;
            lv.x = *reinterpret_cast<const uint32_t *>(&l01);
            lv.y = *reinterpret_cast<const uint32_t *>(&l23);
            *reinterpret_cast<uint2 *>(lo + (uint32_t)i * 8) = lv;
        }
    }
}

template <int FORM>
__device__ __forceinline__ void block_sweep(const float *__restrict__ in, float *__restrict__ out,
                                            const WideParams &p, int ntiles, int ntx)
{
    constexpr bool SPLIT = is_split(FORM), TF = is_tf32(FORM), SCALED = !TF;
    constexpr bool CORR = FORM == kTF32x3;  // hi*lo + lo*hi in an accumulator of their own
    constexpr int CE = TF ? 4 : 8;          // values per 16-byte chunk
    extern __shared__ __align__(1024) unsigned char smem[];
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem);
    int *abort_flag = reinterpret_cast<int *>(smem + 4);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + 16);     // [2] operand buffer staged
    uint64_t *done = reinterpret_cast<uint64_t *>(smem + 32);     // [2] MMAs of a tile complete
    uint64_t *accfree = reinterpret_cast<uint64_t *>(smem + 48);  // [2] accumulator drained
    uint64_t *maxb = reinterpret_cast<uint64_t *>(smem + 64);     // [2] exponent exchange
    uint64_t *eub = reinterpret_cast<uint64_t *>(smem + 80);      // [4] a tile's scale published
    int *wmax = reinterpret_cast<int *>(smem + 128);              // [2][kLoadWarps]
    int *eus = reinterpret_cast<int *>(smem + 256);               // [4] input scale exponent per tile
    const int R = p.R, lines = 2 * R + 1, nc = p.nc, pc = p.pc, gn = p.gn, nbuf = p.nbuf;
    const uint32_t strip_bytes = (uint32_t)(31 + 2 * R) * nc * 128;
    const uint32_t in_bytes = p.in_bytes;
    float *stage = reinterpret_cast<float *>(smem + kHeader);
    unsigned char *Whi = smem + kHeader + kStageBytes;
    unsigned char *Wlo = Whi + strip_bytes;
    unsigned char *ibase = Whi + strip_bytes * (SPLIT ? 2 : 1);
    // operand buffer b (b = 0 when nbuf = 1): hi at ibase + b in_bytes, lo
    // (the 3-product forms) nbuf in_bytes further
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t Ey = p.Ey, Ex = p.Ex, rh = p.rh;
    const int64_t ny = Ey - 2 * rh;
    const int N = 8 * gn;                                  // MMA columns
    const uint32_t aset = (uint32_t)N * (CORR ? 2 : 1);    // TMEM columns of one accumulator set

    if (warp == kMmaWarp) tmem_alloc(tmem_slot, 512);
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(&full[b], kLoaders);
            mbar_init(&done[b], 1);
            mbar_init(&accfree[b], 32 * kEpiWarps);
            mbar_init(&maxb[b], kLoaders);
        }
        for (int s = 0; s < 4; ++s) mbar_init(&eub[s], 1);
        fence_mbar_init();
    }
    // weight strip: core matrix (L, c), L = ky + g, holds line L - 15
    {
        const double wsc = SCALED ? ldexp(1.0, 15 - p.ew) : 1.0;  // |w| 2^(15 - ew) < 2^15: exact scaling
        const int nelem = (31 + 2 * R) * nc * 8 * CE;
        for (int e = tid; e < nelem; e += kThreads) {
            const int j = e % CE, i = (e / CE) & 7, core = e / (8 * CE);
            const int d = core / nc - 15, idx = CE * (core % nc) + j + i - 7;
            const double wv = (d >= 0 && d < lines && idx >= 0 && idx < lines) ? p.w[d * lines + idx] * wsc : 0.0;
            if constexpr (TF) {
                const float h = to_tf32((float)wv);
                reinterpret_cast<float *>(Whi)[e] = h;
                if (SPLIT) reinterpret_cast<float *>(Wlo)[e] = to_tf32((float)(wv - (double)h));
            } else {
                using O = Op<FORM == kBF16x3>;
                const uint16_t h = O::bits(wv);
                reinterpret_cast<uint16_t *>(Whi)[e] = h;
                if (SPLIT) reinterpret_cast<uint16_t *>(Wlo)[e] = O::bits(wv - O::value(h));
            }
        }
    }
    fence_proxy_async_smem();
    fence_before_thread_sync();
    __syncthreads();
    fence_after_thread_sync();
    const uint32_t tmem = *tmem_slot;

    auto bounded_wait = [&](uint64_t *bar, uint32_t parity, unsigned long long limit) -> bool {
        const unsigned long long t0 = clock64();
        while (!mbar_try_wait(bar, parity)) {
            if (*(volatile int *)abort_flag) return false;
            if (clock64() - t0 > limit) {
                atomicExch(abort_flag, 1);
                return false;
            }
        }
        return true;
    };
    auto origin = [&](int id, int64_t *Y0, int64_t *X0) {
        *Y0 = rh + (int64_t)(id / ntx) * (kBY * gn);
        *X0 = (int64_t)(id % ntx) * kTX - p.xshift;
    };

    if (warp == kMmaWarp) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            const uint32_t idesc = instr_desc(TF ? kFmtTF32 : (FORM == kBF16x3 ? kFmtBF16 : kFmtF16), 128, N);
            const uint32_t wbase = smem_u32(Whi), rowb = (uint32_t)pc * 16;
            const uint64_t a_c = smem_desc(wbase, 128, (uint32_t)nc * 128);       // chunk pairs of one row
            const uint64_t a_r = smem_desc(wbase, (uint32_t)nc * 128, (uint32_t)nc * 128);  // one chunk of two rows
            const uint64_t dlo_a = (uint64_t)(strip_bytes >> 4), dlo_b = (uint64_t)((nbuf * in_bytes) >> 4);
            int k = 0;
            for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
                const int b = k & 1;
                if (!bounded_wait(&full[b], (k >> 1) & 1, kWaitCycles)) break;
                if (k >= 2 && !bounded_wait(&accfree[b], ((k - 2) >> 1) & 1, kWaitCycles)) break;
                fence_after_thread_sync();
                const uint32_t ib = smem_u32(ibase + (nbuf == 2 ? b : 0) * in_bytes);
                const uint64_t b_c = smem_desc(ib, TF ? p.plane : 16u, 16 * rowb);
                const uint64_t b_r = smem_desc(ib, rowb, 16 * rowb);
                const uint32_t d = tmem + (uint32_t)b * aset, dc = d + (uint32_t)N;
                uint32_t acc = 0;
                auto issue = [&](uint64_t da, uint64_t db) {
                    if constexpr (TF) {
                        mma_tf32(d, da, db, idesc, acc);
                        if (SPLIT) {
                            mma_tf32(dc, da, db + dlo_b, idesc, acc);
                            mma_tf32(dc, da + dlo_a, db, idesc, 1);
                        }
                    } else {
                        mma_f16(d, da, db, idesc, acc);
                        if (SPLIT) {
                            mma_f16(d, da, db + dlo_b, idesc, 1);
                            mma_f16(d, da + dlo_a, db, idesc, 1);
                        }
                    }
                    acc = 1;
                };
                for (int ky = 0; ky < kBY + 2 * R; ky += 2) {
                    for (int y = ky; y < ky + 2; ++y)
                        for (int c = 0; c + 1 < nc; c += 2)
                            issue(a_c + (uint64_t)(y * nc + c) * 8, b_c + (uint64_t)(y * pc + (TF ? c / 2 : c)));
                    if (nc & 1) {
                        const int c = nc - 1;
                        issue(a_r + (uint64_t)(ky * nc + c) * 8, b_r + (uint64_t)(ky * pc + (TF ? c / 2 : c)));
                    }
                }
                mma_commit(&done[b]);
            }
            // the last tiles' MMAs complete before the TMEM is released
            for (int j = k - 2; j < k; ++j)
                if (j >= 0) {
                    const unsigned long long t0 = clock64();
                    while (!mbar_try_wait(&done[j & 1], (j >> 1) & 1) && clock64() - t0 < kWaitCycles) {
                    }
                }
        }
        __syncwarp();
    } else if (warp < kEpiWarp) {
        // ---------------- loaders / converters ----------------
        const int F4 = 2 * pc;  // float4 items per staged row
        const int rows = kBY * gn + 2 * R, items = rows * F4;
        const bool vec16 = p.vec16 != 0;
        // thread tid takes the items i = tid + m kLoaders; (row, quad) advance by a constant step
        const int row0 = tid / F4, col0 = tid - row0 * F4;
        const int step_r = kLoaders / F4, step_c = kLoaders - step_r * F4;
        // ask L2 for tile `id`'s input rows (one prefetch per 128 bytes, every
        // address inside the stored array), so that its loads wait on L2 rather
        // than DRAM latency
        auto prefetch_l2 = [&](int id) {
            int64_t Y0, X0;
            origin(id, &Y0, &X0);
            const int64_t gx_lo = max((int64_t)0, X0 - R), gx_hi = min(Ex, X0 - R + 8 * pc);
            if (gx_lo >= gx_hi) return;
            const int segs = (int)((gx_hi - gx_lo + 31) / 32);
            for (int e = tid; e < rows * segs; e += kLoaders) {
                const int row = e / segs, l = e - (e / segs) * segs;
                const int64_t gy = Y0 - R + row;
                if (gy < 0 || gy >= Ey) continue;
                const int64_t gx = min(gx_lo + 32 * (int64_t)l, gx_hi - 1);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(in + gy * Ex + gx));
            }
        };
        int es = 12;  // the scale the next tile is first tried with: the previous tile's
        int k = 0;
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
            const int b = k & 1;
            int64_t Y0, X0;
            origin(id, &Y0, &X0);
            if (id + (int)gridDim.x < ntiles) prefetch_l2(id + gridDim.x);
            // the operand buffer is free once the MMAs of tile k - nbuf completed
            if (nbuf == 2 && k >= 2 && !bounded_wait(&done[b], ((k - 2) >> 1) & 1, kWaitCycles)) break;
            if (nbuf == 1 && k >= 1 && !bounded_wait(&done[b ^ 1], ((k - 1) >> 1) & 1, kWaitCycles)) break;
            unsigned char *hi = ibase + (nbuf == 2 ? b : 0) * in_bytes, *lo = hi + nbuf * in_bytes;
            // Interior tiles (the staged region inside the stored array): no
            // per-load bounds tests.  Rows that are not 16-byte multiples are
            // read as the two aligned 16-byte words around each quad (the
            // region then keeps a stored row free above and below, so both
            // words lie inside the array).
            const bool inx = X0 - R >= 0 && X0 - R + 8 * pc <= Ex;
            const bool fast = vec16 && inx && Y0 - R >= 0 && Y0 - R + rows <= Ey;
            const bool fast_u = !vec16 && inx && Y0 - R >= 1 && Y0 - R + rows + 1 <= Ey;
            const int64_t wrap = Ex - 4 * F4, step = step_r * Ex + 4 * step_c;
            for (int attempt = 0;; ++attempt) {
                const float xs = SCALED ? pow2f(es) : 1.0f;
                unsigned mxu = 0;
                auto use = [&](int i, const float4 &v) {
                    if (SCALED) mxu = max_abs(mxu, v);
                    put<FORM>(hi, lo, i, v, xs, p.plane);
                };
                const float *q = in + (Y0 - R + row0) * Ex + (X0 - R + 4 * col0);
                int c4 = col0;
                auto next = [&] {
                    q += step;
                    c4 += step_c;
                    if (c4 >= F4) {
                        c4 -= F4;
                        q += wrap;
                    }
                };
                if (fast) {
                    for (int i0 = tid; i0 < items; i0 += kBatch * kLoaders) {
                        float4 v[kBatch];
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (i0 + u * kLoaders < items) v[u] = __ldcg(reinterpret_cast<const float4 *>(q));
                            next();
                        }
#pragma unroll
                        for (int u = 0; u < kBatch; ++u)
                            if (i0 + u * kLoaders < items) use(i0 + u * kLoaders, v[u]);
                    }
                } else if (fast_u) {
                    for (int i0 = tid; i0 < items; i0 += kBatchU * kLoaders) {
                        float4 a[kBatchU], e[kBatchU];
                        int sh = 0;
#pragma unroll
                        for (int u = 0; u < kBatchU; ++u) {
                            a[u] = e[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                            const int s = (int)(reinterpret_cast<uintptr_t>(q) >> 2) & 3;
                            sh |= s << (2 * u);
                            if (i0 + u * kLoaders < items) {
                                const float4 *a4 = reinterpret_cast<const float4 *>(q - s);
                                a[u] = __ldg(a4);
                                if (s) e[u] = __ldg(a4 + 1);
                            }
                            next();
                        }
#pragma unroll
                        for (int u = 0; u < kBatchU; ++u) {
                            if (i0 + u * kLoaders >= items) continue;
                            // quad = values s .. s + 3 of (a, e): shift by two, then by one
                            const int s = sh >> (2 * u);
                            const float4 a2 = (s & 2) ? make_float4(a[u].z, a[u].w, e[u].x, e[u].y) : a[u];
                            const float n4 = (s & 2) ? e[u].z : e[u].x;
                            use(i0 + u * kLoaders, (s & 1) ? make_float4(a2.y, a2.z, a2.w, n4) : a2);
                        }
                    }
                } else {
                    // edge tiles: every value tested; cells outside the stored array are zero
                    int row = row0;
                    for (int i = tid; i < items; i += kLoaders) {
                        const int64_t gy = Y0 - R + row, gx = X0 - R + 4 * c4;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (gy >= 0 && gy < Ey) {
                            if (vec16) {
                                // X0 - R is a multiple of 4: the quad lies wholly inside or outside the row
                                if (gx >= 0 && gx < Ex) v = __ldcg(reinterpret_cast<const float4 *>(q));
                            } else {
                                if (gx >= 0 && gx < Ex) v.x = __ldcg(q);
                                if (gx + 1 >= 0 && gx + 1 < Ex) v.y = __ldcg(q + 1);
                                if (gx + 2 >= 0 && gx + 2 < Ex) v.z = __ldcg(q + 2);
                                if (gx + 3 >= 0 && gx + 3 < Ex) v.w = __ldcg(q + 3);
                            }
                        }
                        use(i, v);
                        row += step_r + (c4 + step_c >= F4);
                        next();
                    }
                }
                if (!SCALED || attempt == 1) break;
                const int mx = (int)(__reduce_max_sync(0xffffffffu, mxu) >> 23);
                if (lane == 0) wmax[b * kLoadWarps + warp] = mx;
                __syncwarp();
                mbar_arrive(&maxb[b]);
                if (!bounded_wait(&maxb[b], (k >> 1) & 1, kWaitCycles)) {
                    break;  // the abort flag is set
                }
                int emax = wmax[b * kLoadWarps];
#pragma unroll
                for (int w = 1; w < kLoadWarps; ++w) emax = max(emax, wmax[b * kLoadWarps + w]);
                // |x| < 2^(emax - 126): keep the scale while 2^7 <= max |x| 2^es < 2^15 or the tile is
                // zero, else convert again with the largest value in [2^11, 2^12)
                const int top = emax - 126 + es;
                if (emax == 0 || (top <= 15 && top >= 8)) break;
                es = max(-126, min(127, 138 - emax));
            }
            if (*(volatile int *)abort_flag) break;
            // publish the scale: slot k & 3 was last read by the epilogue of tile
            // k - 4, which finished before the MMAs of tile k - 2 could start
            // (and those precede the MMAs of tile k - nbuf waited for above)
            if (SCALED && tid == 0) {
                eus[k & 3] = es;
                mbar_arrive(&eub[k & 3]);
            }
            fence_proxy_async_smem();
            mbar_arrive(&full[b]);
        }
    } else {
        // ---------------- epilogue (warps 12-19) ----------------
        // warp w reads TMEM lanes 32 q .. 32 q + 31 (q = w % 4, the lane quarter
        // a warp may access): rows 12 - 4q .. 15 - 4q of every block; half h of
        // the block-row pairs
        const int q = (warp - kEpiWarp) & 3, h = (warp - kEpiWarp) >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
        float *st = stage + (warp - kEpiWarp) * 4 * kStageRow;
        float *put_at = st + (3 - (lane >> 3)) * kStageRow + 7 - (lane & 7);
        int k = 0;
        bool ok = true;
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
            const int b = k & 1;
            int es = 0;
            if constexpr (SCALED) {
                if (!bounded_wait(&eub[k & 3], (k >> 2) & 1, kWaitCycles)) {
                    ok = false;
                    break;
                }
                es = eus[k & 3];
            }
            if (!bounded_wait(&done[b], (k >> 1) & 1, kWaitCycles)) {
                ok = false;
                break;
            }
            fence_after_thread_sync();
            int64_t Y0, X0;
            origin(id, &Y0, &X0);
            // written columns [x_lo, x_hi) and rows [y_lo, y_hi) of the tile
            const int x_lo = (int)max((int64_t)0, rh + p.band - X0), x_hi = (int)min((int64_t)kTX, Ex - rh - p.band - X0);
            const int y_lo = (int)max((int64_t)0, p.band - (Y0 - rh));
            const int y_hi = (int)min((int64_t)kBY * gn, ny - p.band - (Y0 - rh));
            const int vst = x_lo == 0 && x_hi == kTX ? p.vst : 0;
            // out = acc 2^(ew - 15 - es), as two in-range powers of two
            const int e = p.ew - 15 - es, e1 = e / 2, e2 = e - e1;
            const float s1 = SCALED ? pow2f(max(-126, min(127, e1))) : 1.0f;
            const float s2 = SCALED ? pow2f(max(-126, min(127, e2))) : 1.0f;
            float *const o = out + Y0 * Ex + X0;
            for (int g2 = 2 * h; g2 < gn; g2 += 4) {
                uint32_t v[16], c[16];
                __syncwarp();
                tmem_ld_32x32b_x16(lane_base + (uint32_t)b * aset + (uint32_t)(8 * g2), v);
                if (CORR) tmem_ld_32x32b_x16(lane_base + (uint32_t)b * aset + (uint32_t)(N + 8 * g2), c);
                tmem_ld_wait();
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int y = 16 * (g2 + s) + 12 - 4 * q;  // tile row of staging row 0
                    if (y >= y_hi || y + 4 <= y_lo) continue;
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float f = __uint_as_float(v[8 * s + j]);
                        if (CORR) f += __uint_as_float(c[8 * s + j]);
                        if (SCALED) f = f * s1 * s2;
                        put_at[8 * j] = f;
                    }
                    __syncwarp();
                    if (vst == 4) {
#pragma unroll
                        for (int it = 0; it < 2; ++it) {
                            const int rr = 2 * it + (lane >> 4), col = 4 * (lane & 15);
                            const float4 f = *reinterpret_cast<const float4 *>(st + rr * kStageRow + col);
                            if (y + rr >= y_lo && y + rr < y_hi)
                                *reinterpret_cast<float4 *>(o + (int64_t)(y + rr) * Ex + col) = f;
                        }
                    } else if (vst == 2) {
#pragma unroll
                        for (int rr = 0; rr < 4; ++rr) {
                            const float2 f = *reinterpret_cast<const float2 *>(st + rr * kStageRow + 2 * lane);
                            if (y + rr >= y_lo && y + rr < y_hi)
                                *reinterpret_cast<float2 *>(o + (int64_t)(y + rr) * Ex + 2 * lane) = f;
                        }
                    } else {
#pragma unroll
                        for (int it = 0; it < 8; ++it) {
                            const int rr = it >> 1, col = 32 * (it & 1) + lane;
                            const float f = st[rr * kStageRow + col];
                            if (y + rr >= y_lo && y + rr < y_hi && col >= x_lo && col < x_hi)
                                o[(int64_t)(y + rr) * Ex + col] = f;
                        }
                    }
                }
            }
            fence_before_thread_sync();
            mbar_arrive(&accfree[b]);
        }
        if (ok && p.debug_unmet && k > 0) {
            // test hook: a phase that never completes -> the bounded wait reports it
            bounded_wait(&done[(k - 1) & 1], (((k - 1) >> 1) & 1) ^ 1, kDebugWaitCycles);
        }
    }
    fence_before_thread_sync();
    __syncthreads();
    if (tid == 0 && *(volatile int *)abort_flag) atomicExch(&g_wide_error, 1);
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

// 16-bit forms.
template <int FORM>
__global__ void __launch_bounds__(kThreads, 1)
    tc2d_wide(const float *__restrict__ in, float *__restrict__ out, const __grid_constant__ WideParams p,
              int ntiles, int ntx)
{
    block_sweep<FORM>(in, out, p, ntiles, ntx);
}

// TF32 forms.
template <int FORM>
__global__ void __launch_bounds__(kThreads, 1)
    tc2d_ws(const float *__restrict__ in, float *__restrict__ out, const __grid_constant__ WideParams p, int ntiles,
            int ntx)
{
    block_sweep<FORM>(in, out, p, ntiles, ntx);
}

}  // namespace wide

namespace {

template <int FORM>
stencil_status launch_form(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    using namespace wide;
    const int r = p.pat.r, R = t * r;
    if (R > kMaxR) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core path: fused radius t*r must be <= 12");
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const BlockTile g = tc_block_tile(R, is_tf32(FORM), is_split(FORM), p.dims[1], p.ext[2], std::max(1, sms));
    if (g.gn == 0) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core tile does not fit in shared memory");
    WideParams wp;
    std::memset(&wp, 0, sizeof(wp));
    const std::vector<double> wt = compose_dense(p.pat, p.w, t);
    const int lines = 2 * R + 1;
    double wmax = 0;
    for (int i = 0; i < lines * lines; i++) {
        wp.w[i] = wt[i];
        wmax = std::max(wmax, std::fabs(wt[i]));
    }
    wp.R = R;
    wp.rh = r;
    wp.band = (t - 1) * r;
    wp.gn = g.gn;
    wp.nbuf = g.nbuf;
    wp.nc = g.nc;
    wp.pc = g.pc;
    wp.plane = (uint32_t)g.plane;
    wp.in_bytes = (uint32_t)g.in_bytes;
    wp.ew = 0;
    if (wmax > 0) std::frexp(wmax, &wp.ew);  // wmax < 2^ew
    wp.debug_unmet = p.debug_unmet_wait;
    wp.Ey = p.ext[1];
    wp.Ex = p.ext[2];
    wp.vec16 = (p.ext[2] % 4 == 0) && (reinterpret_cast<uintptr_t>(in) % 16 == 0);
    wp.xshift = wp.vec16 ? (4 - R % 4) % 4 : 0;  // (tile start - R) a multiple of 4
    // output rows start at element Y Ex + 64 k - xshift
    wp.vst = 1;
    for (int v : {4, 2})
        if (wp.vst == 1 && p.ext[2] % v == 0 && wp.xshift % v == 0 && reinterpret_cast<uintptr_t>(out) % (4 * v) == 0)
            wp.vst = v;
    auto kern = [] {
        if constexpr (is_tf32(FORM)) return tc2d_ws<FORM>;
        else return tc2d_wide<FORM>;
    }();
    stencil_status s = ensure_smem((const void *)kern, g.smem);
    if (s != STENCIL_OK) return s;
    const int64_t nty = (p.dims[1] + kBY * g.gn - 1) / (kBY * g.gn), ntx = (p.ext[2] + wp.xshift + kTX - 1) / kTX;
    const int64_t ntiles = nty * ntx;
    if (ntiles > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles, sms);
    kern<<<grid, kThreads, g.smem, st>>>((const float *)in, (float *)out, wp, (int)ntiles, (int)ntx);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "tc2d_wide launch");
}

}  // namespace

stencil_status launch_wide_sweep(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    switch (p.precision) {
    case STENCIL_PREC_F16: return launch_form<wide::kF16>(p, in, out, t, st);
    case STENCIL_PREC_F16X3: return launch_form<wide::kF16x3>(p, in, out, t, st);
    case STENCIL_PREC_BF16X3: return launch_form<wide::kBF16x3>(p, in, out, t, st);
    case STENCIL_PREC_TF32: return launch_form<wide::kTF32>(p, in, out, t, st);
    case STENCIL_PREC_TF32X3: return launch_form<wide::kTF32x3>(p, in, out, t, st);
    }
    return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core path: precision");
}

stencil_status read_wide_error(int *flag)
{
    int v = 0, zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_wide_error, sizeof(int));
    if (e == cudaSuccess && v) e = cudaMemcpyToSymbol(g_wide_error, &zero, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(e, "reading the wide kernel's error word");
    *flag = v;
    return STENCIL_OK;
}

}  // namespace gbs
