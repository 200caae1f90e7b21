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
// bits) and the weights likewise; the epilogue undoes both exactly.  The tile's
// largest |x| lands in [2^14, 65504]: the FP16 normal range starts at 2^-14, so
// values down to 2^-28 of the largest keep 11 bits, and the lo parts of f16x3
// stay exact to 2^-38 of it.  A tile is read once where that can be had: the
// epilogue warps, which wait most of the time, look at 512 values spread over the
// tile two tiles ahead, and the scale that puts the largest of those in
// [2^14, 2^15) cannot be below the rule's, so a tile converted with it keeps at
// least those bits; it is converted again, from L2, only if a value outside the
// sample is 2 to 4 times larger than all of it and would overflow.  The scale
// depends on the tile alone.  (The scale of the CTA's tile before, kept as long as
// the largest value fell in [2^7, 2^15), took seven bits off the small values
// beside a large one: 3 % less time on unaligned rows, none on aligned ones of
// 16384^2.)  BF16 has FP32's exponent range, any scale keeps its bits, and it does keep
// the tile's before.  TF32 needs no scale.
//
// A tile is hx = 1 or 2 such column groups of 64 side by side: an MMA of N = 128
// takes exactly half the time of one of N = 256 (64 / 128 cycles; ~50 is the
// least), so the f16 form takes 256 x 128 tiles (N = 128 twice), whose rows
// load in longer runs with less halo than 512 x 64.
//
// Persistent, warp specialised, one CTA per SM (768 threads): warps 0-14 load
// and convert the next tile into the other operand buffer (each thread keeps
// kBatch 16-byte loads in flight and starts the next tile's before the scale
// exchange), warp 23 issues the MMAs into the other TMEM accumulator, warps
// 15-22 read the previous accumulator back (tcgen05.ld), turn each 4 x 64 group
// of outputs through shared memory and store whole rows.  The MMA warp runs its
// loop converged with one elected lane issuing and the chunk count a
// compile-time constant: issued by a single diverged lane with run-time
// addressing, an MMA took ~70 cycles longer than its arithmetic (196 instead of
// 128 at N = 256, 133 instead of 64 at N = 128).  Every wait is bounded.  Only
// interior points farther than (t-1) r from the boundary are written; the
// CUDA-core band kernel computes the others.
//
// Measured, one fused sweep (line form before, block form now): Box-2D2R f16
// t = 4 on 16384^2 776 -> 476 us (HBM floor 317; a plain tiled copy that
// re-reads the same halo 415), f16x3 t = 4 on 7001 x 6007 (unaligned rows)
// 433 -> 178 us (171 without the sample), Box-2D1R TF32 t = 7 on 10240^2 654 (2:4 sparse form) -> 265 us.
// The loaders set the pace (15k cycles per 256 x 128 tile; MMAs 6.2k).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
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
constexpr int kTX = 64;                       // output columns of one MMA: 8 blocks
constexpr int kLoadWarps = 15;                // warps 0-14
constexpr int kLoaders = 32 * kLoadWarps;
constexpr int kEpiWarp = kLoadWarps;          // warps 15-22: TMEM lane quarter w % 4, two warps each
constexpr int kEpiWarps = 8;
constexpr int kMmaWarp = kLoadWarps + kEpiWarps;  // warp 23
constexpr int kThreads = 32 * (kMmaWarp + 1);
constexpr int kBatch = 8;                     // 16-byte loads kept in flight per loader thread
constexpr int kHeader = 1024;
constexpr int kStageRow = kTX + 8;             // epilogue staging: 4 rows of 64 outputs per warp, padded
constexpr int kStageBytes = kEpiWarps * 4 * kStageRow * 4;
constexpr unsigned long long kWaitCycles = 4ull << 30;       // ~2 s at 2 GHz
constexpr unsigned long long kDebugWaitCycles = 1ull << 22;  // ~2 ms: the test hook's limit

struct WideParams {
    double w[kMaxLines * kMaxLines];  // composite w^(t), (2R+1) x (2R+1), row-major
    int R, rh, band, ew;
    int gn;     // block rows per tile: 16 gn output rows, MMA N = 8 gn
    int hx;     // 64-column halves per tile, each with MMAs of its own
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

// The scale exponent that puts a largest |x| of these bits in [2^14, 2^15) (clamped to FP32's range).
__device__ __forceinline__ int scale_of(unsigned mx)
{
    return max(-126, min(127, 141 - (int)(mx >> 23)));  // |x| < 2^((mx >> 23) - 126)
}

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
    constexpr bool SAMPLED = SCALED && FORM != kBF16x3;  // BF16 has FP32's range: any scale keeps its bits
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
    uint64_t *smpb = reinterpret_cast<uint64_t *>(smem + 112);    // [4] a tile's sample taken
    unsigned *wmax = reinterpret_cast<unsigned *>(smem + 160);    // [2][kLoadWarps] largest |x| of a tile
    unsigned *wsmp = reinterpret_cast<unsigned *>(smem + 288);    // [4][kEpiWarps] and of its sample
    int *eus = reinterpret_cast<int *>(smem + 416);               // [4] input scale exponent per tile
    const int R = p.R, lines = 2 * R + 1, nc = p.nc, pc = p.pc, gn = p.gn, hx = p.hx, nbuf = p.nbuf;
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
    const uint32_t aset = (uint32_t)(N * hx) * (CORR ? 2 : 1);  // TMEM columns of one accumulator set

    // Up to the wait below a block reads kernel parameters only, so the strip is
    // written while the kernel in front of it finishes (launch_chained).  TMEM is
    // taken after the wait: the blocks of that kernel hold none any more.  Measured,
    // unchained before: f16x3 7001 x 6007, 8 steps 346 -> 336 us; TF32 1500 x 1411,
    // 8 steps 53 -> 44 us; f16 300 x 411, 8 steps 50 -> 42 us.
    if (tid == 0) {
        *abort_flag = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(&full[b], kLoaders);
            mbar_init(&done[b], 1);
            mbar_init(&accfree[b], 32 * kEpiWarps);
            mbar_init(&maxb[b], kLoaders);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(&eub[s], 1);
            mbar_init(&smpb[s], kEpiWarps);
        }
        fence_mbar_init();
    }
    // Weight strip: core matrix (L, c), L = ky + g, holds line L - 15.  Each
    // weight is rounded to its operand parts once (FP64 arithmetic runs at two
    // lanes per cycle), then the strip is a copy of table entries.
    {
        uint32_t *const th = reinterpret_cast<uint32_t *>(stage), *const tl = th + kMaxLines * kMaxLines;
        static_assert(2 * 4 * kMaxLines * kMaxLines <= kStageBytes, "the table fits the epilogue's staging rows");
        const double wsc = SCALED ? ldexp(1.0, 15 - p.ew) : 1.0;  // |w| 2^(15 - ew) < 2^15: exact scaling
        for (int e = tid; e < lines * lines; e += kThreads) {
            const double wv = p.w[e] * wsc;
            if constexpr (TF) {
                const float h = to_tf32((float)wv);
                th[e] = __float_as_uint(h);
                if (SPLIT) tl[e] = __float_as_uint(to_tf32((float)(wv - (double)h)));
            } else {
                using O = Op<FORM == kBF16x3>;
                const uint16_t h = O::bits(wv);
                th[e] = h;
                if (SPLIT) tl[e] = O::bits(wv - O::value(h));
            }
        }
        __syncthreads();
        const int nelem = (31 + 2 * R) * nc * 8 * CE;
        for (int e = tid; e < nelem; e += kThreads) {
            const int j = e % CE, i = (e / CE) & 7, core = e / (8 * CE);
            const int d = core / nc - 15, idx = CE * (core % nc) + j + i - 7;
            const bool tap = d >= 0 && d < lines && idx >= 0 && idx < lines;
            const uint32_t h = tap ? th[d * lines + idx] : 0u, l = SPLIT && tap ? tl[d * lines + idx] : 0u;
            if constexpr (TF) {
                reinterpret_cast<uint32_t *>(Whi)[e] = h;
                if (SPLIT) reinterpret_cast<uint32_t *>(Wlo)[e] = l;
            } else {
                reinterpret_cast<uint16_t *>(Whi)[e] = (uint16_t)h;
                if (SPLIT) reinterpret_cast<uint16_t *>(Wlo)[e] = (uint16_t)l;
            }
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (warp == kMmaWarp) tmem_alloc(tmem_slot, 512);
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
        *X0 = (int64_t)(id % ntx) * (kTX * hx) - p.xshift;
    };

    if (warp == kMmaWarp) {
        // ---------------- MMA issuer (the whole warp; one elected lane issues) ----------------
        auto mma_loop = [&](auto nc_const, auto hx_const) {
            constexpr int NC = decltype(nc_const)::value, HX = decltype(hx_const)::value;
            const uint32_t leader = elect_lane();
            const uint32_t idesc = instr_desc(TF ? kFmtTF32 : (FORM == kBF16x3 ? kFmtBF16 : kFmtF16), 128, N);
            const uint32_t wbase = smem_u32(Whi), rowb = (uint32_t)pc * 16;
            // descriptors of chunk pairs of one row (c) and of one chunk of two rows (r): the low
            // word holds LBO and the start address, which advances; SBO sits in the high word
            const uint64_t a_c = smem_desc(wbase, 128, NC * 128), a_r = smem_desc(wbase, NC * 128, NC * 128);
            const uint32_t ahi = (uint32_t)(a_c >> 32), ac0 = (uint32_t)a_c, ar0 = (uint32_t)a_r;
            const uint32_t dlo_a = strip_bytes >> 4, dlo_b = (nbuf * in_bytes) >> 4;
            const uint32_t n_tmem = (uint32_t)N;
            int k = 0;
            for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
                const int b = k & 1;
                bool up = bounded_wait(&full[b], (k >> 1) & 1, kWaitCycles);
                if (k >= 2) up = up && bounded_wait(&accfree[b], ((k - 2) >> 1) & 1, kWaitCycles);
                if (!__all_sync(0xffffffffu, up)) break;
                fence_after_thread_sync();
                const uint32_t ib = smem_u32(ibase + (nbuf == 2 ? b : 0) * in_bytes);
                const uint64_t b_c = smem_desc(ib, TF ? p.plane : 16u, 16 * rowb), b_r = smem_desc(ib, rowb, 16 * rowb);
                const uint32_t bhi = (uint32_t)(b_c >> 32);
                uint32_t ac = ac0, ar = ar0, bc = (uint32_t)b_c, br = (uint32_t)b_r;
                const uint32_t d0 = tmem + (uint32_t)b * aset;
                // one K step of every column group; FIRST: the accumulators start at zero
                auto issue = [&](auto first, uint32_t da, uint32_t db) {
                    constexpr int ACC = decltype(first)::value ? 0 : 1;
#pragma unroll
                    for (int h = 0; h < HX; ++h) {
                        const uint32_t d = d0 + h * n_tmem, dbh = db + 8 * h;  // 8 units: the next 64 columns
                        if constexpr (TF) {
                            mma_tf32_warp<ACC>(leader, d, da, ahi, dbh, bhi, idesc);
                            if constexpr (SPLIT) {
                                const uint32_t dc = d + HX * n_tmem;
                                mma_tf32_warp<ACC>(leader, dc, da, ahi, dbh + dlo_b, bhi, idesc);
                                mma_tf32_warp<1>(leader, dc, da + dlo_a, ahi, dbh, bhi, idesc);
                            }
                        } else {
                            mma_f16_warp<ACC>(leader, d, da, ahi, dbh, bhi, idesc);
                            if constexpr (SPLIT) {
                                mma_f16_warp<1>(leader, d, da, ahi, dbh + dlo_b, bhi, idesc);
                                mma_f16_warp<1>(leader, d, da + dlo_a, ahi, dbh, bhi, idesc);
                            }
                        }
                    }
                };
                auto two_rows = [&](auto first) {
                    constexpr bool F = decltype(first)::value;
#pragma unroll
                    for (int y = 0; y < 2; ++y)
#pragma unroll
                        for (int c = 0; c + 1 < NC; c += 2) {
                            const uint32_t da = ac + (y * NC + c) * 8, db = bc + (y ? pc : 0) + (TF ? c / 2 : c);
                            if (F && y == 0 && c == 0) issue(std::true_type{}, da, db);
                            else issue(std::false_type{}, da, db);
                        }
                    if constexpr ((NC & 1) != 0)
                        issue(std::false_type{}, ar + (NC - 1) * 8, br + (TF ? (NC - 1) / 2 : NC - 1));
                    ac += 2 * NC * 8;
                    ar += 2 * NC * 8;
                    bc += (uint32_t)(2 * pc);
                    br += (uint32_t)(2 * pc);
                };
                two_rows(std::true_type{});
                for (int ky = 2; ky < kBY + 2 * R; ky += 2) two_rows(std::false_type{});
                mma_commit_warp(leader, &done[b]);
            }
            // the last tiles' MMAs complete before the TMEM is released
            for (int j = k - 2; j < k; ++j)
                if (j >= 0) {
                    const unsigned long long t0 = clock64();
                    while (!mbar_try_wait(&done[j & 1], (j >> 1) & 1) && clock64() - t0 < kWaitCycles) {
                    }
                }
        };
        auto with_hx = [&](auto nc_const) {
            if (hx == 2) mma_loop(nc_const, std::integral_constant<int, 2>{});
            else mma_loop(nc_const, std::integral_constant<int, 1>{});
        };
        switch (nc) {
        case 2: if constexpr (!TF) with_hx(std::integral_constant<int, 2>{}); break;
        case 3: with_hx(std::integral_constant<int, 3>{}); break;
        case 4: with_hx(std::integral_constant<int, 4>{}); break;
        case 5: if constexpr (TF) with_hx(std::integral_constant<int, 5>{}); break;
        case 6: if constexpr (TF) with_hx(std::integral_constant<int, 6>{}); break;
        case 7: if constexpr (TF) with_hx(std::integral_constant<int, 7>{}); break;
        case 8: if constexpr (TF) with_hx(std::integral_constant<int, 8>{}); break;
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
        const int64_t wrap = Ex - 4 * F4, step = step_r * Ex + 4 * step_c;
        const float *q = in;  // the next item to load: its address
        int c4 = 0;           // and its quad of the row
        auto next = [&] {
            q += step;
            c4 += step_c;
            if (c4 >= F4) {
                c4 -= F4;
                q += wrap;
            }
        };
        // the staged region lies inside the stored array (no bounds tests), and
        // its rows are 16-byte aligned
        auto is_fast = [&](int64_t Y0, int64_t X0) {
            return vec16 && X0 - R >= 0 && X0 - R + 8 * pc <= Ex && Y0 - R >= 0 && Y0 - R + rows <= Ey;
        };
        float4 v[kBatch] = {};  // loads in flight: items of the current (fast) tile
        auto start_tile = [&](int64_t Y0, int64_t X0) {
            q = in + (Y0 - R + row0) * Ex + (X0 - R + 4 * col0);
            c4 = col0;
        };
        auto start_fast = [&](int64_t Y0, int64_t X0) {
            start_tile(Y0, X0);
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (tid + u * kLoaders < items) v[u] = __ldcg(reinterpret_cast<const float4 *>(q));
                next();
            }
        };
        bool started = false;  // v holds this tile's first items
        int es = 12;  // the tile's scale exponent (BF16: first the tile's before)
        int k = 0;
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
            const int b = k & 1;
            int64_t Y0, X0;
            origin(id, &Y0, &X0);
            // the operand buffer is free once the MMAs of tile k - nbuf completed
            if (nbuf == 2 && k >= 2 && !bounded_wait(&done[b], ((k - 2) >> 1) & 1, kWaitCycles)) break;
            if (nbuf == 1 && k >= 1 && !bounded_wait(&done[b ^ 1], ((k - 1) >> 1) & 1, kWaitCycles)) break;
            unsigned char *hi = ibase + (nbuf == 2 ? b : 0) * in_bytes, *lo = hi + nbuf * in_bytes;
            if constexpr (SAMPLED) {  // first the sample's scale
                if (!bounded_wait(&smpb[k & 3], (k >> 2) & 1, kWaitCycles)) break;
                unsigned m = 0;
#pragma unroll
                for (int w = 0; w < kEpiWarps; ++w) m = max(m, wsmp[(k & 3) * kEpiWarps + w]);
                es = scale_of(m);
            }
            // Interior tiles: no per-load bounds tests.  Rows that are not 16-byte
            // multiples are read as the two aligned 16-byte words around each
            // quad (the region then keeps a stored row free above and below, so
            // both words lie inside the array).
            const bool fast = is_fast(Y0, X0);
            const bool fast_u = !vec16 && X0 - R >= 0 && X0 - R + 8 * pc <= Ex && Y0 - R >= 1 &&
                                Y0 - R + rows + 1 <= Ey;
            for (int attempt = 0;; ++attempt) {
                const float xs = SCALED ? pow2f(es) : 1.0f;
                unsigned mxu = 0;
                auto use = [&](int i, const float4 &x) {
                    if (SCALED) mxu = max_abs(mxu, x);
                    put<FORM>(hi, lo, i, x, xs, p.plane);
                };
                if (fast) {
                    if (!started) start_fast(Y0, X0);
                    for (int i0 = tid; i0 < items; i0 += kBatch * kLoaders) {
#pragma unroll
                        for (int u = 0; u < kBatch; ++u) {
                            const int i = i0 + u * kLoaders;
                            if (i < items) use(i, v[u]);
                            if (i + kBatch * kLoaders < items) v[u] = __ldcg(reinterpret_cast<const float4 *>(q));
                            next();
                        }
                    }
                    started = false;
                    // the next tile's first loads run during the exchange and the waits
                    if (attempt == 0 && id + (int)gridDim.x < ntiles) {
                        int64_t Y1, X1;
                        origin(id + gridDim.x, &Y1, &X1);
                        if (is_fast(Y1, X1)) {
                            start_fast(Y1, X1);
                            started = true;
                        }
                    }
                } else if (fast_u) {
                    start_tile(Y0, X0);
                    constexpr int U = kBatch / 2;  // v[u], v[U + u]: the two words of a quad
                    for (int i0 = tid; i0 < items; i0 += U * kLoaders) {
                        int sh = 0;
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const int s = (int)(reinterpret_cast<uintptr_t>(q) >> 2) & 3;
                            sh |= s << (2 * u);
                            if (i0 + u * kLoaders < items) {
                                const float4 *a4 = reinterpret_cast<const float4 *>(q - s);
                                v[u] = ld_chained(a4);
                                if (s) v[U + u] = ld_chained(a4 + 1);  // in L1: the next lane's first word
                            }
                            next();
                        }
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (i0 + u * kLoaders >= items) continue;
                            // quad = values s .. s + 3 of (a, e): shift by two, then by one
                            const int s = sh >> (2 * u);
                            const float4 a = v[u], e = v[U + u];
                            const float4 a2 = (s & 2) ? make_float4(a.z, a.w, e.x, e.y) : a;
                            const float n4 = (s & 2) ? e.z : e.x;
                            use(i0 + u * kLoaders, (s & 1) ? make_float4(a2.y, a2.z, a2.w, n4) : a2);
                        }
                    }
                } else {
                    // edge tiles: every value tested; cells outside the stored array are zero
                    start_tile(Y0, X0);
                    int row = row0;
                    for (int i = tid; i < items; i += kLoaders) {
                        const int64_t gy = Y0 - R + row, gx = X0 - R + 4 * c4;
                        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (gy >= 0 && gy < Ey) {
                            if (vec16) {
                                // X0 - R is a multiple of 4: the quad lies wholly inside or outside the row
                                if (gx >= 0 && gx < Ex) x = __ldcg(reinterpret_cast<const float4 *>(q));
                            } else {
                                if (gx >= 0 && gx < Ex) x.x = __ldcg(q);
                                if (gx + 1 >= 0 && gx + 1 < Ex) x.y = __ldcg(q + 1);
                                if (gx + 2 >= 0 && gx + 2 < Ex) x.z = __ldcg(q + 2);
                                if (gx + 3 >= 0 && gx + 3 < Ex) x.w = __ldcg(q + 3);
                            }
                        }
                        use(i, x);
                        row += step_r + (c4 + step_c >= F4);
                        next();
                    }
                }
                if (!SCALED || attempt == 1) break;
                mxu = __reduce_max_sync(0xffffffffu, mxu);
                if (lane == 0) wmax[b * kLoadWarps + warp] = mxu;
                __syncwarp();
                mbar_arrive(&maxb[b]);
                if (!bounded_wait(&maxb[b], (k >> 1) & 1, kWaitCycles)) {
                    break;  // the abort flag is set
                }
                mxu = wmax[b * kLoadWarps];
#pragma unroll
                for (int w = 1; w < kLoadWarps; ++w) mxu = max(mxu, wmax[b * kLoadWarps + w]);
                if constexpr (SAMPLED) {
                    // keep the scale if it is the rule's for the whole tile or the largest value still fits FP16
                    const int want = scale_of(mxu);
                    if (es == want || __uint_as_float(mxu) * pow2f(es) <= 65504.0f) break;
                    es = want;
                } else {
                    // keep the scale while 2^7 <= max |x| 2^es < 2^15 or the tile is zero, else [2^11, 2^12)
                    const int emax = (int)(mxu >> 23), top = emax - 126 + es;
                    if (emax == 0 || (top <= 15 && top >= 8)) break;
                    es = max(-126, min(127, 138 - emax));
                }
                started = false;  // converting again reloads the tile into v
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
        // ---------------- epilogue (warps 15-22) ----------------
        // warp w reads TMEM lanes 32 q .. 32 q + 31 (q = w % 4, the lane quarter
        // a warp may access): rows 12 - 4q .. 15 - 4q of every block; every
        // other pair of block rows
        const int q = warp & 3, h = (warp - kEpiWarp) >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
        float *st = stage + (warp - kEpiWarp) * 4 * kStageRow;
        float *put_at = st + (3 - (lane >> 3)) * kStageRow + 7 - (lane & 7);
        // This thread's two of the 512 values of a sample of tile id: 8 values of a row at 64 places spread over
        // the staged region (0 outside the stored array).  Whole 32-byte sectors, because the tile itself comes
        // three tiles later and HBM may read them twice: single values cost f16 on 16384^2 10 %.
        auto take_sample = [&](int id, float *x) {
            x[0] = x[1] = 0.0f;
            if (id >= ntiles) return;
            const int rows = kBY * gn + 2 * R, place = (tid - 32 * kEpiWarp) >> 2;
            int64_t Y0, X0;
            origin(id, &Y0, &X0);
            const int64_t gy = Y0 - R + place * rows / 64;
            const int64_t gx = X0 - R + (37 * place & 63) * (8 * pc - 8) / 63 + 2 * (lane & 3);
            if (gy < 0 || gy >= Ey) return;
            const float *s = in + gy * Ex + gx;
            if (gx >= 0 && gx < Ex) x[0] = __ldcg(s);
            if (gx + 1 >= 0 && gx + 1 < Ex) x[1] = __ldcg(s + 1);
        };
        // post the largest of a sample as that of the CTA's tile k (slot k & 3 was last read for tile k - 4, which
        // the loaders left before the epilogue of tile k - 3 could end)
        auto post_sample = [&](int k, const float *x) {
            const unsigned m = __reduce_max_sync(
                0xffffffffu, max(__float_as_uint(x[0]) & 0x7fffffffu, __float_as_uint(x[1]) & 0x7fffffffu));
            if (lane == 0) {
                wsmp[(k & 3) * kEpiWarps + warp - kEpiWarp] = m;
                mbar_arrive(&smpb[k & 3]);
            }
            __syncwarp();
        };
        float ahead[2];  // the sample of the tile two ahead, in flight while a tile is written
        int k = 0;
        bool ok = true;
        if constexpr (SAMPLED) {
            float next[2];
            take_sample(blockIdx.x, ahead);
            take_sample(blockIdx.x + gridDim.x, next);
            post_sample(0, ahead);
            post_sample(1, next);
            take_sample(blockIdx.x + 2 * gridDim.x, ahead);
        }
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x, ++k) {
            const int b = k & 1;
            int es = 0;
            if constexpr (SAMPLED) {
                post_sample(k + 2, ahead);
                take_sample(id + 3 * (int)gridDim.x, ahead);
            }
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
            // written rows [y_lo, y_hi) of the tile
            const int y_lo = (int)max((int64_t)0, p.band - (Y0 - rh));
            const int y_hi = (int)min((int64_t)kBY * gn, ny - p.band - (Y0 - rh));
            // out = acc 2^(ew - 15 - es), as two in-range powers of two
            const int e = p.ew - 15 - es, e1 = e / 2, e2 = e - e1;
            const float s1 = SCALED ? pow2f(max(-126, min(127, e1))) : 1.0f;
            const float s2 = SCALED ? pow2f(max(-126, min(127, e2))) : 1.0f;
            for (int pr = h; pr < hx * (gn / 2); pr += 2) {
                const int hc = pr >= gn / 2, g2 = 2 * (pr - hc * (gn / 2));  // column half, first block row
                // written columns [x_lo, x_hi) of the half
                const int64_t gx0 = X0 + hc * kTX;
                const int x_lo = (int)max((int64_t)0, rh + p.band - gx0);
                const int x_hi = (int)min((int64_t)kTX, Ex - rh - p.band - gx0);
                const int vst = x_lo == 0 && x_hi == kTX ? p.vst : 0;
                float *const o = out + Y0 * Ex + gx0;
                const uint32_t col = (uint32_t)b * aset + (uint32_t)(hc * N + 8 * g2);
                uint32_t v[16], c[16];
                __syncwarp();
                tmem_ld_32x32b_x16(lane_base + col, v);
                if (CORR) tmem_ld_32x32b_x16(lane_base + col + (uint32_t)(N * hx), c);
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
    const std::vector<double> &wt = composite(p, t);
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
    wp.hx = g.hx;
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
    constexpr size_t kOneBlockSmem = 116 * 1024;  // more than half of an SM's
    stencil_status s = ensure_smem((const void *)kern, std::max(g.smem, kOneBlockSmem));
    if (s != STENCIL_OK) return s;
    const int64_t nty = (p.dims[1] + kBY * g.gn - 1) / (kBY * g.gn), ntx = (p.ext[2] + wp.xshift + kTX * g.hx - 1) / (kTX * g.hx);
    const int64_t ntiles = nty * ntx;
    if (ntiles > 0x7fffffff) return fail(STENCIL_ERR_UNSUPPORTED, "too many tiles");
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles, sms);
    // one block per SM (each takes all of TMEM), also where the tile's shared memory would let two in
    const cudaError_t e = launch_chained(kern, grid, kThreads, std::max(g.smem, kOneBlockSmem), st,
                                         (const float *)in, (float *)out, wp, (int)ntiles, (int)ntx);
    if (e == cudaSuccess) note_launch();
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
