// k_tc.cu -- dispatch of the tensor-core sweeps and the FP64 MMA kernel: the
// t-step composite stencil (kernel fusion, paper Sec. 2.2.3, Eq. 3) run as
// banded Toeplitz GEMM tiles.
//
// FP32 grids run on the tcgen05 kernels of k_wide.cu (2-D) and k_wide3d.cu
// (3-D), FP64 grids in the exact-split form on k_split.cu.  Here:
// dmma2d_sweep, the Toeplitz formulation on the FP64 MMA mma.sync.m8n8k4
// (M = 8 output rows, N = 8 output columns, K = 4).
//
// All write interior points farther than (t-1) r from the boundary only:
// nearer points would need the halo re-imposed between the fused steps; the
// CUDA-core band kernel computes them stepwise.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "cu_kernels.cuh"
#include "launch.h"
#include "tc_layout.h"
#include "tc_ptx.cuh"

namespace gbs {

constexpr int kTcMaxR = 12;
constexpr int kTcMaxLines = 2 * kTcMaxR + 1;

struct TcParams {
    double w[kTcMaxLines * kTcMaxLines];  // composite w^(t), (2R+1) x (2R+1), row-major
    unsigned char kb_lo[kTcMaxLines], kb_hi[kTcMaxLines];
    int R, rh, band, nkb, nch;
    int64_t Ey, Ex;
};

namespace tcs {

__device__ __forceinline__ bool outside_band(int64_t iy, int64_t ix, int64_t ny, int64_t nx, int band)
{
    return iy >= band && ix >= band && ny - 1 - iy >= band && nx - 1 - ix >= band;
}

// ---------------------------------------------------------------------------
// FP64: mma.sync.m8n8k4 (A 8x4 row-major, B 4x8 column-major, C/D 8x8).
// 256 threads; a CTA owns 64 output rows x 64 output columns; warp w owns
// rows 8w..8w+7 and eight 8-column accumulators.
// ---------------------------------------------------------------------------
constexpr int DM_T = 64;

__device__ __forceinline__ void dmma(double &d0, double &d1, double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(d0), "+d"(d1)
                 : "d"(a), "d"(b));
}

__global__ void __launch_bounds__(256) dmma2d_sweep(const double *__restrict__ in, double *__restrict__ out,
                                                    const __grid_constant__ TcParams p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int R = p.R, lines = 2 * R + 1, nkb = p.nkb;  // K step 4
    const int W = DM_T + 8 * 0 + p.nch;                  // smem row length (doubles)
    const int H = DM_T + 2 * R;
    double *S = reinterpret_cast<double *>(smem_raw);
    double *Bf = S + (size_t)H * W;  // [ai][kb][lane] fragments: B[lane%4][lane/4]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t Y0 = p.rh + (int64_t)blockIdx.y * DM_T;
    const int64_t X0 = p.rh + (int64_t)blockIdx.x * DM_T;
    const int64_t ny = p.Ey - 2 * p.rh, nx = p.Ex - 2 * p.rh;

    for (int idx = tid; idx < lines * nkb * 32; idx += blockDim.x) {
        const int l = idx % 32, blk = idx / 32;
        const int ai = blk / nkb, kb = blk % nkb;
        const int k = kb * 4 + (l & 3), n = l >> 2;
        const int b = k - n - R;
        Bf[idx] = (b >= -R && b <= R) ? p.w[ai * lines + (b + R)] : 0.0;
    }
    for (int row = warp; row < H; row += 8) {
        const int64_t gy = Y0 - R + row;
        const bool rowok = gy >= 0 && gy < p.Ey;
        for (int x = lane; x < W; x += 32) {
            const int64_t gx = X0 - R + x;
            S[row * W + x] = (rowok && gx >= 0 && gx < p.Ex) ? __ldg(in + gy * p.Ex + gx) : 0.0;
        }
    }
    __syncthreads();

    const int g = lane >> 2, c = lane & 3;
    double acc[8][2];
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) acc[nb][0] = acc[nb][1] = 0.0;
    for (int ai = 0; ai < lines; ++ai) {
        const double *srow = S + (warp * 8 + g + ai) * W + c;
        for (int kb = p.kb_lo[ai]; kb <= p.kb_hi[ai]; ++kb) {
            const double b = Bf[(ai * nkb + kb) * 32 + lane];
#pragma unroll
            for (int nb = 0; nb < 8; ++nb) dmma(acc[nb][0], acc[nb][1], srow[nb * 8 + kb * 4], b);
        }
    }
    const int64_t gy = Y0 + warp * 8 + g, iy = gy - p.rh;
    if (iy < ny) {
#pragma unroll
        for (int nb = 0; nb < 8; ++nb) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t ix = X0 - p.rh + nb * 8 + 2 * c + h;
                if (ix < nx && outside_band(iy, ix, ny, nx, p.band)) out[gy * p.Ex + p.rh + ix] = acc[nb][h];
            }
        }
    }
}

}  // namespace tcs

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

stencil_status fill_params(const Plan &p, int t, int n_tile, int k_inst, TcParams *tp, TcLines *L)
{
    const int r = p.pat.r, R = t * r;
    if (R > kTcMaxR) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core path: fused radius t*r must be <= 12");
    *L = tc_lines_2d(p.pat.shape, r, t, n_tile, k_inst);
    const std::vector<double> &wt = composite(p, t);
    std::memset(tp, 0, sizeof(*tp));
    const int lines = 2 * R + 1;
    for (int i = 0; i < lines * lines; i++) tp->w[i] = wt[i];
    for (int a = 0; a < lines; a++) {
        tp->kb_lo[a] = (unsigned char)L->kb_lo[a];
        tp->kb_hi[a] = (unsigned char)L->kb_hi[a];
        if (L->kb_lo[a] > L->kb_hi[a]) {  // empty line
            tp->kb_lo[a] = 1;
            tp->kb_hi[a] = 0;
        }
    }
    tp->R = R;
    tp->rh = r;
    tp->band = (t - 1) * r;
    tp->nkb = L->nkb;
    tp->Ey = p.ext[1];
    tp->Ex = p.ext[2];
    return STENCIL_OK;
}

stencil_status launch_dmma2d(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    using namespace tcs;
    TcParams tp;
    TcLines L;
    stencil_status s = fill_params(p, t, 8, 4, &tp, &L);
    if (s != STENCIL_OK) return s;
    const int R = tp.R;
    // smem row: the widest window read is 8*7 + kext columns
    tp.nch = 8 * 7 + L.kext - DM_T;  // extra columns beyond DM_T
    if (tp.nch < 0) tp.nch = 0;
    const int W = DM_T + tp.nch, H = DM_T + 2 * R;
    const size_t smem = ((size_t)H * W + (size_t)(2 * R + 1) * L.nkb * 32) * 8;
    if (smem > 227 * 1024) return fail(STENCIL_ERR_UNSUPPORTED, "FP64 MMA tile does not fit in shared memory");
    s = ensure_smem((const void *)dmma2d_sweep, smem);
    if (s != STENCIL_OK) return s;
    const int64_t ny = p.dims[1], nx = p.dims[2];
    dim3 grid((unsigned)((nx + DM_T - 1) / DM_T), (unsigned)((ny + DM_T - 1) / DM_T));
    dmma2d_sweep<<<grid, 256, smem, st>>>((const double *)in, (double *)out, tp);
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? STENCIL_OK : cuda_fail(e, "dmma2d_sweep launch");
}

}  // namespace

stencil_status launch_tc_sweep(const Plan &p, const void *in, void *out, int t, cudaStream_t st)
{
    if (p.pat.d == 3 && p.dtype == STENCIL_F32 && p.precision == STENCIL_PREC_F16)
        return launch_wide3_sweep(p, in, out, t, st);  // t = 1: no band
    if (p.pat.d != 2) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core path: 3-D grids in FP32 with precision f16 only");
    stencil_status s;
    if (p.dtype == STENCIL_F64 && p.precision == STENCIL_PREC_OZAKI) {
        return launch_split_sweep(p, in, out, t, st);  // includes the band sweep
    } else if (p.dtype == STENCIL_F64) {
        s = launch_dmma2d(p, in, out, t, st);
    } else {
        s = launch_wide_sweep(p, in, out, t, st);  // TF32 / FP16 / BF16 forms (t r <= 12)
    }
    if (s != STENCIL_OK || t == 1) return s;
    // points within (t-1) r of the boundary: stepwise on CUDA cores
    return launch_cu_band(p, in, out, t, (t - 1) * p.pat.r, st);
}

stencil_status read_device_error(int *flag)
{
    int vs = 0, vw = 0, v3 = 0;
    stencil_status s = read_split_error(&vs);
    if (s != STENCIL_OK) return s;
    s = read_wide_error(&vw);
    if (s != STENCIL_OK) return s;
    s = read_wide3_error(&v3);
    if (s != STENCIL_OK) return s;
    *flag = vs | vw | v3;
    return STENCIL_OK;
}

}  // namespace gbs
