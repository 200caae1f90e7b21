// tc_layout.h -- geometry of the tensor-core (Toeplitz) formulation.  The line
// form below is the reference layout: stencil_plan_tc_layout exports it, the
// sparsity factor S (paper Sec. 2.2.2) and the dispatcher's roofs are computed from
// it, and the FP64 MMA kernel (k_tc.cu), the exact-split kernel (k_split.cu) and the
// 3-D kernel (k_wide3d.cu) issue exactly the MMAs counted here.  The 2-D FP32 kernels
// (k_wide.cu) issue the denser block form (BlockTile, further down): fewer MMAs for
// the same products.
//
// The t-step composite kernel w^(t) of radius R = t*r is applied as a sum
// over its rows ("lines"; in 3-D over (plane,row) pairs): for line a,
//     out[y][x0 + n] += sum_k In[y + a][x0 - R + k] * B_a[k][n],
//     B_a[k][n] = w^(t)[a][k - n - R]   (zero outside |k - n - R| <= h_a),
// a GEMM whose M axis runs over output rows y, whose N axis is a window of
// n_tile output columns and whose K axis is the input window of
// n_tile + 2R columns, padded to the MMA K step.  Line a only needs the
// K blocks that touch its band |b| <= h_a; the others are skipped.
// S = useful MACs / issued MACs = sum_a (2 h_a + 1) / sum_a (issued K of a).
#pragma once

#include <algorithm>
#include <cstdlib>
#include <vector>

namespace gbs {

struct TcLines {
    int R = 0, n_tile = 8, k_inst = 8, kext = 0, nkb = 0;
    std::vector<int> half;          // h_a per line (2R+1 lines in 2-D), -1 = empty line
    std::vector<int> kb_lo, kb_hi;  // K-block range issued per line (lo > hi: none)
    double useful = 0, issued = 0;  // per output point
    double sparsity() const { return issued > 0 ? useful / issued : 0.0; }
};

// Half-width of line a (2-D) of the composite: a box line spans R; a star
// line spans r (t - ceil(|a|/r)) (the t-fold star sum is the set of p with
// sum_i ceil(|p_i|/r) <= t).
inline int composite_half(int shape, int r, int t, int a)
{
    const int R = t * r;
    if (shape == 0) return R;
    const int ca = (std::abs(a) + r - 1) / r;
    return ca > t ? -1 : r * (t - ca);
}

inline TcLines tc_lines_2d(int shape, int r, int t, int n_tile, int k_inst)
{
    TcLines L;
    L.R = t * r;
    L.n_tile = n_tile;
    L.k_inst = k_inst;
    L.kext = (n_tile + 2 * L.R + k_inst - 1) / k_inst * k_inst;
    L.nkb = L.kext / k_inst;
    for (int a = -L.R; a <= L.R; a++) {
        const int h = composite_half(shape, r, t, a);
        L.half.push_back(h);
        if (h < 0) {
            L.kb_lo.push_back(1);
            L.kb_hi.push_back(0);
            continue;
        }
        // non-zero k: R - h <= k <= R + h + n_tile - 1
        const int lo = (L.R - h) / k_inst;
        const int hi = std::min(L.nkb - 1, (L.R + h + n_tile - 1) / k_inst);
        L.kb_lo.push_back(lo);
        L.kb_hi.push_back(hi);
        L.useful += 2 * h + 1;
        L.issued += (double)(hi - lo + 1) * k_inst;
    }
    return L;
}

// MMA N (output columns per Toeplitz block) of the TF32 / TF32x3 line form: the widest of 32, 16, 8 whose operands fit in 227 KB of
// shared memory -- B blocks (x2 split) plus double-buffered A tiles (hi, and
// lo when split) of 128 + 2R rows (rounded up to 8) by (NACC-1)*N + kext columns.
inline int tc_ws_ntile(int shape, int r, int t, bool split)
{
    const int R = t * r;
    const int hs = (128 + 2 * R + 7) / 8 * 8;  // chunk columns 128-byte aligned (TMA destinations)
    const int cand[3][2] = {{32, 2}, {16, 2}, {8, 4}};
    for (auto &c : cand) {
        const int n = c[0], nacc = c[1];
        TcLines L = tc_lines_2d(shape, r, t, n, 8);
        const long a = (long)((n * (nacc - 1) + L.kext) / 4) * hs * 16;
        const long b = (long)(2 * R + 1) * L.nkb * (n / 8) * 256;
        const long smem = 128 + b * (split ? 2 : 1) + a * (split ? 4 : 2);
        if (smem <= 227 * 1024) return n;
    }
    return 8;
}

// Line form of the FP16 / BF16 precisions: the Toeplitz factor of line a over
// 128 output columns (stored in reverse order, A[m'][k] depends on k + m' only)
// and the window of 128 + 2R columns in K blocks of 16.  This is the layout
// stencil_plan_tc_layout exports and the sparsity S and the model of these
// precisions refer to (every R <= kWideMaxR has one); rows per tile as the
// operands of that form fit in 227 KB.  The 2-D kernels issue the denser block
// form below; the 3-D kernel (tc3d_wide) issues the line form.
constexpr int kWideMaxR = 12;

inline int tc_wide_nrows(int r, int t, bool split)
{
    const int R = t * r;
    if (R > kWideMaxR) return 0;
    return !split && R <= 9 ? 256 : 128;
}

// Block form of the 2-D kernels (k_wide.cu): MMA rows = the 16 x 8 outputs of a
// block, MMA columns = 8 gn block positions (8 across, gn down), K = the
// 16-byte chunks of the block's (16 + 2R) x (8 + 2R) neighbourhood; a tile has
// hx such groups of 64 columns side by side.
struct BlockTile {
    int gn = 0;    // block rows: the tile is 16 gn x 64 hx outputs (0: no tile)
    int hx = 1;
    int nbuf = 0;  // operand buffers
    int nc = 0;    // 16-byte chunks of a neighbourhood row
    int pc = 0;    // 8-column units of a staged row
    int mmas = 0;  // MMAs of a tile (one product)
    size_t plane = 0, in_bytes = 0, smem = 0;
};

inline BlockTile tc_block_geom(int R, bool tf32, bool split, int gn, int hx, int nbuf)
{
    BlockTile g;
    const int ce = tf32 ? 4 : 8, rows = 16 * gn + 2 * R;
    g.gn = gn;
    g.hx = hx;
    g.nbuf = nbuf;
    g.nc = (8 + 2 * R + ce - 1) / ce;
    g.pc = 8 * hx + (tf32 ? (g.nc - 1) / 2 : g.nc - 1);
    g.mmas = (16 + 2 * R) / 2 * g.nc * hx;
    const size_t row = (size_t)g.pc * 16;
    // TF32: the odd-chunk plane starts 64 bytes off a 128-byte boundary
    // distance, so that a quarter warp's four even and four odd chunks hit
    // distinct banks
    g.plane = tf32 ? ((size_t)rows * row + 127) / 128 * 128 + 64 : 0;
    g.in_bytes = ((tf32 ? g.plane : 0) + (size_t)rows * row + 127) / 128 * 128;
    // 1 KB header, 8 epilogue warps' staging (4 x 72 FP32), strips, buffers
    g.smem = 1024 + 8 * 4 * 72 * 4 +
             ((size_t)(31 + 2 * R) * g.nc * 128 + nbuf * g.in_bytes) * (split ? 2 : 1);
    return g;
}

// The tile of a grid with ny interior rows and ex stored columns on `sms` SMs:
// the least (rounds of CTAs) x (cycles per tile) over gn = 32 .. 4, hx = 2 or 1
// and two operand buffers or one (one only where no two fit).  Cycles per
// tile: an MMA takes N / 2 = 4 gn cycles, at least 50 (measured); staging 1.0 per
// 16 bytes; HBM 1.15 x 8 bytes per output at 21.5 bytes per cycle and SM.  They
// overlap with two operand buffers; with one, staging and MMAs take turns.
// 2000 cycles per tile do not overlap (first loads, scale exchange, hand-over).
// The terms rank tiles; their sum is no prediction: fitted to FP16 t = 4 on 16384^2
// (16k cycles per 256 x 128 tile, 18k measured), it gives 9k for the TF32 t = 7 tile on
// 10240^2 that takes 13k, and half of what a sweep of a few rounds takes, whose
// strips and first loads it leaves out.
inline BlockTile tc_block_tile(int R, bool tf32, bool split, int64_t ny, int64_t ex, int sms)
{
    BlockTile best;
    double best_cost = 0;
    for (int hx : {2, 1})
        for (int gn : {32, 24, 16, 12, 8, 6, 4}) {
            // N = 8 gn: a multiple of 16 up to 256; TMEM holds two sets of hx accumulators
            // (TF32x3: two accumulators each)
            if (8 * gn * hx * (tf32 && split ? 4 : 2) > 512) continue;
            for (int nbuf : {2, 1}) {
                const BlockTile g = tc_block_geom(R, tf32, split, gn, hx, nbuf);
                if (g.smem > 227 * 1024) continue;
                const double mma = g.mmas * (split ? 3.0 : 1.0) * std::max(50.0, 4.0 * gn);
                const double load = 1.0 * (16 * gn + 2 * R) * 2 * g.pc;
                const double hbm = 1.15 * 8.0 * (16.0 * gn * 64.0 * hx) / 21.5;
                const int64_t tiles = ((ny + 16 * gn - 1) / (16 * gn)) * ((ex + 3 + 64 * hx - 1) / (64 * hx));
                const double cost = (double)((tiles + sms - 1) / sms) *
                                    (std::max(hbm, nbuf == 2 ? std::max(mma, load) : mma + load) + 2000.0);
                if (best.gn == 0 || cost < 0.999 * best_cost) {
                    best = g;
                    best_cost = cost;
                }
                break;
            }
        }
    return best;
}

// 3-D wide FP16 kernel (tc3d_wide, one step per sweep): the Toeplitz factor
// of line (dz, dy) is the A operand as in tc2d_wide (one strip per line, two
// strip sets: the weights are rescaled per output plane), the input is
// staged one plane tile of nr + 2R rows at a time into a ring of 2R + 2
// slots.  Lines: the (dz, dy) pairs with a non-zero weight, (2r+1)^2 for a
// box and 4r + 1 for a star.
struct Wide3Geom {
    int nkb, delta, hs, slots;
    size_t strip_bytes, in_bytes, smem;
};

inline int tc_wide3_lines(int shape, int r) { return shape == 0 ? (2 * r + 1) * (2 * r + 1) : 4 * r + 1; }  // 0: box

inline Wide3Geom tc_wide3_geom(int R, int nlines, int nr)
{
    Wide3Geom g;
    g.nkb = (128 + 2 * R + 15) / 16;
    g.delta = std::max(2 * g.nkb, (127 + 2 * R) / 8 + 1);
    g.hs = (nr + 2 * R) | 1;
    g.slots = 2 * R + 2;
    g.strip_bytes = (size_t)((nlines - 1) * g.delta + 2 * g.nkb + 15) * 128;
    g.in_bytes = (size_t)(2 * g.nkb) * g.hs * 16;
    // 1 KB header, two strip sets, the ring of input slots
    g.smem = 1024 + 2 * g.strip_bytes + (size_t)g.slots * g.in_bytes;
    return g;
}

// Output rows per tile of the 3-D kernel: the first of 128, 64, 32 whose
// operands fit in 227 KB; 0 if none does or r > 3.
inline int tc_wide3_nrows(int shape, int r)
{
    if (r < 1 || r > 3) return 0;
    for (int nr : {128, 64, 32})
        if (tc_wide3_geom(r, tc_wide3_lines(shape, r), nr).smem <= 227 * 1024) return nr;
    return 0;
}

// ---------------------------------------------------------------------------
// 2:4-structured sparse form (paper Sec. 4.3), TF32 1:2 on mma.sp m16n8k16.
//
// The sparse operand must be A, so the Toeplitz block of line a is the A
// operand: A_a[m][k] = w^(t)[a][k - m] (0 <= k - m <= 2R) with M = 16 output
// columns and K = the 16 + 2R input columns of the window; B is the im2col
// of the input (K x 8 output rows).  TF32 sparsity keeps one element of every
// pair of consecutive logical K positions, so K is permuted ("strided
// swapping"): the window is cut into 16-byte chunks (4 columns) and chunk c is
// paired with a chunk at least ceil((2R+1)/4) chunks away, so no row's band
// holds both members of a pair.  Instruction s takes the chunk pairs 2s and
// 2s+1; its logical pair p is element p/2 of chunk pair 2s + (p mod 2).  A
// chunk index of -1 is a dummy (zero operand).
// ---------------------------------------------------------------------------
#ifdef __CUDACC__
#define GBS_HD __host__ __device__ __forceinline__
#else
#define GBS_HD inline
#endif

constexpr int kSpMaxNs = 4;  // instructions per line (R <= 12)

struct SpLayout {
    int R = 0, nc = 0, ns = 0, sigma = 0, pitch_q = 0, rl = 0;
    int cf[2 * kSpMaxNs], cs[2 * kSpMaxNs];  // chunk pairs (first, second); -1 = dummy
    int bchunk[4 * kSpMaxNs];                // chunk each lane class q of instruction s loads B from
                                             // (a dummy gets a filler chunk; its A is zero)
    std::vector<int> mask;                   // per line: bit s = instruction s issued
    double useful = 0, issued = 0;           // per output point (issued: logical K)
    double sparsity() const { return issued > 0 ? useful / issued : 0.0; }
};

// Round an FP32 value to TF32 (nearest, ties away from zero), as the
// conversion instruction does for finite values.
GBS_HD float tf32_round(float x)
{
    union {
        float f;
        unsigned u;
    } v;
    v.f = x;
    v.u = (v.u + 0x1000u) & 0xFFFFE000u;
    return v.f;
}

// Value and selector (0: first, 1: second member) of compressed A element
// (row m, logical pair p) of instruction s for line a.  w: the composite
// kernel, (2R+1) x (2R+1) row-major.
GBS_HD float sp_a_value(const double *w, int R, const int *cf, const int *cs, int a, int s, int m, int p,
                        int *sel)
{
    const int cp = 2 * s + (p & 1), i = p >> 1, lines = 2 * R + 1;
    const int fc = cf[cp], sc = cs[cp];
    *sel = 0;
    if (fc >= 0) {
        const int b = 4 * fc + i - m;
        if (b >= 0 && b <= 2 * R && w[a * lines + b] != 0.0) return tf32_round((float)w[a * lines + b]);
    }
    if (sc >= 0) {
        const int b = 4 * sc + i - m;
        if (b >= 0 && b <= 2 * R && w[a * lines + b] != 0.0) {
            *sel = 1;
            return tf32_round((float)w[a * lines + b]);
        }
    }
    return 0.0f;
}

inline SpLayout sp_layout_2d(int shape, int r, int t)
{
    SpLayout L;
    const int R = t * r;
    L.R = R;
    L.nc = (16 + 2 * R + 3) / 4;
    const int dc = (2 * R + 1 + 3) / 4;  // minimum chunk distance of a pair
    std::vector<int> pf, ps, used(L.nc, 0);
    for (int c = 0; c < L.nc; c++) {
        if (used[c]) continue;
        used[c] = 1;
        int partner = -1;
        for (int c2 = c + dc; c2 < L.nc; c2++)
            if (!used[c2]) {
                partner = c2;
                used[c2] = 1;
                break;
            }
        pf.push_back(c);
        ps.push_back(partner);
    }
    L.ns = ((int)pf.size() + 1) / 2;
    for (int i = 0; i < 2 * kSpMaxNs; i++) {
        L.cf[i] = i < (int)pf.size() ? pf[i] : -1;
        L.cs[i] = i < (int)ps.size() ? ps[i] : -1;
    }
    // B chunk of lane class q (0..3) of instruction s: first / second member
    // of chunk pair 2s + q/2.  Rows 8 apart XOR their 16-byte chunk index
    // with sigma; sigma and the filler chunks of dummies are chosen so that
    // the eight 16-byte loads of a quarter warp (two rows, four chunks) hit
    // eight distinct bank groups where possible.
    int best = 1 << 30;
    for (int sg = 0; sg < 8; sg++) {
        int total = 0, pick[4 * kSpMaxNs];
        for (int s = 0; s < L.ns; s++) {
            const int fixed[4] = {L.cf[2 * s], L.cs[2 * s], L.cf[2 * s + 1], L.cs[2 * s + 1]};
            int bestc = 1 << 30, choice[4] = {0, 0, 0, 0};
            // enumerate fillers for the dummy slots (nc <= 10 choices each)
            int slots[4], nd = 0;
            for (int j = 0; j < 4; j++)
                if (fixed[j] < 0) slots[nd++] = j;
            int combos = 1;
            for (int j = 0; j < nd; j++) combos *= L.nc;
            for (int cidx = 0; cidx < combos; cidx++) {
                int c[4], v = cidx;
                for (int j = 0; j < 4; j++) c[j] = fixed[j];
                for (int j = 0; j < nd; j++) {
                    c[slots[j]] = v % L.nc;
                    v /= L.nc;
                }
                int cnt[8] = {0};
                for (int j = 0; j < 4; j++) {
                    cnt[c[j] & 7]++;
                    cnt[(c[j] & 7) ^ sg]++;
                }
                int conf = 0;
                for (int b = 0; b < 8; b++) conf += cnt[b] > 1 ? cnt[b] - 1 : 0;
                if (conf < bestc) {
                    bestc = conf;
                    for (int j = 0; j < 4; j++) choice[j] = c[j];
                }
            }
            total += bestc;
            for (int j = 0; j < 4; j++) pick[4 * s + j] = choice[j];
        }
        if (total < best) {
            best = total;
            L.sigma = sg;
            for (int i = 0; i < 4 * L.ns; i++) L.bchunk[i] = pick[i];
        }
    }
    L.rl = 48 + 4 * L.nc;                 // staged row: 3 strips of 16 + the last window
    L.pitch_q = (L.rl / 4 + 7) / 8 * 8;  // 16-byte chunks per row, multiple of 8
    for (int a = -R; a <= R; a++) {
        const int h = composite_half(shape, r, t, a);
        int m = 0;
        if (h >= 0) {
            // non-zero columns of the line over the 16 rows: [R-h, R+h+15]
            for (int s = 0; s < L.ns; s++) {
                bool hit = false;
                for (int j = 0; j < 2; j++) {
                    const int cp = 2 * s + j;
                    for (int c : {L.cf[cp], L.cs[cp]}) {
                        if (c < 0) continue;
                        if (4 * c + 3 >= R - h && 4 * c <= R + h + 15) hit = true;
                    }
                }
                if (hit) m |= 1 << s;
            }
            L.useful += 2 * h + 1;
            L.issued += 16.0 * __builtin_popcount((unsigned)m);
        }
        L.mask.push_back(m);
    }
    return L;
}

}  // namespace gbs
