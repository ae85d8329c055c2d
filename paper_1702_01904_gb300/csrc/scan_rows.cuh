// scan_rows.cuh -- the PRISM scan of a raster whose rows each share one y position (k_rows_sum,
// k_rows_window), templated on the window sides; kernels_scan_rows*.cu instantiate it.
//
// The coefficients of Eq. PRISMfinal separate, alpha_mn(r0) = a_mn e^{-2 pi i q_n y0} e^{-2 pi i q_m x0},
// and the probes of a raster row share y0 and the window rows.  So the beams of one m are summed once
// per raster row, T_m(x, y) = sum_n a_mn e^{-2 pi i q_n y0} S_mn(x, y), for every column the row's
// windows reach, and each probe only sums its distinct m: 13 instead of 129 products per window
// pixel for the 20 mrad beams of a 50 A cell at f = 8.  With the beam set symmetric in m,
//   psi(x) = T_0 + sum_{m>0} cos(t_m) A_m + sin(t_m) B_m,   A_m = T_m + T_-m,  B_m = i (T_m - T_-m),
// t_m = -2 pi q_m x0: two real-by-complex products per pair (two packed FMAs).  The window's column
// transform commutes with the sum over m and with the choice of window columns (the window rows are
// the row's), so it is made on A_m and B_m once per raster row instead of once per probe:
//   k_rows_sum     per (4 raster rows, 16 columns (8 of 128-pixel windows), pair +-m): T, A, B, their column transforms, written
//                  to W[row][ky][plane][column] (planes T_0, A_1, B_1, A_2, ...).
//                  S comes beam by beam: the FP32 S-matrix itself, or what the windows reach of an FP16
//                  value + remainder S-matrix, unpacked once per scan (k_rows_unpack);
//   k_rows_window  per (raster row, Lp consecutive probes): psi on (x, ky), the row transforms, the
//                  intensities, folded over +-kx and +-ky (the annular bins depend on |kx|, |ky|)
//                  into shared memory, then the bins -- or the full pattern.
//
// Measured (40 000 probes of the 1024^2 carbon cell, 129 beams, 64-pixel windows): 5.03 ms with the
// blocks of scan_gemm.cuh, 1.51 ms here (k_rows_sum 0.61, k_rows_window 0.84); 32 x 32 probes of the
// 2048^2 cell (529 beams, 128-pixel windows) 2.70 -> 0.73 ms; 16 x 16 probes of a 256^2 cell 68 -> 25 us.
// 33 x 31 probes of a 512^2 cell from value + remainder storage (213 beams): 382 us on the tensor cores,
// 110 us here, nearer to 64 bits (2.3e-6 against 4.9e-6 off).
// Bound: k_rows_sum by the load/store pipe (57 % busy) and its loads' latency at 16 warps per SM (its S reads hit
// the L2, 1.9 GB of them), k_rows_window by the same pipe (61 %) and dependent latency (issue slots 49 %);
// leaving out the products saves 32 % of its time, the loads of the planes 20 %, the transforms 12 %,
// the bins 8 %, the folding 5 %.
// Against 64 bits from the same S (10 grids, windows of 16 to 128 pixels, 13 to 529 beams): 3 wide bins 0.28 to
// 1.02 of the block scan's error, 100 bins of 1 mrad 0.80 to 1.13 of it (0.97 on average; 0.7 to 1.0e-7, a tenth
// of what the S-matrix carries).  Neither the phase of a coefficient, rounded once per factor, nor the folding
// is what differs: taking the remainder of the phases along, or folding with the products, moved nothing.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

#include "fft.cuh"
#include "launch.cuh"
#include "params.h"
#include "scan_common.cuh"

namespace prism {

// raster rows per k_rows_sum unit: each S value loaded feeds four sums (6 or 8 rows cost the registers and
// shared memory of the third CTA per SM: 40 000 probes 1.50 ms with 4, 1.50 to 1.60 with 6, 1.70 with 8)
constexpr int ROWS_R = 4;

// ------------------------------------------------------------------ sums over n, column transforms
// SMALL: for scans of few units, where a unit's latency counts and not the units an SM holds: more threads
// (fewer sweeps over the rows) and more loads together
template <int NWY, bool SMALL = false>
struct RowsSumCfg {
    using FS = FftShape<NWY>;
    // 128-pixel windows: the columns' buffers (79 KB) leave two CTAs on an SM anyway, so they take more threads and
    // loads in flight (529 beams, 32 x 32 probes, whole scan: 762 us with 192 threads and 7 loads, 765 with 288
    // and 7, 731 with 192 and 14, 717 with 288 and 9, 714 so)
    static constexpr bool WIDE = NWY >= 128;
    static constexpr int BLOCK = SMALL || WIDE ? 256 : 192;
    static constexpr int MINB = SMALL ? 1 : WIDE ? 2 : 3;
    static constexpr int XC = WIDE ? 8 : 16;             // columns per unit: 64- or 128-byte runs of S and of W
    static constexpr int PAIRS = XC / 2;                 // a thread takes two neighbouring columns
    static constexpr int YSTEP = BLOCK / PAIRS;          // union rows per sweep of the block
    // beams whose loads a thread issues together (of one m; the last batch of a sum may be short: 529 beams have up
    // to 27 of one m, 129 up to 13, 49 up to 9)
    static constexpr int U = SMALL ? 14 : WIDE ? 13 : 7;
    // A column of one plane and raster row: NWY values, in place the transform's exchange.  The second
    // column of a pair starts 16 banks on (mod 32), so the columns two slots of a half-warp transform
    // fall on different banks; pairs are 4 banks apart (8 for the 4 pairs of 8 columns), so that the
    // half-warp's pairs and neighbouring rows written by the sums do too.
    static constexpr int LEN = FS::N1 * (FS::N2 + 1);
    static_assert(LEN >= NWY, "the exchange holds a column");
    static constexpr int up(int n, int rem) { return (n + 15 - rem) / 16 * 16 + rem; }  // smallest >= n, rem (mod 16)
    static constexpr int SECOND = up(LEN, 8);
    static constexpr int PAIR = up(SECOND + LEN, PAIRS == 8 ? 2 : 4);
    static constexpr int ROW = PAIRS * PAIR;             // float2 of one plane and raster row
    static constexpr size_t BUF = (size_t)2 * ROWS_R * ROW * sizeof(float2);
    __device__ static int at(int c) { return (c >> 1) * PAIR + (c & 1) * SECOND; }
    __host__ __device__ static constexpr size_t smem(int max_beams) {  // beams of one m at most
        return BUF + (size_t)2 * max_beams * (ROWS_R * sizeof(float2) + sizeof(int));
    }
};

template <int NWY, bool SMALL = false>
__global__ void __launch_bounds__(RowsSumCfg<NWY, SMALL>::BLOCK, RowsSumCfg<NWY, SMALL>::MINB) k_rows_sum(const __grid_constant__ ScanArgs a) {
    using C = RowsSumCfg<NWY, SMALL>;
    using FS = FftShape<NWY>;
    using Fwd = FwdFft<NWY>;
    constexpr int BLOCK = C::BLOCK, R = ROWS_R, XC = C::XC, T = FS::T, E = FS::E;
    extern __shared__ __align__(16) unsigned char sm_rows[];
    float2 *buf = reinterpret_cast<float2 *>(sm_rows);                        // [plane][row][column]
    float2 *coef = reinterpret_cast<float2 *>(sm_rows + C::BUF);              // [beam][row]
    const int tid = threadIdx.x, j = blockIdx.y;
    const int row0 = blockIdx.z * R;  // of this launch
    const int M = a.rows_m;
    // beams of +j, then of -j (none when j = 0)
    const int pb = __ldg(a.m_off + M + j), np = __ldg(a.m_off + M + j + 1) - pb;
    const int mb = __ldg(a.m_off + M - j), nm = j ? __ldg(a.m_off + M - j + 1) - mb : 0;
    int *beam = reinterpret_cast<int *>(coef + (np + nm) * R);
    __shared__ int wy0[R];   // window row origins relative to the first union row (out of reach: no such row)
    __shared__ int geo[2];   // first union row, union rows
    next_may_start();
    for (int i = tid; i < np + nm; i += BLOCK) beam[i] = __ldg(a.m_beam + (i < np ? pb + i : mb + i - np));
    for (int i = tid; i < (np + nm) * R; i += BLOCK) {
        const int k = i / R, r = i - k * R;
        const int b = __ldg(a.m_beam + (k < np ? pb + k : mb + k - np));
        float2 v = make_float2(0.f, 0.f);
        if (row0 + r < a.rows_n) {
            double c = a.qy[b] * (a.y0[(size_t)(a.rows_0 + row0 + r) * a.scan_px] - a.shift_y);
            c -= rint(c);
            float sn, cs;
            sincospif(-2.0f * (float)c, &sn, &cs);
            v = cmul(__ldg(a.base + b), make_float2(cs, sn));
        }
        coef[i] = v;
    }
    if (tid < 32) {
        const bool valid = tid < R && row0 + tid < a.rows_n;
        int sy = 0;
        if (valid) sy = ((int)floor(a.y0[(size_t)(a.rows_0 + row0 + tid) * a.scan_px] / a.py_s + 0.5) - NWY / 2) & (a.ny_s - 1);
        const int sy0 = __shfl_sync(0xffffffffu, sy, 0);
        const int dy = valid ? ((sy - sy0 + a.ny_s / 2) & (a.ny_s - 1)) - a.ny_s / 2 : 0;
        const int lo = __reduce_min_sync(0xffffffffu, dy), hi = __reduce_max_sync(0xffffffffu, dy);
        if (tid < R) wy0[tid] = valid ? dy - lo : 1 << 28;
        if (tid == 0) {
            geo[0] = (sy0 + lo) & (a.ny_s - 1);
            geo[1] = hi - lo + NWY;
        }
    }
    __syncthreads();
    after_previous();
    const int ytop = geo[0], yn = geo[1];
    const int col = 2 * (tid % C::PAIRS);
    // even: the pair is one aligned load
    const int x = (a.rows_g0 + blockIdx.x * XC + col - a.rows_x0) & (a.nx_s - 1);
    const size_t npix = (size_t)a.rows_ry * a.rows_pitch;
    for (int yv = tid / C::PAIRS; yv < yn; yv += C::YSTEP) {
        bool any = false;
#pragma unroll
        for (int r = 0; r < R; ++r) any = any || (unsigned)(yv - wy0[r]) < (unsigned)NWY;
        if (!any) continue;  // between the windows of rows far apart
        const float2 *sp = a.rows_src + (size_t)((ytop + yv - a.rows_y0) & (a.ny_s - 1)) * a.rows_pitch + x;
#pragma unroll 1
        for (int sg = 0; sg < 2; ++sg) {
            // T = sum_b Re S_b c_b + i sum_b Im S_b c_b, both as packed FMAs, combined at the end (the
            // coefficients of two rows come in one 16-byte load)
            float2 re[R][2], im[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) re[r][h] = im[r][h] = make_float2(0.f, 0.f);
            const int b0 = sg ? np : 0, b1 = sg ? np + nm : np;
            for (int bb = b0; bb < b1; bb += C::U) {
                float4 s[C::U];
#pragma unroll
                for (int i = 0; i < C::U; ++i)
                    if (bb + i < b1) s[i] = __ldg(reinterpret_cast<const float4 *>(sp + (size_t)beam[bb + i] * npix));
#pragma unroll
                for (int i = 0; i < C::U; ++i) {
                    if (bb + i >= b1) break;
                    const float2 x0 = make_float2(s[i].x, s[i].x), y0 = make_float2(s[i].y, s[i].y);
                    const float2 x1 = make_float2(s[i].z, s[i].z), y1 = make_float2(s[i].w, s[i].w);
                    const float4 *cp = reinterpret_cast<const float4 *>(coef + (bb + i) * R);
#pragma unroll
                    for (int r = 0; r < R; r += 2) {
                        const float4 c2 = cp[r / 2];
                        const float2 c[2] = {make_float2(c2.x, c2.y), make_float2(c2.z, c2.w)};
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            re[r + q][0] = __ffma2_rn(x0, c[q], re[r + q][0]);
                            im[r + q][0] = __ffma2_rn(y0, c[q], im[r + q][0]);
                            re[r + q][1] = __ffma2_rn(x1, c[q], re[r + q][1]);
                            im[r + q][1] = __ffma2_rn(y1, c[q], im[r + q][1]);
                        }
                    }
                }
            }
            // T_j goes to the columns of plane A and is read back by this thread for A and B
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int w = yv - wy0[r];
                if ((unsigned)w < (unsigned)NWY) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float2 *b = buf + r * C::ROW + C::at(col + h) + w;
                        const float2 v = make_float2(re[r][h].x - im[r][h].y, re[r][h].y + im[r][h].x);
                        if (sg == 0) {
                            *b = v;
                        } else {
                            const float2 plus = *b, d = csub(plus, v);
                            *b = cadd(plus, v);
                            b[R * C::ROW] = make_float2(-d.y, d.x);
                        }
                    }
                }
            }
            if (j == 0) break;
        }
    }
    __syncthreads();
    // column transforms, T lanes of one warp each (rows past the raster's end hold no values; they are
    // transformed with their neighbours and not stored)
    const int t = tid % T;
    const int planes = j ? 2 : 1, plane0 = j ? 2 * j - 1 : 0, nplanes = 2 * M + 1;
    for (int f = tid / T; f < planes * R * XC; f += BLOCK / T) {
        const int pl = f / (R * XC), r = (f / XC) % R, c = f % XC;
        float2 *b = buf + (pl * R + r) * C::ROW + C::at(c);
        WarpExchange<FS::N1, FS::N2, T> ex{b};
        float2 v[E];
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = b[Fwd::in_elem(e, t)];
        Fwd::template run<decltype(ex), TW_GLOBAL>(v, t, a.tw_fwd_y, a.tw, ex);
        if (row0 + r < a.rows_n) {
            float2 *w = a.rows_w + ((size_t)(row0 + r) * NWY * nplanes + plane0 + pl) * a.rows_cols + blockIdx.x * XC + c;
#pragma unroll
            for (int e = 0; e < E; ++e) w[(size_t)Fwd::out_elem(e, t) * nplanes * a.rows_cols] = v[e];
        }
    }
}

// ------------------------------------------------------------------ windows
// A warp owns the row pairs +-ky = warp, warp + 8, ...: its lanes hold the planes of 32 neighbouring
// columns of both rows in registers and sum every probe whose window reaches them into the warp's
// window rows in shared memory; then T lanes transform a probe's row.  No block barrier until the bins.
// Pairs of m are taken KP at a time (the planes held in registers).
template <int NWX, int NWY>
struct RowsWinCfg {
    using FS = FftShape<NWX>;
    // 16 warps on an SM: two CTAs of 8, or one of 16 where the windows are too large to be held by two
    static constexpr int WARPS = NWX * NWY >= 128 * 128 ? 16 : 8, BLOCK = 32 * WARPS;
    static constexpr int CTAS = 16 / WARPS;
    static constexpr int PITCH = FS::N1 * (FS::N2 + 1);  // a window row, in place the transform's exchange
    static constexpr int SLOTS = 32 / FS::T;             // window rows a warp transforms at once
    static constexpr int FX = NWX / 2 + 1, FY = NWY / 2 + 1;
    __host__ __device__ static constexpr int padded(int lp) { return (lp + SLOTS - 1) / SLOTS * SLOTS; }
    // the coefficients, the warps' window rows, the folded intensities, and the bins' lists (16-bit)
    __host__ __device__ static constexpr size_t smem(int lp, int mp, int lists) {
        return (size_t)lp * mp * sizeof(float4) + (size_t)2 * WARPS * padded(lp) * PITCH * sizeof(float2) +
               (((size_t)lp * FX * FY * sizeof(float) + 15) & ~(size_t)15) + (size_t)lists * sizeof(uint16_t);
    }
};

// pairs of m rounded up to whole chunks of KP (at least one: T_0 rides in the first)
template <int KP>
__host__ __device__ constexpr int rows_padded(int m) { return m < 1 ? KP : (m + KP - 1) / KP * KP; }

template <int NWX, int NWY, int KP>
__global__ void __launch_bounds__(RowsWinCfg<NWX, NWY>::BLOCK, RowsWinCfg<NWX, NWY>::CTAS) k_rows_window(const __grid_constant__ ScanArgs a) {
    using C = RowsWinCfg<NWX, NWY>;
    using FS = FftShape<NWX>;
    using Fwd = FwdFft<NWX>;
    constexpr int BLOCK = C::BLOCK, PITCH = C::PITCH, T = FS::T, E = FS::E, SLOTS = C::SLOTS, FX = C::FX, FY = C::FY;
    extern __shared__ __align__(16) unsigned char sm_rows[];
    __shared__ int dxs[32];  // window column origins relative to the group's first column
    __shared__ int geo[2];   // first column, columns
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int M = a.rows_m, LP = a.rows_lp, npl = 2 * M + 1;
    const int MP = rows_padded<KP>(M);  // coefficients per probe, zero past M
    const int ngc = (a.scan_px + LP - 1) / LP;
    // row of this launch (the last first: its sums are still in the L2), first probe in it
    const int rb = blockIdx.x / ngc, row = a.rows_n - 1 - rb, p0 = (blockIdx.x - rb * ngc) * LP;
    const int np = min(LP, a.scan_px - p0);
    const int pr0 = (a.rows_0 + row) * a.scan_px + p0;
    float4 *cs = reinterpret_cast<float4 *>(sm_rows);                    // [LP][MP] (cos, cos, sin, sin)
    float2 *win = reinterpret_cast<float2 *>(cs + LP * MP) + (size_t)warp * 2 * C::padded(LP) * PITCH;  // [2][probe][PITCH]
    const int row1 = C::padded(LP) * PITCH;  // to the second row of a pair
    float *fold = reinterpret_cast<float *>(reinterpret_cast<float2 *>(cs + LP * MP) + (size_t)C::WARPS * 2 * C::padded(LP) * PITCH);  // [LP][FY][FX]
    next_may_start();
    // the bins' offsets and lists, read after the windows
    uint16_t *lists = reinterpret_cast<uint16_t *>(fold + ((LP * FX * FY + 3) & ~3));
    for (int i = tid; i < a.n_fold16 / 8; i += BLOCK) cp_async16(lists + 8 * i, a.fold16 + 8 * i);
    cp_async_commit();
    for (int i = tid; i < np * MP; i += BLOCK) {
        const int p = i / MP, j = i - p * MP + 1;
        if (j > M) {
            cs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        double c = a.m_qx[j] * (a.x0[pr0 + p] - a.shift_x);
        c -= rint(c);
        float sn, co;
        sincospif(-2.0f * (float)c, &sn, &co);
        cs[i] = make_float4(co, co, sn, sn);
    }
    if (warp == 0) {
        const bool valid = lane < np;
        int sx = 0;
        if (valid) sx = ((int)floor(a.x0[pr0 + lane] / a.px_s + 0.5) - NWX / 2) & (a.nx_s - 1);
        const int sx0 = __shfl_sync(0xffffffffu, sx, 0);
        const int dx = valid ? ((sx - sx0 + a.nx_s / 2) & (a.nx_s - 1)) - a.nx_s / 2 : 0;
        const int lo = __reduce_min_sync(0xffffffffu, dx), hi = __reduce_max_sync(0xffffffffu, dx);
        dxs[lane] = dx - lo;
        if (lane == 0) {
            geo[0] = (sx0 + lo) & (a.nx_s - 1);
            geo[1] = hi - lo + NWX;
        }
    }
    __syncthreads();
    after_previous();
    const int xf = geo[0], vc = geo[1];
    const size_t rstride = (size_t)npl * a.rows_cols;  // W: one ky
    const float2 *wrow = a.rows_w + (size_t)row * NWY * rstride;
    // The warp's steps, in order: the row pairs ky = jy and its mirror (jy = 0: the two rows that are
    // their own mirror, 0 and NWY/2), jy = warp, warp + 8, ...; of each the chunks of KP pairs of m; of
    // each the chunks of 32 columns.  Both rows of a pair share the coefficients read.  The planes of a
    // pair's first step load before the transforms of the pair before.
    auto load = [&](float2 (&t0)[2 * KP + 1], float2 (&t1)[2 * KP + 1], int jy, int mc, int v0) {
        const int v = min(v0 + lane, vc - 1);
        // (columns between far-apart windows may not be held: any held one serves, no window reads it)
        const int c = min((((xf + v) & (a.nx_s - 1)) - a.rows_g0) & (a.nx_s - 1), a.rows_cols - 1);
        const float2 *w0 = wrow + (size_t)jy * rstride + (size_t)(2 * mc) * a.rows_cols + c;
        const float2 *w1 = w0 + (size_t)(jy ? NWY - 2 * jy : NWY / 2) * rstride;
        const int left = npl - 2 * mc;  // planes from the chunk's first on (T_0, or the last of the chunk before)
#pragma unroll
        for (int k = 0; k <= 2 * KP; ++k) {
            t0[k] = t1[k] = make_float2(0.f, 0.f);
            if (k < left) {
                t0[k] = __ldcg(w0 + (size_t)k * a.rows_cols);
                t1[k] = __ldcg(w1 + (size_t)k * a.rows_cols);
            }
        }
    };
    const int slot = lane / T, t = lane % T;
    static_assert(Fwd::out_elem(1, 0) == T && Fwd::out_elem(E - 1, T - 1) == NWX - 1, "kx = t + T e");
    int jy = warp, mc = 0, v0 = 0;
    float2 t0[2 * KP + 1], t1[2 * KP + 1];
    if (jy < NWY / 2) load(t0, t1, jy, 0, 0);
#pragma unroll 1
    while (jy < NWY / 2) {
        for (int p = 0; p < np; ++p) {
            const int d = dxs[p];
            if (v0 + 31 < d || v0 >= d + NWX) continue;
            const int u = v0 + lane - d;
            const bool in = (unsigned)u < (unsigned)NWX;
            float2 *wp = win + p * PITCH + u;
            float2 s0 = t0[0], s1 = t1[0];
            if (mc > 0 && in) {
                s0 = wp[0];
                s1 = wp[row1];
            }
            const float4 *cp = cs + p * MP + mc;
#pragma unroll
            for (int k = 0; k < KP; ++k) {
                const float4 q = cp[k];
                const float2 co = make_float2(q.x, q.y), sn = make_float2(q.z, q.w);
                s0 = __ffma2_rn(t0[2 * k + 1], co, s0);
                s1 = __ffma2_rn(t1[2 * k + 1], co, s1);
                s0 = __ffma2_rn(t0[2 * k + 2], sn, s0);
                s1 = __ffma2_rn(t1[2 * k + 2], sn, s1);
            }
            if (in) {
                wp[0] = s0;
                wp[row1] = s1;
            }
        }
        const int jc = jy;
        v0 += 32;
        if (v0 >= vc) {
            v0 = 0;
            mc += KP;
            if (mc >= MP) {
                mc = 0;
                jy += C::WARPS;
            }
        }
        if (jy < NWY / 2) load(t0, t1, jy, mc, v0);
        if (jy == jc) continue;  // more of this pair of rows
        __syncwarp();
        // row transforms, T lanes per probe (register e of lane t is kx = t + T e), the intensities and
        // their sum over +-kx: kx < NWX/2 in the registers e < E/2, its mirror NWX - kx in register E-1-e
        // of lane T-t (lane 0: its own register E-e); kx = NWX/2 on lane 0
#pragma unroll 1
        for (int i = 0; i < 2 * np; i += 2 * SLOTS) {
            const int p = i / 2 + slot;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int ky = h == 0 ? jc : jc ? NWY - jc : NWY / 2;
                float2 *b = win + p * PITCH + (h ? row1 : 0);
                WarpExchange<FS::N1, FS::N2, T> ex{b};
                float2 z[E];
#pragma unroll
                for (int e = 0; e < E; ++e) z[e] = b[Fwd::in_elem(e, t)];
                Fwd::template run<decltype(ex), TW_GLOBAL>(z, t, a.tw_fwd, a.tw, ex);
                float inten[E];
#pragma unroll
                for (int e = 0; e < E; ++e) inten[e] = fmaf(z[e].x, z[e].x, z[e].y * z[e].y);
                if (a.cbed) {
                    if (p < np) {
                        float *o = a.cbed + ((size_t)(pr0 + p) * NWY + ky) * NWX + t;
                        const float fnorm = (float)a.inv_norm;
#pragma unroll
                        for (int e = 0; e < E; ++e) o[T * e] = inten[e] * fnorm;
                    }
                } else {
                    float *fo = fold + ((size_t)p * FY + (ky <= NWY / 2 ? ky : NWY - ky)) * FX + t;
                    const bool add = h == 1 && jc != 0;  // onto the mirror's row, from the same lanes
#pragma unroll
                    for (int e = 0; e < E / 2; ++e) {
                        const float m = __shfl_sync(0xffffffffu, inten[E - 1 - e], (T - t) & (T - 1), T);
                        const float f = t ? inten[e] + m : e ? inten[e] + inten[E - e] : inten[0];
                        if (p < np) fo[T * e] = add ? fo[T * e] + f : f;
                    }
                    if (p < np && t == 0) fo[NWX / 2] = add ? fo[NWX / 2] + inten[E / 2] : inten[E / 2];
                }
            }
        }
        __syncwarp();
    }
    if (!a.out) return;
    cp_async_wait<0>();
    __syncthreads();
    // annular bins as in window_epilogue, over the folded quadrant: four interleaved FP32 partial sums of
    // a bin's entries, added and scaled in FP64
    const int nb = a.nbins;
    for (int i = tid; i < np * nb; i += BLOCK) {
        const int p = i / nb, k = i - p * nb;
        const float *fo = fold + (size_t)p * FY * FX;
        const int e = lists[k + 1] - lists[k];
        const uint16_t *ix = lists + nb + 1 + lists[k];
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        int q = 0;
        for (; q + 4 <= e; q += 4) {
            s0 += fo[ix[q]];
            s1 += fo[ix[q + 1]];
            s2 += fo[ix[q + 2]];
            s3 += fo[ix[q + 3]];
        }
        for (; q < e; ++q) s0 += fo[ix[q]];
        const float val = (float)((((double)s0 + (double)s1) + ((double)s2 + (double)s3)) * a.inv_norm);
        float *o = a.out + (size_t)(pr0 + p) * nb + k;
        *o = a.accumulate ? *o + a.acc_w * val : val;
    }
}

// ------------------------------------------------------------------ launches
// pairs of m a lane holds at once: all of them up to 8, else chunks of 6, 7 or 8, the fewest chunks with the
// fewest pairs left empty
static inline int rows_kp(int m) {
    if (m <= 4) return 4;
    const int chunks = (m + 7) / 8, kp = (m + chunks - 1) / chunks;
    return kp < 6 ? 6 : kp;
}
static inline int rows_mp(int m) {
    const int kp = rows_kp(m);
    return m < 1 ? kp : (m + kp - 1) / kp * kp;
}

// probes per k_rows_window CTA: as many as leave 16 warps on an SM, fewer where that takes no longer
// (0: the scan does not fit).  A CTA's time goes about as its probes and a part (reading the planes and
// lists) worth some 3; the CTAs run in rounds of 152 SMs.
template <int NWX, int NWY>
static int rows_lp(int m, int max_beams, int lists, int px, int rows) {
    using C = RowsWinCfg<NWX, NWY>;
    const int mp = rows_mp(m);
    if (C::smem(1, mp, lists) > 226 * 1024 || RowsSumCfg<NWY>::smem(max_beams) > 226 * 1024) return 0;
    int best = 1;
    double best_t = 1e300;
    for (int l = 1; l <= 32 && (l == 1 || C::smem(l, mp, lists) <= 226 * 1024 / C::CTAS - 1024); ++l) {
        const long long ctas = (long long)rows * ((px + l - 1) / l), slots = 152 * C::CTAS;
        const double t = (double)((ctas + slots - 1) / slots) * (l + 3);
        if (t <= best_t) {
            best_t = t;
            best = l;
        }
    }
    return best;
}

template <int NWX, int NWY>
static cudaError_t rows_launch(const ScanArgs &args, cudaStream_t s) {
    using A = RowsSumCfg<NWY>;
    using B = RowsWinCfg<NWX, NWY>;
    ScanArgs a = args;
    if (reinterpret_cast<uintptr_t>(a.rows_src) & 15) return cudaErrorMisalignedAddress;  // pixel pairs are read as one load
    const int kp = rows_kp(a.rows_m);
    const size_t sa = A::smem(a.rows_maxn), sb = B::smem(a.rows_lp, rows_mp(a.rows_m), a.n_fold16);
    // (few units: a chunk of rows makes no more than 2 per SM)
    const bool small = (long long)(a.rows_cols / A::XC) * (a.rows_m + 1) * ((std::min(a.rows_chunk, a.scan_py) + ROWS_R - 1) / ROWS_R) <= 2 * 152;
    void (*sum)(const ScanArgs) = small ? k_rows_sum<NWY, true> : k_rows_sum<NWY>;
    const int sum_block = small ? RowsSumCfg<NWY, true>::BLOCK : A::BLOCK;
    static_assert(RowsSumCfg<NWY, true>::XC == A::XC && RowsSumCfg<NWY, true>::BUF == A::BUF, "the same unit");
    void (*win)(const ScanArgs) = kp == 4   ? k_rows_window<NWX, NWY, 4>
                                  : kp == 6 ? k_rows_window<NWX, NWY, 6>
                                  : kp == 7 ? k_rows_window<NWX, NWY, 7>
                                            : k_rows_window<NWX, NWY, 8>;
    cudaError_t e = cudaSuccess;
    if (!a.attrs_set && ((e = allow_max_dynamic_smem(k_rows_sum<NWY>)) != cudaSuccess ||
                         (e = allow_max_dynamic_smem(k_rows_sum<NWY, true>)) != cudaSuccess || (e = allow_max_dynamic_smem(win)) != cudaSuccess))
        return e;
    const int ngc = (a.scan_px + a.rows_lp - 1) / a.rows_lp;
    for (int r0 = 0; r0 < a.scan_py; r0 += a.rows_chunk) {
        a.rows_0 = r0;
        a.rows_n = std::min(a.rows_chunk, a.scan_py - r0);
        const dim3 ga(a.rows_cols / A::XC, a.rows_m + 1, (a.rows_n + ROWS_R - 1) / ROWS_R);
        // the first launch is a plain one: the positions and coefficients that both kernels read before
        // they wait (in their prologues) come from the launch or copies before it
        if (r0 == 0) {
            sum<<<ga, sum_block, sa, s>>>(a);
            e = cudaGetLastError();
        } else {
            e = launch_chained(sum, ga, sum_block, sa, s, a);
        }
        if (e != cudaSuccess) return e;
        if ((e = launch_chained(win, a.rows_n * ngc, B::BLOCK, sb, s, a)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace prism
