// scan_list.cuh -- the FP32 PRISM scan of positions too far apart to share S values (k_scan_list): scattered
// position lists, sparse rasters.  One CTA per probe: a thread owns a few window pixels and walks the beams,
// several beams' loads in flight; the window then goes through shared memory for its transform and bins.
//
// Bound by the S values read, B nw^2 8 bytes per probe once from the L2 (900 scattered probes of 129 beams
// and 64-pixel windows: 3.8 GB in 0.33 ms).  The blocks of scan_gemm.cuh run such probes one after another
// with one warp in eight at work, and a list of positions fills 4 of their 32 slots: 1.32 ms for those 900,
// 0.32 for 10 of them (29 us here).  900 jittered positions of 32 x 16 windows and 25 beams: 69 -> 20 us on
// the device.
// Few probes: a cluster of up to 8 CTAs shares a probe's beams, and their windows are added in the first
// one's shared memory, rank by rank.  Bins of short lists (up to 1024-pixel windows) take a thread each
// (4000 probes of 16 x 16 windows: 162 us with a warp each, 89 so).
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "fft.cuh"
#include "params.h"
#include "scan_common.cuh"

namespace prism {

template <int NWX, int NWY>
struct ListCfg {
    static constexpr int NP = NWX * NWY;
    static constexpr int BLOCK = NP <= 1024 ? 128 : NP <= 4096 ? 256 : 512;
    static constexpr int PIX = NP / BLOCK;                    // window pixels per thread
    // a batch of loads: U beams' values of a thread's pixels, or, of 32 pixels, a quarter of one beam's (the
    // batch after the one being summed is in flight)
    static constexpr int U = PIX >= 16 ? 1 : 16 / PIX;
    static constexpr int PB = PIX > 16 ? 8 : PIX;             // pixels of a batch
    static constexpr int NB = PIX / PB;                       // batches per U beams
    static constexpr int PW = NWX + 4;                        // window row pitch (bank spread)
    static constexpr int EX = ExSize<NWX, NWY, BLOCK>::value;
    static constexpr size_t FIXED = (size_t)(NWY * PW + EX + NWX + NWY) * sizeof(float2);
    static_assert(BLOCK % NWX == 0 || NWX % BLOCK == 0, "a thread's pixels lie in one column");
};

template <int NWX, int NWY>
__global__ void __launch_bounds__(ListCfg<NWX, NWY>::BLOCK) k_scan_list(const __grid_constant__ ScanArgs a) {
    using C = ListCfg<NWX, NWY>;
    constexpr int BLOCK = C::BLOCK, PIX = C::PIX, U = C::U, PW = C::PW, RS = BLOCK / NWX;  // rows between a thread's pixels
    extern __shared__ __align__(16) float2 sm_list[];
    float2 *win = sm_list;              // [NWY][PW]
    float2 *ex = win + NWY * PW;
    float2 *twx = ex + C::EX, *twy = twx + NWX;
    float2 *alpha = twy + NWY;          // [n_beams]
    const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int cr = (int)cl.block_rank(), cn = (int)cl.num_blocks();
    const int tid = threadIdx.x, p = blockIdx.x / cn;
    const int bb = cr * a.n_beams / cn, be = (cr + 1) * a.n_beams / cn;  // this CTA's beams
    for (int i = tid; i < NWX; i += BLOCK) twx[i] = a.tw_fwd[i];
    for (int i = tid; i < NWY; i += BLOCK) twy[i] = a.tw_fwd_y[i];
    const double x0 = a.x0[p], y0 = a.y0[p];
    for (int b = bb + tid; b < be; b += BLOCK) {
        double c = a.qx[b] * (x0 - a.shift_x) + a.qy[b] * (y0 - a.shift_y);
        c -= rint(c);
        float s, co;
        sincospif(-2.0f * (float)c, &s, &co);
        alpha[b] = cmul(__ldg(a.base + b), make_float2(co, s));
    }
    const int sx = ((int)floor(x0 / a.px_s + 0.5) - NWX / 2) & (a.nx_s - 1);
    const int sy = ((int)floor(y0 / a.py_s + 0.5) - NWY / 2) & (a.ny_s - 1);
    const int wx = tid % NWX, wy = tid / NWX;  // this thread's pixels: column wx, rows wy + RS k
    const float2 *Sx = a.S + ((sx + wx) & (a.nx_s - 1));
    const size_t bstride = (size_t)a.ny_s * a.nx_s;
    // Up to 8 pixels: the two sums of scan_gemm.cuh, sum_b S_b Re alpha_b and sum_b S_b Im alpha_b, advanced
    // by one packed FMA each: the same windows bit by bit.  More: the registers hold one sum, rounded twice per
    // beam by its two FMAs, so every 16 beams it goes to the window in shared memory (400 probes of 213 beams,
    // bins against 64 bits: 1.2e-7 off in one chain, 0.95e-7 by two sums, 0.80e-7 so; 0.46 -> 0.48 ms for 900.
    // Two sums with half the loads in flight: 0.63 ms)
    constexpr bool TWO = PIX <= 8;
    constexpr int RUN = 16;
    float2 acc[PIX], aci[TWO ? PIX : 1];
#pragma unroll
    for (int k = 0; k < PIX; ++k) acc[k] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < (TWO ? PIX : 1); ++k) aci[k] = make_float2(0.f, 0.f);
    auto out = [&](int k) -> float2 & { return win[(wy + RS * k) * PW + wx]; };
    __syncthreads();
    constexpr int PB = C::PB, NB = C::NB;
    auto load = [&](float2 (&s)[U][PB], int b0, int h) {  // batch h of beams b0 ... b0 + U - 1
#pragma unroll
        for (int i = 0; i < U; ++i)
            if (b0 + i < be) {
                const float2 *Sb = Sx + (size_t)(b0 + i) * bstride;
#pragma unroll
                for (int k = 0; k < PB; ++k) s[i][k] = __ldg(Sb + (size_t)((sy + wy + RS * (h * PB + k)) & (a.ny_s - 1)) * a.nx_s);
            }
    };
    float2 cur[U][PB], nxt[U][PB];
    load(cur, bb, 0);
#pragma unroll 1
    for (int b0 = bb; b0 < be; b0 += U) {
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            if (h + 1 < NB) load(nxt, b0, h + 1);
            else load(nxt, b0 + U, 0);
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (b0 + i < be) {
                    const float2 al = alpha[b0 + i];
#pragma unroll
                    for (int k = 0; k < PB; ++k) {
                        const float2 s = cur[i][k];
                        if constexpr (TWO) {
                            acc[h * PB + k] = __ffma2_rn(s, make_float2(al.x, al.x), acc[h * PB + k]);
                            aci[h * PB + k] = __ffma2_rn(s, make_float2(al.y, al.y), aci[h * PB + k]);
                        } else {
                            float2 &c = acc[h * PB + k];
                            c.x = fmaf(al.x, s.x, fmaf(-al.y, s.y, c.x));
                            c.y = fmaf(al.x, s.y, fmaf(al.y, s.x, c.y));
                        }
                    }
                }
#pragma unroll
            for (int i = 0; i < U; ++i)
#pragma unroll
                for (int k = 0; k < PB; ++k) cur[i][k] = nxt[i][k];
        }
        if constexpr (!TWO) {
            static_assert(TWO || U == 1, "a beam per step");
            const int done = b0 - bb + 1;
            if (done % RUN == 0 || b0 + 1 == be) {
#pragma unroll
                for (int k = 0; k < PIX; ++k) {
                    out(k) = done <= RUN ? acc[k] : cadd(out(k), acc[k]);
                    acc[k] = make_float2(0.f, 0.f);
                }
            }
        }
    }
    if (TWO || bb == be) {
#pragma unroll
        for (int k = 0; k < PIX; ++k) out(k) = TWO ? make_float2(acc[k].x - aci[TWO ? k : 0].y, acc[k].y + aci[TWO ? k : 0].x) : acc[k];
    }
    if (cn > 1) {
        // every rank's window is written; the first adds the others' to its own, then they may leave
        cl.sync();
        if (cr == 0) {
#pragma unroll
            for (int k = 0; k < PIX; ++k) acc[k] = out(k);
            for (int r = 1; r < cn; ++r) {
                const float2 *o = cl.map_shared_rank(win, r);
#pragma unroll
                for (int k = 0; k < PIX; ++k) acc[k] = cadd(acc[k], o[(wy + RS * k) * PW + wx]);
            }
#pragma unroll
            for (int k = 0; k < PIX; ++k) out(k) = acc[k];
        }
        cl.sync();
        if (cr != 0) return;
    }
    __syncthreads();
    window_transforms<NWX, NWY, BLOCK, 1, PW>(a, win, ex, twx, twy, 1, tid);
    __shared__ int row;
    if constexpr (C::NP <= 1024) {
        // short lists: a thread per bin
        if (tid == 0) row = p;
        __syncthreads();
        window_outputs<NWX, NWY, BLOCK, 1, PW>(a, win, 1, &row, tid);
        return;
    }
    constexpr int LNW = NWX == 16 ? 4 : NWX == 32 ? 5 : NWX == 64 ? 6 : 7;
    if (a.cbed) {
        const float fnorm = (float)a.inv_norm;
        for (int u = tid; u < C::NP; u += BLOCK) {
            const float2 z = win[(u >> LNW) * PW + (u & (NWX - 1))];
            a.cbed[(size_t)p * C::NP + u] = (z.x * z.x + z.y * z.y) * fnorm;
        }
    }
    if (!a.out) return;
    // a warp per annular bin: lanes over its pixel list, their FP32 sums folded to four (of the entries i mod 4;
    // no more additions deep than the four of window_outputs), which one lane per bin adds and scales in
    // FP64, 32 bins at a time
    constexpr int WARPS = BLOCK / 32;
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll 1
    for (int k0 = warp; k0 < a.nbins; k0 += 32 * WARPS) {
        float4 part = make_float4(0.f, 0.f, 0.f, 0.f);  // of bin k0 + WARPS lane
#pragma unroll 1
        for (int j = 0; j < 32; ++j) {
            const int k = k0 + WARPS * j;
            if (k >= a.nbins) break;
            float s = 0.f;
            const int e = __ldg(a.bin_off + k + 1);
            for (int i = __ldg(a.bin_off + k) + lane; i < e; i += 32) {
                const int u = __ldg(a.bin_idx + i);
                const float2 z = win[(u >> LNW) * PW + (u & (NWX - 1))];
                s = fmaf(z.x, z.x, fmaf(z.y, z.y, s));
            }
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const float4 q = make_float4(__shfl_sync(0xffffffffu, s, 0), __shfl_sync(0xffffffffu, s, 1), __shfl_sync(0xffffffffu, s, 2),
                                         __shfl_sync(0xffffffffu, s, 3));
            if (lane == j) part = q;
        }
        const int k = k0 + WARPS * lane;
        if (k < a.nbins) {
            const float val = (float)((((double)part.x + (double)part.y) + ((double)part.z + (double)part.w)) * a.inv_norm);
            float *o = a.out + (size_t)p * a.nbins + k;
            *o = a.accumulate ? *o + a.acc_w * val : val;
        }
    }
}

template <int NWX, int NWY>
static size_t list_smem(int n_beams) {
    return ListCfg<NWX, NWY>::FIXED + (size_t)n_beams * sizeof(float2);
}

template <int NWX, int NWY>
static cudaError_t list_launch(const ScanArgs &a, cudaStream_t s) {
    if (!a.attrs_set) {
        const cudaError_t e = allow_max_dynamic_smem(k_scan_list<NWX, NWY>);
        if (e != cudaSuccess) return e;
    }
    // CTAs per probe: as many (up to 8, of 4 beams or more) as leave two CTAs per SM or fewer
    int cn = 1;
    while (cn < 8 && (long long)a.n_probes * cn * 2 <= 2 * 152 && a.n_beams >= 8 * cn) cn *= 2;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cn;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)(a.n_probes * cn));
    c.blockDim = dim3(ListCfg<NWX, NWY>::BLOCK);
    c.dynamicSmemBytes = list_smem<NWX, NWY>(a.n_beams);
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k_scan_list<NWX, NWY>, a);
}

}  // namespace prism
