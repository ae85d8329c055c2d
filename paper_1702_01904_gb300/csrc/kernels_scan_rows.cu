// kernels_scan_rows.cu -- the raster-row scan (scan_rows.cuh) for windows of 16 and 32 columns, and the
// dispatch over all windows (64 and 128 columns in kernels_scan_rows_64.cu, compiled in parallel).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "params.h"
#include "scan_rows.cuh"

namespace prism {

int scan_rows_lp_64(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows);
cudaError_t launch_scan_rows_64(int nwx, int nwy, const ScanArgs &a, cudaStream_t s);

#define PRISM_ROWS_SIDES(X) X(16, 16) X(16, 32) X(16, 64) X(32, 16) X(32, 32) X(32, 64)

// FP16 value + remainder rows of S16 (pixel by pixel) -> FP32 planes (beam by beam) of the columns and rows
// under the windows: 32 pixels x 32 beams per CTA through shared memory, 128-byte runs of beams read,
// 256-byte runs of pixels written.  value + remainder is exact in FP32 (22 bits), the scale a power of two.
// Bound by memory: 1 KB read and written per 128 beams and pixel.
__global__ void __launch_bounds__(256) k_rows_unpack(const __grid_constant__ ScanArgs a, float2 *out) {
    __shared__ float2 tile[32][33];
    const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x0 = blockIdx.x * 32, y = blockIdx.y, b0 = blockIdx.z * 32;
    const int b = b0 + lane;
    next_may_start();
    after_previous();
    const uint32_t *src = reinterpret_cast<const uint32_t *>(a.S16) + (size_t)((a.rows_y0 + y) & (a.ny_s - 1)) * a.nx_s * a.kp;
    if (b < a.n_beams) {
        const float sc = a.beam_scale[b];
        for (int p = ty; p < 32 && x0 + p < a.rows_pitch; p += 8) {
            const uint32_t *w = src + (size_t)((a.rows_x0 + x0 + p) & (a.nx_s - 1)) * a.kp + b;
            const uint32_t wh = __ldg(w), wl = __ldg(w + a.kp / 2);
            const float2 hi = __half22float2(*reinterpret_cast<const __half2 *>(&wh)), lo = __half22float2(*reinterpret_cast<const __half2 *>(&wl));
            tile[lane][p] = make_float2((hi.x + lo.x) * sc, (hi.y + lo.y) * sc);
        }
    }
    __syncthreads();
    if (x0 + lane >= a.rows_pitch) return;
    for (int j = ty; j < 32 && b0 + j < a.n_beams; j += 8)
        out[((size_t)(b0 + j) * a.rows_ry + y) * a.rows_pitch + x0 + lane] = tile[j][lane];
}

size_t scan_rows_unpack_bytes(const ScanArgs &a) { return (size_t)a.n_beams * a.rows_ry * a.rows_pitch * sizeof(float2); }

int scan_rows_lp(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows) {
#define PRISM_ROWS_LP(x, y) \
    if (nwx == x && nwy == y) return rows_lp<x, y>(m, max_beams, lists, px, rows);
    PRISM_ROWS_SIDES(PRISM_ROWS_LP)
#undef PRISM_ROWS_LP
    return scan_rows_lp_64(nwx, nwy, m, max_beams, lists, px, rows);
}

cudaError_t launch_scan_rows(int nwx, int nwy, const ScanArgs &a, cudaStream_t s) {
    if (!a.rows_w || !a.rows_src || a.rows_lp <= 0 || a.rows_chunk <= 0 || a.scan_px <= 0 || a.scan_py <= 0) return cudaErrorInvalidValue;
    if (a.rows_unpack) {
        const dim3 grid((a.rows_pitch + 31) / 32, a.rows_ry, (a.n_beams + 31) / 32);
        const cudaError_t e = launch_chained(k_rows_unpack, grid, 256, 0, s, a, const_cast<float2 *>(a.rows_src));
        if (e != cudaSuccess) return e;
    }
#define PRISM_ROWS_LAUNCH(x, y) \
    if (nwx == x && nwy == y) return rows_launch<x, y>(a, s);
    PRISM_ROWS_SIDES(PRISM_ROWS_LAUNCH)
#undef PRISM_ROWS_LAUNCH
    return launch_scan_rows_64(nwx, nwy, a, s);
}

}  // namespace prism
