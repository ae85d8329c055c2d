// kernels_scan_rows.cu -- the raster-row scan (scan_rows.cuh) for windows of 16 and 32 columns, and the
// dispatch over all windows (64 and 128 columns in kernels_scan_rows_64.cu, compiled in parallel).
#include <cuda_runtime.h>

#include "params.h"
#include "scan_rows.cuh"

namespace prism {

int scan_rows_lp_64(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows);
cudaError_t launch_scan_rows_64(int nwx, int nwy, const ScanArgs &a, cudaStream_t s);

#define PRISM_ROWS_SIDES(X) X(16, 16) X(16, 32) X(16, 64) X(32, 16) X(32, 32) X(32, 64)

int scan_rows_lp(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows) {
#define PRISM_ROWS_LP(x, y) \
    if (nwx == x && nwy == y) return rows_lp<x, y>(m, max_beams, lists, px, rows);
    PRISM_ROWS_SIDES(PRISM_ROWS_LP)
#undef PRISM_ROWS_LP
    return scan_rows_lp_64(nwx, nwy, m, max_beams, lists, px, rows);
}

cudaError_t launch_scan_rows(int nwx, int nwy, const ScanArgs &a, cudaStream_t s) {
    if (!a.rows_w || a.rows_lp <= 0 || a.rows_chunk <= 0 || a.scan_px <= 0 || a.scan_py <= 0) return cudaErrorInvalidValue;
#define PRISM_ROWS_LAUNCH(x, y) \
    if (nwx == x && nwy == y) return rows_launch<x, y>(a, s);
    PRISM_ROWS_SIDES(PRISM_ROWS_LAUNCH)
#undef PRISM_ROWS_LAUNCH
    return launch_scan_rows_64(nwx, nwy, a, s);
}

}  // namespace prism
