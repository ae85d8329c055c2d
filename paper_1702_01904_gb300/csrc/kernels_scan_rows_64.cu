// kernels_scan_rows_64.cu -- the raster-row scan (scan_rows.cuh) for windows of 64 and 128 columns.
#include <cuda_runtime.h>

#include "params.h"
#include "scan_rows.cuh"

namespace prism {

#define PRISM_ROWS_SIDES(X) X(64, 16) X(64, 32) X(64, 64) X(128, 128)

int scan_rows_lp_64(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows) {
#define PRISM_ROWS_LP(x, y) \
    if (nwx == x && nwy == y) return rows_lp<x, y>(m, max_beams, lists, px, rows);
    PRISM_ROWS_SIDES(PRISM_ROWS_LP)
#undef PRISM_ROWS_LP
    return 0;
}

cudaError_t launch_scan_rows_64(int nwx, int nwy, const ScanArgs &a, cudaStream_t s) {
#define PRISM_ROWS_LAUNCH(x, y) \
    if (nwx == x && nwy == y) return rows_launch<x, y>(a, s);
    PRISM_ROWS_SIDES(PRISM_ROWS_LAUNCH)
#undef PRISM_ROWS_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace prism
