// kernels_scan_list.cu -- the position-list scan (scan_list.cuh) for every window of 16 to 128 pixels.
#include <cuda_runtime.h>

#include "params.h"
#include "scan_list.cuh"

namespace prism {

#define PRISM_LIST_SIDES(X) \
    X(16, 16) X(16, 32) X(16, 64) X(32, 16) X(32, 32) X(32, 64) X(64, 16) X(64, 32) X(64, 64) X(128, 128)

bool scan_list_supported(int nwx, int nwy, int n_beams) {
#define PRISM_LIST_FITS(x, y) \
    if (nwx == x && nwy == y) return list_smem<x, y>(n_beams) <= 226 * 1024;
    PRISM_LIST_SIDES(PRISM_LIST_FITS)
#undef PRISM_LIST_FITS
    return false;
}

cudaError_t launch_scan_list(int nwx, int nwy, const ScanArgs &a, cudaStream_t s) {
    if (a.n_probes <= 0) return cudaSuccess;
#define PRISM_LIST_LAUNCH(x, y) \
    if (nwx == x && nwy == y) return list_launch<x, y>(a, s);
    PRISM_LIST_SIDES(PRISM_LIST_LAUNCH)
#undef PRISM_LIST_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace prism
