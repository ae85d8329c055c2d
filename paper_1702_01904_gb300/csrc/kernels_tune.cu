// kernels_tune.cu -- the autotuner's launch shapes of the two multislice passes (ROW_STD and
// COL_STD, N = 256 ... 2048): names, lookups and the dispatch on N to the kernels_tune_<N>.cu units,
// which instantiate the shapes (tune_pass.cuh).  A shape changes only how rows or columns are spread
// over threads, whether the next row/tile is staged through shared memory (with cp.async, by bulk or
// tiled TMA copies completing on an mbarrier), and the FFT radix: the split of the 32- and 64-point
// register DFTs (DftSplit) of the pass's forward and inverse transform.  Shapes of one radix variant
// compute bitwise the same transform; the variants round differently.
#include <cuda_runtime.h>

#include "params.h"
#include "tune_pass.cuh"

namespace prism {

namespace {

using tune::COL_SHAPES;
using tune::N_COL;
using tune::N_ROW;
using tune::ROW_SHAPES;
const char *ROW_NAMES[N_ROW] = {"128 thr",
                                "256 thr",
                                "128 thr, staged",
                                "256 thr, staged",
                                "128 thr, TMA",
                                "256 thr, TMA",
                                "384 thr, staged",
                                "384 thr, TMA",
                                "384 thr, TMA, radix-4 first: forward",
                                "384 thr, TMA, radix-4 first: inverse",
                                "384 thr, TMA, radix-4 first: both",
                                "128 thr, radix-4 first: both",
                                "128 thr, staged, radix-4 first: both",
                                "384 thr, radix-4 first: both"};
const char *COL_NAMES[N_COL] = {"W4, staged",
                                "W8, staged",
                                "W16, staged",
                                "W4, TMA, 3/SM",
                                "W8",
                                "W8, TMA",
                                "W8, 2/SM",
                                "W4, staged, 3/SM",
                                "W4, TMA, 3/SM, radix-4 first: forward",
                                "W4, TMA, 3/SM, radix-4 first: inverse",
                                "W4, TMA, 3/SM, radix-4 first: both",
                                "W8, staged, radix-4 first: both",
                                "W8, radix-4 first: both",
                                "W4, staged, radix-4 first: both"};
static_assert(sizeof(ROW_NAMES) / sizeof(ROW_NAMES[0]) == N_ROW && sizeof(COL_NAMES) / sizeof(COL_NAMES[0]) == N_COL, "one name per shape");

}  // namespace

int tune_shapes(int kind) { return kind == 0 ? N_ROW : kind == 1 ? N_COL : 0; }

const char *tune_shape_name(int kind, int v) {
    if (kind == 0 && v >= 0 && v < N_ROW) return ROW_NAMES[v];
    if (kind == 1 && v >= 0 && v < N_COL) return COL_NAMES[v];
    return "?";
}

int tune_default_shape(int kind, int n) {
    const int rv = default_fft_variant(n);
    if (kind == 0) {
        const int thr = n >= 2048 ? 384 : n >= 512 ? 128 : 256;  // row_default_threads, unstaged
        for (int v = 0; v < N_ROW; ++v)
            if (ROW_SHAPES[v].a == thr && !ROW_SHAPES[v].stg && !ROW_SHAPES[v].tma && ROW_SHAPES[v].rv == rv) return v;
    } else if (kind == 1) {
        const int w = n >= 1024 ? 8 : 16;  // col_default_w
        const bool stg = n < 2048;         // col_default_stg
        for (int v = 0; v < N_COL; ++v)
            if (COL_SHAPES[v].a == w && COL_SHAPES[v].stg == stg && COL_SHAPES[v].mb == 0 && !COL_SHAPES[v].tma &&
                COL_SHAPES[v].rv == rv)
                return v;
    }
    return -1;
}

int tune_default_fft_variant(int n) { return default_fft_variant(n); }

int tune_shape_fft_variant(int kind, int v) {
    if (kind == 0 && v >= 0 && v < N_ROW) return ROW_SHAPES[v].rv;
    if (kind == 1 && v >= 0 && v < N_COL) return COL_SHAPES[v].rv;
    return -1;
}

bool tune_shape_needs_map(int kind, int v) { return kind == 1 && v >= 0 && v < N_COL && COL_SHAPES[v].tma; }

bool tune_shape_fills_sm(int kind, int v) { return kind == 1 && v >= 0 && v < N_COL && COL_SHAPES[v].mb >= 3; }

static int tune_row_find(int thr, bool stg, bool tma) {
    for (int v = 0; v < N_ROW; ++v)
        if (ROW_SHAPES[v].a == thr && ROW_SHAPES[v].stg == stg && ROW_SHAPES[v].tma == tma && ROW_SHAPES[v].rv == 0) return v;
    return -1;
}

// The row pass's launch shape when none is tuned or pinned (-1: the default launcher).  N = 1024: 384
// threads (12 warps per SM) with the next row's two kept quarters staged by bulk TMA copies (0.292 ms
// per launch for 129 beams, against 0.315 for 256 threads staged by cp.async and 0.333 for 128 threads
// unstaged).  N = 512: 384 threads staged by cp.async from 16 384 rows on (213 beams: 123 us against
// 132 for 128 threads unstaged; 829 beams 446 against 490; 49 beams 33.4 against 33.5; with 13 beams,
// 6656 rows, the small CTAs are faster, 12.9 against 14.0).  In a batch graph, whose branches share the
// SMs, the default launcher: smaller CTAs up to N = 1024 (the 1024 shape holds 163 KB of shared memory per CTA).
// At N = 2048 it is one CTA of 384 threads per SM there too, which loses less by the other branches' kernels than
// it gains: four 2048^2 cells in 4 branches 51.4 ms per run, with CTAs of 128 threads 55.8; two beside six
// 1024^2 cells 31.2 against 32.9; one beside twelve 256^2 cells 14.1 against 14.4.
int tune_row_default(int nx, long long rows, bool shared) {
    if (shared) return -1;
    const int v = nx == 1024 ? tune_row_find(384, false, true) : nx == 512 && rows >= 16384 ? tune_row_find(384, true, false) : -1;
    return v >= 0 && tune_row_valid(nx, v) ? v : -1;
}

cudaError_t launch_row_std(int nx, const RowArgs &a, cudaStream_t s) {
    const int v = tune_row_default(nx, a.n_rows, false);
    return v >= 0 ? tune_row_launch(nx, v, a, s) : launch_row(nx, ROW_STD, a, s);
}

static int tune_col_find(int w, bool stg, bool tma) {
    for (int v = 0; v < N_COL; ++v)
        if (COL_SHAPES[v].tma == tma && COL_SHAPES[v].a == w && COL_SHAPES[v].stg == stg && COL_SHAPES[v].rv == 0 &&
            (tma || COL_SHAPES[v].mb == 0))
            return v;
    return -1;
}

// The column pass's launch shape when none is tuned or pinned (-1: the default launcher), for `cols`
// columns in all and with (maps) or without tensor maps of the wave stack.  N = 1024: 4 columns per CTA
// staged by TMA, 3 CTAs per SM (0.200 ms for 129 beams, against 0.293 for 8 columns by TMA and 0.320
// by cp.async).  N = 512: the same from 8192 columns on (213 beams, 54 528 columns: 88 us against 125 for
// 16 columns by cp.async; 49 beams 24.2 against 31.2), below that 8 columns unstaged (13 beams, 3328
// columns: 10.8 against 12.4 by TMA and 12.8).  N = 256: 8 columns by TMA from 16 384 columns on (829
// beams, 106 112 columns: 82 us against 110 for 16 columns by cp.async; 213 beams 23.1 against 30.9),
// below that 8 columns unstaged (49 beams, 6272 columns: 8.7 against 10.8 for either).
// In a batch graph with parallel branches the passes of different cells share the SMs, and a shape that
// fills an SM by itself (3 CTAs of 66 KB and 168 x 128 registers) leaves no room for the other branches'
// kernels: there the default is 8 columns by TMA at N = 1024 (one 131 KB CTA per SM) and the default
// launcher elsewhere, and the autotuner skips the SM-filling shapes (64 uneven cells, 4 branches: 2.78 s
// per run with them, 2.25 s without).
int tune_col_default(int ny, long long cols, bool maps, bool shared) {
    int v = -1;
    if (ny == 1024) v = maps ? tune_col_find(shared ? 8 : 4, false, true) : -1;
    else if (shared) v = -1;
    else if (ny == 512) v = maps && cols >= 8192 ? tune_col_find(4, false, true) : tune_col_find(8, false, false);
    else if (ny == 256) v = maps && cols >= 16384 ? tune_col_find(8, false, true) : tune_col_find(8, false, false);
    return v >= 0 && tune_shape_valid(1, ny, v) ? v : -1;
}

bool tune_row_valid(int n, int v) {
    switch (n) {
        case 256: return tune::row_valid<256>(v, tune::RowSeq{});
        case 512: return tune::row_valid<512>(v, tune::RowSeq{});
        case 1024: return tune::row_valid<1024>(v, tune::RowSeq{});
        case 2048: return tune::row_valid<2048>(v, tune::RowSeq{});
    }
    return false;
}

cudaError_t tune_row_launch(int nx, int v, const RowArgs &a, cudaStream_t s) {
    switch (nx) {
        case 256: return tune::row_launch_n256(v, a, s);
        case 512: return tune::row_launch_n512(v, a, s);
        case 1024: return tune::row_launch_n1024(v, a, s);
        case 2048: return tune::row_launch_n2048(v, a, s);
    }
    return cudaErrorInvalidValue;
}

bool tune_shape_valid(int kind, int n, int v) {
    if (kind == 0) {
        return tune_row_valid(n, v);
    } else if (kind == 1) {
        switch (n) {
            case 256: return tune::col_valid<256>(v, tune::ColSeq{});
            case 512: return tune::col_valid<512>(v, tune::ColSeq{});
            case 1024: return tune::col_valid<1024>(v, tune::ColSeq{});
            case 2048: return tune::col_valid<2048>(v, tune::ColSeq{});
        }
    }
    return false;
}

cudaError_t launch_row_shape(int nx, int v, const RowArgs &a, cudaStream_t s) {
    if (!tune_shape_valid(0, nx, v)) return cudaErrorInvalidValue;
    return tune_row_launch(nx, v, a, s);
}

cudaError_t launch_col_shape(int ny, int v, const ColArgs &a, cudaStream_t s) {
    if (!tune_shape_valid(1, ny, v)) return cudaErrorInvalidValue;
    switch (ny) {
        case 256: return tune::col_launch_n256(v, a, s);
        case 512: return tune::col_launch_n512(v, a, s);
        case 1024: return tune::col_launch_n1024(v, a, s);
        case 2048: return tune::col_launch_n2048(v, a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace prism
