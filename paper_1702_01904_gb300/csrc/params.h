// params.h -- kernel parameter blocks and launcher declarations shared by the host engine
// (engine.cpp, plain C++) and the CUDA translation units.  Parameters travel by value in
// kernel parameter space (__grid_constant__), which keeps the 64 register-DFT twiddles in the
// constant bank.
#pragma once
#include <cuda.h>  // CUtensorMap
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace prism {

struct Tw64 {
    float2 w[64];   // W_64^j = exp(-2 pi i j / 64)
    // tangent form of the same twiddles, W_64^j = s (1 + i k) when |cos| >= |sin| (s = cos, k = tan;
    // (j mod 32) <= 8 or >= 24), else W_64^j = s (k + i) (s = sin, k = cot): sc[j] = (s, s), tk[j] = k
    float2 sc[64];
    float tk[64];
};

enum RowMode { ROW_STD = 0, ROW_PLANE = 1, ROW_OUT = 2 };
enum ColMode { COL_STD = 0, COL_PROBE = 1, COL_DETECT = 2 };

// Row pass over rows of length nx of a wave stack [batch][ny][nx] (x-Fourier between passes).
struct RowArgs {
    float2 *wave;              // [batch][ny][nx]
    const float2 *trans;       // t_p, [ny][nx]   (STD, PLANE)
    const float2 *tw_fwd;      // inter-stage twiddles of the forward split  [N1][N2]
    const float2 *tw_inv;      // inter-stage twiddles of the inverse split  [N2][N1]
    float2 *s_out;             // OUT: S-matrix [B][ny_s][nx_s]
    const int *beam_mn;        // PLANE: [B][2] (m, n)
    int ny;
    int n_rows;                // rows processed by this launch
    int f;                     // PLANE: interpolation factor along x
    int f_y;                   // PLANE: interpolation factor along y
    int beam0;                 // first beam of this batch (PLANE, OUT)
    int downsample;            // OUT
    int kx_half;               // > 0: only kx = -(kx_half-1) ... kx_half-1 of the mixed-domain wave are
                               // non-zero (the propagator's anti-aliasing aperture zeroes the rest):
                               // loads there are replaced by exact zeros and stores are skipped
                               // (STD, PLANE, OUT); 0: every kx
    int *err;                  // device error word: a TMA wait that ran out sets bit 2
    Tw64 tw;
};

// Column pass over columns of length ny.
struct ColArgs {
    CUtensorMap wave_map;      // TMA staging (STD): `wave` as FP32 [batch][ny][2 nx], boxes of 16 floats
                               // (8 columns) x min(ny, 256) rows x 1; valid when wave_map_ok
    CUtensorMap wave_map4;     // the same with boxes of 8 floats (4 columns)
    CUtensorMap out_map;       // TMA stores (STD): `wave` as FP32 [batch][lanes][regs][2 nx] with row
                               // y = lane + lanes * reg (lanes, regs: the column transform's threads
                               // and registers per column, col_fft_geometry), boxes of 16 floats x
                               // (regs + 1) x 32/8 x 1 -- one warp's rows of a finished tile in the
                               // padded exchange layout; the pad entry lies past `regs` and is not stored
    CUtensorMap out_map4;      // the same for 4 columns: boxes of 8 floats x (regs + 1) x 32/4 x 1
    float2 *wave;              // [batch][ny][nx]
    float *inten;              // DETECT: [batch][ny][nx] |Psi|^2 (scaled later)
    const float2 *prop_x;      // [nx]  exp(-i pi lambda dz qx^2)
    const float2 *prop_y;      // [ny]  exp(-i pi lambda dz qy^2) / (nx ny)
    const int *aa_kmax;        // [nx]  largest |ky| inside the AA aperture on column kx, -1 if none
    const float2 *tw_fwd;
    const float2 *tw_inv;
    const float2 *probe_base;  // PROBE: [ny][nx] A(q) exp(-i chi(q))
    const float2 *shift_x;     // PROBE: [batch][nx] exp(-2 pi i qx x0)
    const float2 *shift_y;     // PROBE: [batch][ny] exp(-2 pi i qy y0)
    int nx;
    int batch;
    float probe_scale;         // PROBE: 1 / (nx ny)
    int kx_half;               // > 0: only the column tiles holding kx = -(kx_half-1) ... kx_half-1 are
                               // processed (every other column is zero after the propagator); 0: all
    int band4;                 // 1: the aperture keeps |ky| < ny/4 on every column (aa_kmax < ny/4), so
                               // the column transforms may drop that band's complement at compile
                               // time (STD, DETECT)
    int wave_map_ok;           // 1: the four maps describe `wave` (the TMA-staged shapes may run)
    int *tile_ctr;             // TMA-staged shapes: [2] the next tile and the CTAs done (zero between
                               // launches; the launch that ends last zeroes them), or NULL: tiles by a
                               // fixed stride
    int *err;                  // device error word: a TMA wait that ran out sets bit 1
    Tw64 tw;
};

// PRISM probe scan (coefficients, window gather, beam sum, window FFT, |.|^2, bins).
struct ScanArgs {
    const float2 *S;           // [B][ny_s][nx_s]
    const double *x0;          // [P]
    const double *y0;          // [P]
    const double *qx;          // [B] beam qx = m f / cell_x
    const double *qy;          // [B]
    const float2 *base;        // [B] A(q_b) exp(-i chi(q_b))
    const float2 *tw_fwd;      // window FFT inter-stage twiddles (rows, length nw_x)
    const float2 *tw_fwd_y;    // window FFT inter-stage twiddles (columns, length nw_y)
    const float2 *tw_inv;      // (unused by the forward-only window FFT; kept for symmetry)
    const int *bin_off;        // [nbins+1] CSR offsets into bin_idx
    const int *bin_idx;        // window pixel indices (ky*nw + kx) grouped by bin
    const int *bin_idx_t;      // the same lists by rank: entry i of bin k at [i * nbins + k] (rows of
                               // the longest bin; bin k's list ends at bin_off[k+1] - bin_off[k])
    const uint16_t *bin_idx16; // bin_idx as 16-bit entries, 16-byte aligned and padded to 16 bytes (the
                               // copy a scan stages in shared memory where it fits), or NULL
    int n_bin_idx;             // entries of bin_idx (bin_off[nbins])
    float *out;                // [P][nbins] annular bins, or NULL
    float *cbed;               // [P][nw][nw] full window diffraction patterns (FFT order), or NULL
    float acc_w;               // accumulate: out += acc_w * I (else out = I)
    int accumulate;
    double px_s, py_s;         // stored pixel size
    double shift_x, shift_y;   // h tan(theta): the coefficients use r0 - shift (probe tilt)
    double inv_norm;           // 1 / (nw^4 * sum_b A_b)
    int n_beams;
    int nx_s, ny_s;
    int nbins;
    int n_probes;
    int probe0;
    // 16-bit mode (tensor-core beam sum)
    const void *S16;           // [ny_s * nx_s][kp] 16-bit (re, im) of each beam, zero-padded beams
                               // (split mode: [ny_s * nx_s][2][kp], value row then remainder row)
    const float *beam_scale;   // [B] power of two: S_b = S16_b * beam_scale[b]
    float2 *win;               // window scratch [slots][probes per group][nw][nw]
    int *win_cnt;              // [gridDim.x] parts finished per split block, then the next work unit and
                               // the CTAs done (all zero between launches)
    int *err;                  // device error word (a bounded wait that ran out sets bit 0)
    int kp;                    // K = 2 * roundup(B, 8)
    int scan_px, scan_py;      // probe raster, probe index = row * scan_px + col
    // raster rows of one y each (scan_rows.cuh); rows_lp = 0: not such a scan
    const int *m_off;          // [2 M + 2] CSR over m = -M ... M: the beams of m, n ascending
    const int *m_beam;         // [B]
    const double *m_qx;        // [M + 1] qx of the beams m = 0 ... M
    int rows_m;                // M
    int rows_maxn;             // beams of one m at most
    float2 *rows_w;            // [rows_chunk][nw_y][2 M + 1][rows_cols] transformed sums over n
    int rows_g0, rows_cols;    // columns held: rows_g0 ... rows_g0 + rows_cols - 1 (mod nx_s), multiples of 16
    int rows_chunk;            // raster rows whose sums are held at once
    const float2 *rows_src;    // the beams' values under the windows, [B][rows_ry][rows_pitch] from pixel
    int rows_x0, rows_y0;      // (rows_x0, rows_y0) on (mod the stored grid): S itself, or (rows_unpack) the
    int rows_pitch, rows_ry;   // reach of the windows unpacked from the value + remainder rows of S16
    int rows_unpack;
    int rows_lp;               // probes per CTA
    int rows_0, rows_n;        // set per launch: first raster row, raster rows
    int attrs_set;             // the row or list kernels' shared-memory limits are set (by this plan, before)
    int list;                  // 1: probe by probe (scan_list.cuh), positions too far apart to share S values
    const uint16_t *fold16;    // the bins over the quadrant 0 <= kx <= nw_x/2, 0 <= ky <= nw_y/2: CSR offsets
                               // [nbins + 1], then the lists (ky * (nw_x/2 + 1) + kx); 16-byte aligned
    int n_fold16;              // its entries, padded to 8 (0: no bins)
    Tw64 tw;
};

// FP32 S of one beam batch -> per-beam scale and pixel-major 16-bit S
struct QuantArgs {
    const float2 *S;           // [nb][npix]
    void *S16;                 // [npix][kp]
    float *scale;              // [B]
    int beam0, nb, npix, kp;
    int mode;                  // 0: FP16, 1: BF16, 2: FP16 value + FP16 remainder (two rows of kp)
};

struct ShiftArgs {
    const double *x0, *y0;     // [batch]
    float2 *shift_x;           // [batch][nx]
    float2 *shift_y;           // [batch][ny]
    int nx, ny, batch;
    double cell_x, cell_y;
};

// The detector's pixel lists of a full grid, made on the device: CSR of the pixels ky * nx + kx (FFT order)
// by bin = floor((1000 lambda |q| - start) / step), q = (kx / cell_x, ky / cell_y), each list in pixel order
struct BinListArgs {
    int nx, ny, nbins;
    double cell_x, cell_y, lam, start, step;
    uint16_t *map;             // [ny/2 + 1][nx/2 + 1] bin of (|ky|, |kx|), 0xffff: none
    int *rows;                 // [ny/2 + 1][nbins] pixels of a row per bin
    int *base;                 // [ny][nbins] pixels of the rows before
    int *total;                // [nbins]
    int *off;                  // [nbins + 1]
    int *idx;                  // [nx * ny] at most
};
// the entries of a probe's aperture: base[idx[i]] = val[i], every other pixel zero
struct ProbeBaseArgs {
    const int *idx;
    const float2 *val;
    float2 *base;
    int n;
};

struct BinArgs {
    const float *inten;        // [batch][npix]
    const int *bin_off;        // [nbins+1]
    const int *bin_idx;
    float *out;                // [batch][nbins]
    double scale;
    int npix, nbins, batch;
    const int *err;            // optional device error word of the passes: non-zero -> the bins are NaN
};

// Small tables that travel as kernel parameters (launch_put): `data` holds n0 8-byte words for dst0, then
// n1 for dst1
constexpr int PUT_SMALL = 448, PUT_LARGE = 2000;  // words: about 4 and 16 KB of parameters
template <int N>
struct PutArgs {
    unsigned long long *dst0, *dst1;
    int n0, n1;
    unsigned long long data[N];
};

// launchers (kernels_build.cu, kernels_scan.cu); return cudaSuccess or the launch error
cudaError_t launch_transmission(const float *V, float2 *t, size_t n, double sigma_cycles, cudaStream_t s);
// first-slice rows of beams beam0 .. beam0+nb-1 from T0 = FFT_x(t_0) [ny][nx] (kept columns only)
cudaError_t launch_plane(const float2 *T0, float2 *wave, const int *beam_mn, int beam0, int nb, int nx, int ny, int f, int f_y,
                         int kx_half, cudaStream_t s);
cudaError_t launch_row(int nx, RowMode mode, const RowArgs &a, cudaStream_t s);
cudaError_t launch_col(int ny, ColMode mode, const ColArgs &a, cudaStream_t s);
// the column transform of length ny: threads (lanes) per column and registers per thread, whose
// result row is lane + lanes * register (false for an unsupported ny)
bool col_fft_geometry(int ny, int *lanes, int *regs);
cudaError_t launch_scan(int nw, const ScanArgs &a, cudaStream_t s);
// nw_x x nw_y windows (separate f_x, f_y): square ones as launch_scan, rectangular ones (16, 32, 64
// per side) through the grouped kernel; scan_rect_supported says whether a launch can succeed
cudaError_t launch_scan_rect(int nwx, int nwy, const ScanArgs &a, cudaStream_t s);
bool scan_rect_supported(int nwx, int nwy, int n_beams);
// FP32 GEMM scan over raster blocks of 32 probes (window sides 16, 32, 64) in one of the
// contraction tile shapes (0 = default 4 x 8 blocks; the others for square windows): persistent
// grid (0 if it does not fit), launch, and the window scratch it needs
int scan_gemm_grid(int nwx, int nwy, int shape, int n_beams, int scan_px, int scan_py);
cudaError_t launch_scan_gemm(int nwx, int nwy, int shape, int grid, const ScanArgs &a, cudaStream_t s);
// window scratch of the FP32 GEMM scan: one slot per CTA plus one per split group of the last round
size_t scan_gemm_win_bytes(int nwx, int nwy, int shape, int grid, int scan_px, int scan_py);
// the contraction shapes: count, whether one is compiled for a window, its name; the tuned unit
int scan_gemm_shapes();
bool scan_gemm_shape_valid(int nwx, int nwy, int shape);
const char *scan_gemm_shape_name(int shape);
int scan_gemm_grid_tuned(int nwx, int nwy, int shape, int n_beams, int scan_px, int scan_py);
cudaError_t launch_scan_gemm_tuned(int nwx, int nwy, int shape, int grid, const ScanArgs &a, cudaStream_t s);
// scan counters: completion counters of the split groups (int[grid]), the next work unit and the
// CTAs done (int[2]); zeroed once, each launch leaves them zero
size_t scan_gemm_cnt_bytes(int grid);
// the raster-row scan (scan_rows.cuh): probes per CTA for rows of px probes
// and so many 16-bit entries of bin lists (0: these windows, beams
// or sizes are not for it), launch
size_t scan_rows_unpack_bytes(const ScanArgs &a);  // bytes of rows_src where it is unpacked
int scan_rows_lp(int nwx, int nwy, int m, int max_beams, int lists, int px, int rows);
// the position-list scan (scan_list.cuh): whether it takes these windows and beams, launch
bool scan_list_supported(int nwx, int nwy, int n_beams);
cudaError_t launch_scan_list(int nwx, int nwy, const ScanArgs &a, cudaStream_t s);
cudaError_t launch_scan_rows(int nwx, int nwy, const ScanArgs &a, cudaStream_t s);
cudaError_t launch_shift(const ShiftArgs &a, cudaStream_t s);
cudaError_t launch_bins(const BinArgs &a, cudaStream_t s);
// two host arrays of 8-byte words to the device in one launch (n0 + n1 <= PUT_LARGE); the arrays are read
// before it returns
cudaError_t launch_put(void *dst0, const void *src0, int n0, void *dst1, const void *src1, int n1, cudaStream_t s);
cudaError_t launch_bin_lists(const BinListArgs &a, cudaStream_t s);
cudaError_t launch_probe_base(const ProbeBaseArgs &a, size_t npix, cudaStream_t s);
cudaError_t launch_tc_selftest(float *out, int *status, cudaStream_t s);
cudaError_t launch_wait_selftest(int *status, long long limit_cycles, int arrive, cudaStream_t s);
// 16-bit mode (kernels_tc.cu)
cudaError_t launch_quantize(const QuantArgs &a, cudaStream_t s);
cudaError_t launch_dequantize(const void *S16, const float *scale, float2 *out, int n_beams, int npix, int kp,
                              int mode, cudaStream_t s);
cudaError_t launch_scan_tc(int nw, int mode, int shape, int grid, const ScanArgs &a, cudaStream_t s);
bool scan_tc_supported(int nw);
// persistent grid of the tensor-core scan (resident CTAs, at most the probe groups), 0 if it does
// not fit; window scratch bytes for that grid
int scan_tc_grid(int nw, int kp, int mode, int shape, int scan_px, int scan_py);
// ring shapes of the tensor-core scan's A operand (scan_tc.cuh): count for a mode, name; the
// non-default shapes (kernels_tc_tune.cu)
int scan_tc_shapes(int mode);
const char *scan_tc_shape_name(int shape);
int scan_tc_grid_tuned(int nw, int kp, int mode, int shape, int scan_px, int scan_py);
cudaError_t launch_scan_tc_tuned(int nw, int mode, int shape, int grid, const ScanArgs &a, cudaStream_t s);
// window scratch of the tensor-core scan: one slot per CTA plus one per split block of the last round
size_t scan_tc_win_bytes(int nw, int grid, int scan_px, int scan_py);
// autotuner launch shapes of ROW_STD (kind 0) and COL_STD (kind 1), N = 256 ... 2048 (kernels_tune.cu)
int tune_shapes(int kind);
const char *tune_shape_name(int kind, int v);
int tune_default_shape(int kind, int n);
bool tune_shape_valid(int kind, int n, int v);
bool tune_shape_needs_map(int kind, int v);  // the shape stages through TMA (ColArgs::wave_map)
int tune_shape_fft_variant(int kind, int v);  // its FFT radix variant (DftSplit), -1 if unknown
int tune_default_fft_variant(int n);          // the radix variant of the default launchers at N
// the shape of a standard pass when none is tuned or pinned (-1: the default launcher): rows of all
// waves; columns of all waves, whether tensor maps of the waves are at hand; shared: beside other
// kernels on the same SMs
int tune_row_default(int nx, long long rows, bool shared);
int tune_col_default(int ny, long long cols, bool maps, bool shared);
bool tune_shape_fills_sm(int kind, int v);    // 3 or more CTAs per SM, each with a third of its resources
cudaError_t launch_row_shape(int nx, int v, const RowArgs &a, cudaStream_t s);
// the standard row pass in its default shape (tune_row_default); every shape computes the same rows
cudaError_t launch_row_std(int nx, const RowArgs &a, cudaStream_t s);
cudaError_t launch_col_shape(int ny, int v, const ColArgs &a, cudaStream_t s);
// smallest scan-window / FFT sizes the kernels are instantiated for
bool row_supported(int n);
bool col_supported(int n);
bool scan_supported(int nw);
// FFT split used by the kernels for length n: forward (n1, n2)
void fft_split(int n, int *n1, int *n2);

}  // namespace prism
