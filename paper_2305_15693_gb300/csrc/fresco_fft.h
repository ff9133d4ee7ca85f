// Transforms of the FP32 fine grids fused with the steps around them (fresco_fft.cu): host side.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "fresco_internal.h"

namespace fresco {

constexpr int kFftMaxPasses = 8;

// A complex transform of length n = r[0] r[1] ... r[np - 1], in place in shared memory: pass p
// splits blocks of length m[p] r[p] into r[p] parts of m[p]. pos[k] is the place of frequency k
// after the forward passes; tw[k] = exp(-2 pi i k / n).
struct FftDesc {
    int n = 0, np = 0;
    int r[kFftMaxPasses] = {}, m[kFftMaxPasses] = {};
    FastDiv dm[kFftMaxPasses];   // division by m[p]
    FastDiv db[kFftMaxPasses];   // division by n / r[p], the butterflies of one transform
    const float2 *tw = nullptr;
    const int *pos = nullptr;
    int shift = 31, words = 0;   // padding (fft_place), elements a padded row takes
    int threads = 0;             // threads per block
    int rows = 1;                // transforms per block
};

// padded place of element i (shift 31: no padding): strides that are powers of two would meet in one
// shared-memory bank
__host__ __device__ inline int fft_place(const FftDesc &f, int i) { return i + (i >> f.shift); }
inline size_t fft_bytes(const FftDesc &f, int rows) {
    return sizeof(float2) * (size_t)rows * f.words;
}
// Most threads of a block, and the blocks per SM the registers leave room for. The transforms wait on
// shared-memory and global loads, so warps in flight count more than fewer passes: with radices up to
// 20 (100 registers, two or three blocks) the x pass of 6480^2 took 141 .. 197 us and the column
// kernel 182 .. 361 us, with radices up to 10 in 64 registers 144 and 159 us.
constexpr int kFftThreads = 256;
constexpr int kFftBlocks = 4;

// largest length whose one transform fits a block's shared memory
constexpr size_t kFftSmem = 224 * 1024;

// Whether n factors into the radices used and fits; fills everything but the device tables.
bool fft_describe(int n, FftDesc &f);
// Device tables of a described transform (allocations appended to allocs)
fresco_status fft_tables(FftDesc &f, std::vector<void *> &allocs, int64_t &bytes);
// Transforms per block and threads for the row kernels; rows: rows of a launch
void fft_size_rows(FftDesc &f, int64_t rows);
// Threads for one transform per block
void fft_size_cols(FftDesc &f);

// Real rows of 2 M floats -> columns k = 0 .. kx of their half spectra, transposed: xt[k][row].
// f: the transform of length M; tws: exp(-2 pi i k / 2M), k <= M / 2.
cudaError_t fft_rows_forward(const FftDesc &f, const float *grid, float2 *xt, const float2 *tws,
                             int64_t rows, int kx, cudaStream_t s);
// The inverse: transposed half spectra bt[k][row], k = 0 .. kx, -> real rows.
cudaError_t fft_rows_inverse(const FftDesc &f, const float2 *bt, float *grid, const float2 *tws,
                             int64_t rows, int kx, cudaStream_t s);
// Transposed columns bt[c][row], c = 0 .. 2 kx + 1 for n_x = c - kx - 1, -> complex rows of length n.
cudaError_t fft_rows_inverse_c(const FftDesc &f, const float2 *bt, float2 *g, int64_t rows, int kx,
                               cudaStream_t s);

// 2D column pass: for every column n_x = 0 .. kx, the forward transform along y, the mask (S, loss,
// gradient coefficients) and the inverse transform, in shared memory.
struct ColsArgs {
    MaskGeom m;
    const float2 *xt;             // [kx + 1][nf1]
    float2 *bt;                   // kderiv: [kx + 1][nf1]; direct: [2 kx + 2][nf1]
    const int *rep_n;             // representatives, n_x major
    const float *rep_s0, *rep_w;
    const int *rep_first;         // [kx + 2] first representative of every column
    const float *ip0, *ip1;
    double *partial;              // [kx + 1] loss partials
};
cudaError_t fft_cols_mask(const FftDesc &f, const ColsArgs &a, double loss_const, double *loss,
                          unsigned *done, cudaStream_t s);
// The same steps for the size classes of an ensemble, up to kFftClasses of them in a launch: blocks
// first[i] .. first[i + 1] - 1 work on class i, `blocks` of them on each of its `count` grids.
constexpr int kFftClasses = 16;
struct FftClass {
    FftDesc f;
    int64_t in0 = 0, in_stride = 0;     // the first grid's input and the next one's, in elements
    int64_t out0 = 0, out_stride = 0;
    int64_t tw0 = 0;                    // row steps: the class's part of the twiddles
    int rows = 0, kx = 0, blocks = 0, count = 0;
    int list0 = 0;                      // column step: the class's first entry of ColsBatch::list
};
struct FftClassSet {
    int n = 0, threads = 0;
    size_t smem = 0;
    int first[kFftClasses + 1] = {};
    FftClass c[kFftClasses];
};
static_assert(sizeof(FftClassSet) <= 16384, "passed as a kernel argument");
// launches for the classes of one step; col_buffers: buffers of a column (0: a row step)
std::vector<FftClassSet> fft_class_sets(std::vector<FftClass> cls, int col_buffers);
cudaError_t fft_rows_forward_b(const FftClassSet &q, const float *grid, float2 *xt,
                               const float2 *tws, cudaStream_t s);
cudaError_t fft_rows_inverse_b(const FftClassSet &q, const float2 *bt, float *grid,
                               const float2 *tws, cudaStream_t s);
cudaError_t fft_rows_inverse_cb(const FftClassSet &q, const float2 *bt, float2 *g, cudaStream_t s);
struct ColsBatch {
    const BInst *inst;
    const int *list;              // instances, class by class
    const int *rep_first;         // per instance at rep_off[i]
    const int64_t *rep_off;
    const float2 *xt;
    float2 *bt;
    const int *rep_n;
    const float *rep_s0, *rep_w, *ip;
    double *partial;              // instance i's columns at partial + part_off[i]
    const int64_t *part_off;
};
cudaError_t fft_cols_mask_b(const FftClassSet &q, const ColsBatch &a, bool kderiv, cudaStream_t s);
// The weights-on-a-grid form of the two kernels (fresco_uwu_*): the columns with that form's mask
// (a.partial [2 (kx + 1)]; scal: rho0 in, loss and F out at 2 and 3), and the rows back less (4 F /
// rho0) c.
cudaError_t fft_cols_weights(const FftDesc &f, const ColsArgs &a, double loss_const, double *scal,
                             double *loss, unsigned *done, cudaStream_t s);
cudaError_t fft_rows_inverse_w(const FftDesc &f, const float2 *bt, float *grad, const float2 *tws,
                               int64_t rows, int kx, const float *c, const double *scal,
                               cudaStream_t s);
// the column spectra themselves: out[k][row] = forward transform of xt[k] along y
cudaError_t fft_cols_spectrum(const FftDesc &f, const float2 *xt, float2 *out, int kx,
                              cudaStream_t s);
// whether a column (with its scratch) fits a block
bool fft_cols_fit(const FftDesc &f, bool kderiv);
// allow the kernels their shared memory (once per process and device)
cudaError_t fft_allow_smem();

// The transforms of one fine grid: x rows as complex rows of half the length, complex rows of the
// direct mode's inverse, and 2D columns.
struct FftSet {
    FftDesc x, xc, y;
    bool fwd = false, inv = false, cols = false;   // which steps run here
    int *rep_first = nullptr;                      // single plans, [kx + 2]
    std::vector<void *> allocs;
    int64_t bytes = 0;
};
// Chooses and builds the transforms of an FP32 grid, `rows` rows to a launch; steps whose lengths do
// not fit keep cuFFT, and, unless `always`, all of a 2D grid on which cuFFT's are the faster ones.
fresco_status fft_set_build(FftSet &f, const int nf[3], int dim, bool kderiv, int64_t rows,
                            bool always);
// Whether an FP32 ensemble of `cells` fine-grid cells in all, in so many size classes, runs these
// transforms: they save the library form's launches, six and more for every class, and cost more per
// cell (the direct mode's above all, with two columns and complex rows back). Measured on GB300,
// transforms and mask, cuFFT / these kernels (us). kderiv: one class of 4.2e6 cells 58 / 55, 9.4e6
// (3072^2) 129 / 111, 1.7e7 (16 grids of 1024^2) 127 / 146, 6.7e7 (64 of 1024^2) 434 / 515; two of 2.7e7
// together 265 / 263, 8.2e7 689 / 729; four of 6.8e7 566 / 556, 2.0e8 1378 / 1590; nine of 1.6e7
// 427 / 160, 9.6e7 1003 / 804, 2.0e8 1824 / 1608. Direct: one class of 2.4e6 73 / 71, 4.2e6 (four of
// 1024^2) 76 / 82, 6.7e7 573 / 830; two of 1.1e7 224 / 181, 1.3e7 215 / 225; four of 1.7e7 303 / 241,
// 3.3e7 496 / 546; nine of 5.2e7 852 / 720, 9.6e7 1330 / 1313, 1.1e8 1398 / 1637. Over 80 ensembles of
// both modes the form not taken is at most 1.02 (kderiv) and 1.04 (direct) times as fast as a whole.
inline bool fft_ensemble_pays(double cells, int classes, bool kderiv) {
    return cells <= (kderiv ? 2.4e7 * classes - 1.4e7 : 6.65e6 * classes - 2.65e6);
}
void fft_set_free(FftSet *f);
// first[k] = index of the first representative with n_x >= k, k = 0 .. kx + 1 (rep_n is n_x major)
std::vector<int> rep_columns(const std::vector<int32_t> &rep_n, int dim, int kx);

}  // namespace fresco
