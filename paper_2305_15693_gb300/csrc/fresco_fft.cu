// Transforms of the FP32 fine grids, fused with the steps around them.
//
// With library transforms an evaluation moves the grid through memory once per step: the x pass,
// the split into half spectra with the transpose, the y pass, the mask, the y pass back, the merge
// and transpose, the x pass back: fourteen reads or writes of (part of) the grid and seven launches
// and more. Here they are three kernels that read and write it once each:
//   k_fft_rows_fwd   real rows in, the needed columns of their half spectra out, transposed;
//   k_fft_cols       a column in; along y forward, the mask (S, loss, gradient coefficients), along
//                    y back; a column out;
//   k_fft_rows_inv   columns in, real rows out (k_fft_rows_inv_c: complex rows, the direct mode).
// A block holds its rows (or its column) in shared memory and runs the passes in place
// (fresco_fft.cuh).
//
// What bounds them: shared-memory passes and instruction issue at about equal parts (three or four
// passes, each element read and written once per pass), with the global reads and writes in
// between (fft_set_build has what they measured against cuFFT and where the line lies).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fresco_fft.cuh"
#include "fresco_kernels.cuh"

namespace fresco {

using namespace fft_detail;

namespace {

// Rows r0 .. of one grid, f.rows of them, in each of the next three; rows: the grid's.
__device__ __forceinline__ void rows_fwd(const FftDesc &f, const float *__restrict__ grid,
                                         float2 *__restrict__ xt, const float2 *__restrict__ tws,
                                         int64_t rows, int64_t r0, int kx) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    const int M = f.n, pitch = f.words;
    const int nr = (int)min((int64_t)f.rows, rows - r0);
    const float2 *in = reinterpret_cast<const float2 *>(grid) + r0 * M;
    xt += r0;
    fft_forward(f, nr, s, pitch, [&](int row, int i) { return in[(int64_t)row * M + i]; });
    // X[k] = E + tau_k O and X[M - k] = conj(E - tau_k O) from Z[k], Z[M - k] (as k_rfft_split_cols)
    const int half = M / 2, shift = __popc(f.rows - 1);   // f.rows is a power of two
    for (int t = threadIdx.x; t < (half + 1) << shift; t += blockDim.x) {
        const int row = t & (f.rows - 1), k = t >> shift;
        const int km = M - k;
        if (row >= nr || (k > kx && km > kx)) continue;
        const float2 a = s[row * pitch + fft_place(f, __ldg(f.pos + k))];
        const float2 b = s[row * pitch + fft_place(f, __ldg(f.pos + (k == 0 ? 0 : km)))];
        const float2 w = __ldg(tws + k);
        const float ex = 0.5f * (a.x + b.x), ey = 0.5f * (a.y - b.y);
        const float ox = 0.5f * (a.y + b.y), oy = -0.5f * (a.x - b.x);
        const float px = w.x * ox - w.y * oy, py = w.x * oy + w.y * ox;
        if (k <= kx) xt[(int64_t)k * rows + row] = {ex + px, ey + py};
        if (km > half && km <= kx) xt[(int64_t)km * rows + row] = {ex - px, -(ey - py)};
    }
}

// WEIGHTS: the result less (4 F / rho0) c, c the weights on the same grid and scal[0] = rho0, scal[3]
// = F (the weight gradient's second term). PAIRS: grid lies on an 8-byte boundary (the plans' own grids
// do; a caller's gradient need not).
template <bool WEIGHTS, bool PAIRS>
__device__ __forceinline__ void rows_inv(const FftDesc &f, const float2 *__restrict__ bt,
                                         float *__restrict__ grid, const float2 *__restrict__ tws,
                                         int64_t rows, int64_t r0, int kx,
                                         const float *__restrict__ c,
                                         const double *__restrict__ scal) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    const int M = f.n, pitch = f.words;
    const int nr = (int)min((int64_t)f.rows, rows - r0);
    bt += r0;
    float *out = grid + 2 * r0 * M;
    auto store = [&](int row, int i, float2 v) {
        float *p = out + 2 * ((int64_t)row * M + i);
        if constexpr (PAIRS) {
            *reinterpret_cast<float2 *>(p) = v;
        } else {
            p[0] = v.x;
            p[1] = v.y;
        }
    };
    // Z[k] = P + i Q, Z[M - k] = conj P + i conj Q (as k_rfft_merge_rows), parts exchanged
    const int half = M / 2, shift = __popc(f.rows - 1);
    for (int t = threadIdx.x; t < (half + 1) << shift; t += blockDim.x) {
        const int row = t & (f.rows - 1), k = t >> shift;
        if (row >= nr) continue;
        const int km = M - k;
        float2 a = {0.f, 0.f}, b = {0.f, 0.f};
        if (k <= kx) a = bt[(int64_t)k * rows + row];
        if (km <= kx) b = bt[(int64_t)km * rows + row];
        const float2 w = __ldg(tws + k);
        const float px = a.x + b.x, py = a.y - b.y;
        const float dx = a.x - b.x, dy = a.y + b.y;
        const float qx = dx * w.x + dy * w.y, qy = dy * w.x - dx * w.y;
        s[row * pitch + fft_place(f, __ldg(f.pos + k))] = {py + qx, px - qy};
        if (km > half && km < M) s[row * pitch + fft_place(f, __ldg(f.pos + km))] = {-py + qx, px + qy};
    }
    __syncthreads();
    if constexpr (WEIGHTS) {
        const float coef = (float)(4.0 * scal[3] / scal[0]);
        const float2 *cr = reinterpret_cast<const float2 *>(c) + r0 * M;
        fft_adjoint(f, nr, s, pitch, [&](int row, int i, float2 v) {
            const float2 w = cr[(int64_t)row * M + i];
            store(row, i, {v.y - coef * w.x, v.x - coef * w.y});
        });
    } else {
        fft_adjoint(f, nr, s, pitch, [&](int row, int i, float2 v) { store(row, i, {v.y, v.x}); });
    }
}

__device__ __forceinline__ void rows_inv_c(const FftDesc &f, const float2 *__restrict__ bt,
                                           float2 *__restrict__ g, int64_t rows, int64_t r0,
                                           int kx) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    const int n = f.n, pitch = f.words;
    const int nr = (int)min((int64_t)f.rows, rows - r0);
    bt += r0;
    g += r0 * n;
    const int shift = __popc(f.rows - 1), ncol = 2 * kx + 2;
    for (int t = threadIdx.x; t < n << shift; t += blockDim.x) {
        const int row = t & (f.rows - 1), x = t >> shift;
        if (row >= nr) continue;
        // x = n_x modulo n; n_x = c - kx - 1
        const int c = x <= kx ? x + kx + 1 : x - (n - kx - 1);
        float2 v = {0.f, 0.f};
        if (c >= 0 && c < ncol) v = bt[(int64_t)c * rows + row];
        s[row * pitch + fft_place(f, __ldg(f.pos + x))] = {v.y, v.x};
    }
    __syncthreads();
    fft_adjoint(f, nr, s, pitch,
                [&](int row, int i, float2 v) { g[(int64_t)row * n + i] = {v.y, v.x}; });
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_fwd(const __grid_constant__ FftDesc f, const float *__restrict__ grid,
                   float2 *__restrict__ xt, const float2 *__restrict__ tws, int64_t rows, int kx) {
    rows_fwd(f, grid, xt, tws, rows, (int64_t)blockIdx.x * f.rows, kx);
}

template <bool WEIGHTS, bool PAIRS>
__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_inv(const __grid_constant__ FftDesc f, const float2 *__restrict__ bt,
                   float *__restrict__ grid, const float2 *__restrict__ tws, int64_t rows, int kx,
                   const float *__restrict__ c, const double *__restrict__ scal) {
    rows_inv<WEIGHTS, PAIRS>(f, bt, grid, tws, rows, (int64_t)blockIdx.x * f.rows, kx, c, scal);
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_inv_c(const __grid_constant__ FftDesc f, const float2 *__restrict__ bt,
                     float2 *__restrict__ g, int64_t rows, int kx) {
    rows_inv_c(f, bt, g, rows, (int64_t)blockIdx.x * f.rows, kx);
}

// The size classes of an ensemble in one launch: a class's blocks alone leave most SMs idle and each
// launch waits for the last of the one before. An ensemble of 128 in nine classes: 27 launches of 4
// to 36 us, 323 us in all, now three of 52, 65 and 57.
__device__ __forceinline__ int class_of(const FftClassSet &q, int &block) {
    int i = 0;
    while (i + 1 < q.n && (int)blockIdx.x >= q.first[i + 1]) ++i;
    block = (int)blockIdx.x - q.first[i];
    return i;
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_fwd_b(const __grid_constant__ FftClassSet q, const float *__restrict__ grid,
                     float2 *__restrict__ xt, const float2 *__restrict__ tws) {
    int b;
    const FftClass &c = q.c[class_of(q, b)];
    const int z = b / c.blocks;
    rows_fwd(c.f, grid + c.in0 + z * c.in_stride, xt + c.out0 + z * c.out_stride, tws + c.tw0,
             c.rows, (int64_t)(b - z * c.blocks) * c.f.rows, c.kx);
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_inv_b(const __grid_constant__ FftClassSet q, const float2 *__restrict__ bt,
                     float *__restrict__ grid, const float2 *__restrict__ tws) {
    int b;
    const FftClass &c = q.c[class_of(q, b)];
    const int z = b / c.blocks;
    rows_inv<false, true>(c.f, bt + c.in0 + z * c.in_stride, grid + c.out0 + z * c.out_stride,
                          tws + c.tw0, c.rows, (int64_t)(b - z * c.blocks) * c.f.rows, c.kx,
                          nullptr, nullptr);
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_rows_inv_cb(const __grid_constant__ FftClassSet q, const float2 *__restrict__ bt,
                      float2 *__restrict__ g) {
    int b;
    const FftClass &c = q.c[class_of(q, b)];
    const int z = b / c.blocks;
    rows_inv_c(c.f, bt + c.in0 + z * c.in_stride, g + c.out0 + z * c.out_stride, c.rows,
               (int64_t)(b - z * c.blocks) * c.f.rows, c.kx);
}

// One column of the 2D problem (see k_mask for the mask's arithmetic; the thread's loss terms are an
// exact float pair). Returns the thread's loss sum.
template <bool KD>
__device__ __forceinline__ double cols_column(const FftDesc &f, const MaskGeom &m, int k,
                                              const float2 *__restrict__ in, float2 *__restrict__ bt,
                                              const int *__restrict__ rep_n,
                                              const float *__restrict__ rep_s0,
                                              const float *__restrict__ rep_w, int e0, int e1,
                                              const float *__restrict__ ip0,
                                              const float *__restrict__ ip1) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int n = f.n, words = f.words, nbit = (words + 31) / 32;
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    float2 *t = s + words;                                        // direct mode only
    unsigned *bits = reinterpret_cast<unsigned *>(s + (KD ? 1 : 2) * words);
    for (int i = threadIdx.x; i < nbit; i += blockDim.x) bits[i] = 0;
    fft_forward(f, 1, s, 0, [&](int, int i) { return in[i]; });
    const float inv_n = (float)m.inv_n, ipx = ip0[k];
    float ah = 0.f, al = 0.f;
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        const int ny = rep_n[2 * e + 1];
        const int ry = ny < 0 ? ny + n : ny;
        const int p = fft_place(f, __ldg(f.pos + ry));
        const float2 F = s[p];
        const float ip = ipx * ip1[ny < 0 ? -ny : ny];
        const float re = F.x * ip, im = F.y * ip;
        const float S = (re * re + im * im) * inv_n;
        const float wgt = rep_w[e];
        float dh, dl;
        two_sum(S, -rep_s0[e], dh, dl);
        const float pr = dh * dh;
        const float pl = fmaf(2.f * dh, dl, fmaf(dh, dh, -pr));
        const float th = wgt * pr;
        const float tl = fmaf(wgt, pl, fmaf(wgt, pr, -th));
        float sh, se;
        two_sum(ah, th, sh, se);
        ah = sh;
        al += se + tl;
        const float E = 4.f * wgt * dh * inv_n;
        const float h = 0.5f * ip * E;
        const float er = re * h, ei = im * h;
        // kderiv: the scalar E / Psi with its parts exchanged; direct: kept for both columns
        s[p] = KD ? float2{ei, er} : float2{er, ei};
        atomicOr(&bits[p >> 5], 1u << (p & 31));
        if (KD && k == 0) {   // the conjugate at -n, which the real inverse along x reads
            const int p2 = fft_place(f, __ldg(f.pos + (ny > 0 ? n - ny : -ny)));
            s[p2] = {-ei, er};
            atomicOr(&bits[p2 >> 5], 1u << (p2 & 31));
        }
    }
    __syncthreads();
    if constexpr (KD) {
        for (int i = threadIdx.x; i < words; i += blockDim.x)
            if (!(bits[i >> 5] >> (i & 31) & 1)) s[i] = {0.f, 0.f};
        __syncthreads();
        float2 *out = bt + (int64_t)k * n;
        fft_adjoint(f, 1, s, 0, [&](int, int i, float2 v) { out[i] = {v.y, v.x}; });
    } else {
        // H[n] = (a_x + i a_y) ip / 2 at n and at -n (columns n_x = k and -k)
        const float kxs = (float)(m.kscale[0] * k);
#pragma unroll 1
        for (int side = 0; side < (k ? 2 : 1); ++side) {
            for (int i = threadIdx.x; i < words; i += blockDim.x) t[i] = {0.f, 0.f};
            __syncthreads();
            for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
                const int ny = rep_n[2 * e + 1];
                const int p = fft_place(f, __ldg(f.pos + (ny < 0 ? ny + n : ny)));
                const int p2 = fft_place(f, __ldg(f.pos + (ny > 0 ? n - ny : -ny)));
                const float er = s[p].x, ei = s[p].y, ky = (float)(m.kscale[1] * ny);
                if (side == 0) t[p] = {er * kxs - ei * ky, -er * ky - ei * kxs};
                if (side == 1 || k == 0) t[p2] = {-er * kxs - ei * ky, er * ky - ei * kxs};
            }
            __syncthreads();
            float2 *out = bt + (int64_t)((side ? -k : k) + m.kx + 1) * n;
            fft_adjoint(f, 1, t, 0, [&](int, int i, float2 v) { out[i] = {v.y, v.x}; });
            __syncthreads();
        }
    }
    return (double)ah + (double)al;
}

template <bool KD>
__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_cols(const __grid_constant__ FftDesc f, const __grid_constant__ ColsArgs a,
               double loss_const, double *__restrict__ loss, unsigned *__restrict__ done) {
    __shared__ bool s_last;
    const int k = blockIdx.x, e0 = a.rep_first[k], e1 = a.rep_first[k + 1];
    // (a column without representatives stays zero from plan time)
    const double l = e0 == e1 ? 0.0
                              : cols_column<KD>(f, a.m, k, a.xt + (int64_t)k * f.n, a.bt, a.rep_n,
                                                a.rep_s0, a.rep_w, e0, e1, a.ip0, a.ip1);
    const double b = block_sum(l);
    if (threadIdx.x == 0) {
        a.partial[k] = b;
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // the block that finishes last adds the columns' sums in a fixed order
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) v += __ldcg(a.partial + i);
    const double t = block_sum(v);
    if (threadIdx.x == 0) {
        *loss = t + loss_const;
        *done = 0;
    }
}

template <bool KD>
__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_cols_b(const __grid_constant__ FftClassSet q, const __grid_constant__ ColsBatch a) {
    int b0;
    const FftClass &c = q.c[class_of(q, b0)];
    const int z = b0 / c.blocks, i = a.list[c.list0 + z], k = b0 - z * c.blocks;
    const BInst &I = a.inst[i];
    const int *first = a.rep_first + a.rep_off[i];
    const int e0 = first[k], e1 = first[k + 1];
    const double l =
        e0 == e1 ? 0.0
                 : cols_column<KD>(c.f, I.m, k, a.xt + I.ato + (int64_t)k * c.f.n, a.bt + I.hco,
                                   a.rep_n + 2 * I.reo, a.rep_s0 + I.reo, a.rep_w + I.reo, e0, e1,
                                   a.ip + I.ipo[0], a.ip + I.ipo[1]);
    const double b = block_sum(l);
    if (threadIdx.x == 0) a.partial[a.part_off[i] + k] = b;
}

// The columns of the weights-on-a-grid form (exact transforms, no kernel): S = |rho|^2 / rho0, the
// loss and F = sum W S (S - S0), and (E / 2) rho, E = 4 W (S - S0) / rho0, back along y. Both sums
// run in FP64 term by term, as in the cuFFT form (k_uwu_mask). scal[0] = rho0 on entry; the last
// block leaves the loss (and its constant) in scal[2] and *loss, F in scal[3].
__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_cols_w(const __grid_constant__ FftDesc f, const __grid_constant__ ColsArgs a,
                 double loss_const, double *__restrict__ scal, double *__restrict__ loss,
                 unsigned *__restrict__ done) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ bool s_last;
    const int n = f.n, words = f.words, nbit = (words + 31) / 32, k = blockIdx.x;
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    unsigned *bits = reinterpret_cast<unsigned *>(s + words);
    const int e0 = a.rep_first[k], e1 = a.rep_first[k + 1];
    double bl = 0.0, bf = 0.0;
    if (e0 != e1) {   // (a column without representatives stays zero from plan time)
        for (int i = threadIdx.x; i < nbit; i += blockDim.x) bits[i] = 0;
        const float2 *in = a.xt + (int64_t)k * n;
        fft_forward(f, 1, s, 0, [&](int, int i) { return in[i]; });
        const double inv_rho0 = 1.0 / scal[0];
        const float inv = (float)inv_rho0;
        for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
            const int ny = a.rep_n[2 * e + 1];
            const int p = fft_place(f, __ldg(f.pos + (ny < 0 ? ny + n : ny)));
            const float2 F = s[p];
            const float S = (F.x * F.x + F.y * F.y) * inv;
            const double w = (double)a.rep_w[e], d = (double)S - (double)a.rep_s0[e];
            bl = fma(w * d, d, bl);
            bf = fma(w * (double)S, d, bf);
            const float h = (float)(2.0 * w * d * inv_rho0);
            s[p] = {h * F.y, h * F.x};   // parts exchanged for the inverse
            atomicOr(&bits[p >> 5], 1u << (p & 31));
            if (k == 0) {
                const int p2 = fft_place(f, __ldg(f.pos + (ny > 0 ? n - ny : -ny)));
                s[p2] = {-h * F.y, h * F.x};
                atomicOr(&bits[p2 >> 5], 1u << (p2 & 31));
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < words; i += blockDim.x)
            if (!(bits[i >> 5] >> (i & 31) & 1)) s[i] = {0.f, 0.f};
        __syncthreads();
        float2 *out = a.bt + (int64_t)k * n;
        fft_adjoint(f, 1, s, 0, [&](int, int i, float2 v) { out[i] = {v.y, v.x}; });
        bl = block_sum(bl);
        bf = block_sum(bf);
    }
    if (threadIdx.x == 0) {
        a.partial[k] = bl;
        a.partial[gridDim.x + k] = bf;
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double v = 0.0, u = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        v += __ldcg(a.partial + i);
        u += __ldcg(a.partial + gridDim.x + i);
    }
    v = block_sum(v);
    u = block_sum(u);
    if (threadIdx.x == 0) {
        scal[2] = v + loss_const;
        scal[3] = u;
        *loss = v + loss_const;
        *done = 0;
    }
}

__global__ void __launch_bounds__(kFftThreads, kFftBlocks)
    k_fft_cols_spec(const __grid_constant__ FftDesc f, const float2 *xt, float2 *out) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    float2 *s = reinterpret_cast<float2 *>(sm_raw);
    const float2 *in = xt + (int64_t)blockIdx.x * f.n;
    fft_forward(f, 1, s, 0, [&](int, int i) { return in[i]; });
    for (int i = threadIdx.x; i < f.n; i += blockDim.x)
        out[(int64_t)blockIdx.x * f.n + i] = s[fft_place(f, __ldg(f.pos + i))];
}

}  // namespace

// Radices, and the arithmetic of a butterfly with its twiddles per element (instructions, counted
// from the code).
constexpr int kRadix[] = {10, 9, 8, 7, 6, 5, 4, 3, 2};
static double radix_cost(int r) {
    switch (r) {
        case 2: return 6.0;
        case 3: return 12.0;
        case 4: return 10.0;
        case 5: return 15.0;
        case 7: return 21.0;
        case 8: return 14.5;
        default: return 9.0 + 1.0 * r;
    }
}

// Shared-memory wavefronts per element and pass, read and write, of pass p with the padding shift
// given: the first warps' accesses (64-bit: half a warp at a time over 16 pairs of banks).
static double pass_wavefronts(const FftDesc &f, int p, int shift) {
    const int r = f.r[p], m = f.m[p], nb = f.n / r;
    double waves = 0.0;
    int groups = 0;
    for (int i0 = 0; i0 < std::min(nb, 128); i0 += 16) {
        int hit[16] = {}, most = 0;
        for (int i = i0; i < std::min(nb, i0 + 16); ++i) {
            const int a = i / m * m * r + i % m;
            most = std::max(most, ++hit[(a + (a >> shift)) & 15]);
        }
        waves += most;
        ++groups;
    }
    return waves / groups;
}

static void set_radices(FftDesc &f, const std::vector<int> &r) {
    f.np = (int)r.size();
    int len = f.n;
    for (int p = 0; p < f.np; ++p) {
        f.r[p] = r[(size_t)p];
        f.m[p] = len / f.r[p];
        len = f.m[p];
    }
}

// The factorisation with the least arithmetic, in the order and with the padding that meet the
// fewest bank conflicts.
bool fft_describe(int n, FftDesc &f) {
    f = FftDesc();
    f.n = n;
    if (n < 2 || sizeof(float2) * (size_t)n > kFftSmem) return false;
    std::vector<int> best, cur;
    double best_cost = 1e300;
    // (descending radices: every multiset once)
    auto search = [&](auto &&self, int rest, int from, double cost) -> void {
        if (cost >= best_cost || (int)cur.size() > kFftMaxPasses) return;
        if (rest == 1) {
            best = cur;
            best_cost = cost;
            return;
        }
        for (int i = from; i < (int)(sizeof(kRadix) / sizeof(kRadix[0])); ++i)
            if (rest % kRadix[i] == 0) {
                cur.push_back(kRadix[i]);
                self(self, rest / kRadix[i], i, cost + radix_cost(kRadix[i]) + 10.0);
                cur.pop_back();
            }
    };
    search(search, n, 0, 0.0);
    if (best.empty() || (int)best.size() > kFftMaxPasses) return false;
    std::sort(best.begin(), best.end());
    std::vector<int> order;
    int shift = 31;
    double waves = 1e300;
    int tried = 0;
    do {
        set_radices(f, best);
        for (int s : {31, 4, 3, 5}) {
            if (sizeof(float2) * (size_t)(n + (n >> s) + 1) > kFftSmem) continue;
            double w = s == 31 ? 0.0 : 0.2 * f.np;   // (the padding's own arithmetic)
            for (int p = 0; p < f.np; ++p) w += pass_wavefronts(f, p, s);
            if (w < waves - 1e-9) {
                waves = w;
                order = best;
                shift = s;
            }
        }
    } while (std::next_permutation(best.begin(), best.end()) && ++tried < 120);
    if (order.empty()) return false;
    set_radices(f, order);
    for (int p = 0; p < f.np; ++p) {
        f.dm[p] = FastDiv(f.m[p]);
        f.db[p] = FastDiv(n / f.r[p]);
    }
    f.shift = shift;
    f.words = n + (n >> shift) + 1;
    if (!(f.words & 1)) ++f.words;   // rows of a block start in different banks
    return sizeof(float2) * (size_t)f.words <= kFftSmem;
}

fresco_status fft_tables(FftDesc &f, std::vector<void *> &allocs, int64_t &bytes) {
    std::vector<float2> tw((size_t)f.n);
    std::vector<int> pos((size_t)f.n);
    for (int k = 0; k < f.n; ++k) {
        const double a = 2.0 * M_PI * (double)k / (double)f.n;
        tw[(size_t)k] = make_float2((float)std::cos(a), (float)-std::sin(a));
        int rest = k, at = 0;
        for (int p = 0; p < f.np; ++p) {
            at += rest % f.r[p] * f.m[p];
            rest /= f.r[p];
        }
        pos[(size_t)k] = at;
    }
    void *d[2] = {nullptr, nullptr};
    const size_t b[2] = {sizeof(float2) * tw.size(), sizeof(int) * pos.size()};
    const void *h[2] = {tw.data(), pos.data()};
    for (int i = 0; i < 2; ++i) {
        if (cudaMalloc(&d[i], b[i]) != cudaSuccess) {
            cudaGetLastError();
            return FRESCO_ERR_OOM;
        }
        allocs.push_back(d[i]);
        bytes += (int64_t)b[i];
        if (cudaMemcpy(d[i], h[i], b[i], cudaMemcpyHostToDevice) != cudaSuccess)
            return FRESCO_ERR_CUDA;
    }
    f.tw = (const float2 *)d[0];
    f.pos = (const int *)d[1];
    return FRESCO_OK;
}

// Steps x threads of the passes of `rows` transforms (idle lanes included), fewer threads dearer where
// it is close.
static double thread_cost(const FftDesc &f, int rows, int t) {
    double cost = 0.0;
    for (int p = 0; p < f.np; ++p) {
        const int nb = rows * (f.n / f.r[p]);
        cost += (double)((nb + t - 1) / t) * t * f.r[p];
    }
    return cost * (1.0 + 0.25 * 64.0 / t);
}

// the number of threads (a multiple of 32, from 64) of least cost
template <class Cost>
static int least_threads(Cost cost) {
    int best = 64;
    double best_cost = 1e300;
    for (int t = 64; t <= kFftThreads; t += 32) {
        const double c = cost(t);
        if (c < best_cost) {
            best_cost = c;
            best = t;
        }
    }
    return best;
}
static int fft_threads(const FftDesc &f, int rows) {
    return least_threads([&](int t) { return thread_cost(f, rows, t); });
}

void fft_size_rows(FftDesc &f, int64_t rows) {
    // rows per block: up to sixteen (a column's write is then whole 32-byte sectors from four on)
    // while kFftBlocks blocks fit an SM and every SM has two
    f.rows = 1;
    while (f.rows < 16 && fft_bytes(f, 2 * f.rows) * kFftBlocks <= kFftSmem &&
           rows / (2 * f.rows) >= 2 * 152)
        f.rows *= 2;
    f.threads = fft_threads(f, f.rows);
}

void fft_size_cols(FftDesc &f) {
    f.rows = 1;
    f.threads = fft_threads(f, 1);
}

static size_t cols_bytes(const FftDesc &f, int buffers) {
    const int words = f.words;
    return sizeof(float2) * (size_t)buffers * words + 4 * (size_t)((words + 31) / 32);
}

cudaError_t fft_allow_smem() {
    const int b = (int)kFftSmem;
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(k_fft_rows_fwd, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv<false, true>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv<true, true>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv<true, false>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols_w, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv_c, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols<true>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols<false>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_fwd_b, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv_b, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_rows_inv_cb, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols_b<true>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols_b<false>, attr, b);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fft_cols_spec, attr, b);
    return e;
}

bool fft_cols_fit(const FftDesc &f, bool kderiv) {
    return cols_bytes(f, kderiv ? 1 : 2) <= kFftSmem;
}

constexpr double kOwnCells = 1.2e6;
constexpr int kOwnRow = 9000;

fresco_status fft_set_build(FftSet &f, const int nf[3], int dim, bool kderiv, int64_t rows,
                            bool always) {
    // 2D single grids beyond kOwnCells stay on cuFFT, whose larger radices then outweigh its extra
    // passes over memory; ensembles (fft_ensemble_pays) and the 3D rows have rules of their own.
    // Measured, x passes, y passes and mask, cuFFT against these kernels (us): 432^2 46 / 36, 784^2
    // 53 / 38, 2500^2 95 / 109, 6480^2 448 / 471; the 324^3 grid's x passes with cuFFT's (z, y)
    // transforms 468 / 374. So do grids of few rows longer than kOwnRow, each of which one block
    // transforms by itself: 8064 x 14 48 / 47, 12096 x 14 51 / 67, 16128 x 42 57 / 81
    if (dim == 2 && !always && ((double)nf[0] * nf[1] > kOwnCells || nf[0] > kOwnRow))
        return FRESCO_OK;
    // (the kernels work on whole rows of nf[0] floats; nf[0] is even)
    f.fwd = fft_describe(nf[0] / 2, f.x);
    f.inv = kderiv ? f.fwd : fft_describe(nf[0], f.xc);
    f.cols = dim == 2 && f.fwd && f.inv && fft_describe(nf[1], f.y) && fft_cols_fit(f.y, kderiv);
    if (!f.fwd && !f.inv) return FRESCO_OK;
    if (fft_allow_smem() != cudaSuccess) return FRESCO_ERR_CUDA;
    fresco_status st = FRESCO_OK;
    if (f.fwd) {
        fft_size_rows(f.x, rows);
        st = fft_tables(f.x, f.allocs, f.bytes);
    }
    if (!st && f.inv && !kderiv) {
        fft_size_rows(f.xc, rows);
        st = fft_tables(f.xc, f.allocs, f.bytes);
    }
    if (!st && f.cols) {
        fft_size_cols(f.y);
        st = fft_tables(f.y, f.allocs, f.bytes);
    }
    return st;
}

void fft_set_free(FftSet *f) {
    if (!f) return;
    for (void *p : f->allocs) cudaFree(p);
    delete f;
}

std::vector<int> rep_columns(const std::vector<int32_t> &rep_n, int dim, int kx) {
    std::vector<int> first((size_t)kx + 2, 0);
    const size_t n = rep_n.size() / (size_t)dim;
    size_t e = 0;
    for (int k = 0; k <= kx + 1; ++k) {
        while (e < n && rep_n[e * (size_t)dim] < k) ++e;
        first[(size_t)k] = (int)e;
    }
    return first;
}

cudaError_t fft_rows_forward(const FftDesc &f, const float *grid, float2 *xt, const float2 *tws,
                             int64_t rows, int kx, cudaStream_t s) {
    k_fft_rows_fwd<<<(unsigned)((rows + f.rows - 1) / f.rows), f.threads, fft_bytes(f, f.rows), s>>>(
        f, grid, xt, tws, rows, kx);
    return cudaGetLastError();
}

cudaError_t fft_rows_inverse(const FftDesc &f, const float2 *bt, float *grid, const float2 *tws,
                             int64_t rows, int kx, cudaStream_t s) {
    k_fft_rows_inv<false, true><<<(unsigned)((rows + f.rows - 1) / f.rows), f.threads,
                                  fft_bytes(f, f.rows), s>>>(f, bt, grid, tws, rows, kx, nullptr,
                                                             nullptr);
    return cudaGetLastError();
}

cudaError_t fft_rows_inverse_w(const FftDesc &f, const float2 *bt, float *grad, const float2 *tws,
                               int64_t rows, int kx, const float *c, const double *scal,
                               cudaStream_t s) {
    const auto kern = (uintptr_t)grad % sizeof(float2) ? k_fft_rows_inv<true, false>
                                                       : k_fft_rows_inv<true, true>;
    kern<<<(unsigned)((rows + f.rows - 1) / f.rows), f.threads, fft_bytes(f, f.rows), s>>>(
        f, bt, grad, tws, rows, kx, c, scal);
    return cudaGetLastError();
}

cudaError_t fft_cols_weights(const FftDesc &f, const ColsArgs &a, double loss_const, double *scal,
                             double *loss, unsigned *done, cudaStream_t s) {
    k_fft_cols_w<<<(unsigned)(a.m.kx + 1), f.threads, cols_bytes(f, 1), s>>>(f, a, loss_const, scal,
                                                                             loss, done);
    return cudaGetLastError();
}

cudaError_t fft_rows_inverse_c(const FftDesc &f, const float2 *bt, float2 *g, int64_t rows, int kx,
                               cudaStream_t s) {
    k_fft_rows_inv_c<<<(unsigned)((rows + f.rows - 1) / f.rows), f.threads, fft_bytes(f, f.rows),
                       s>>>(f, bt, g, rows, kx);
    return cudaGetLastError();
}

cudaError_t fft_cols_mask(const FftDesc &f, const ColsArgs &a, double loss_const, double *loss,
                          unsigned *done, cudaStream_t s) {
    const unsigned cols = (unsigned)(a.m.kx + 1);
    if (a.m.kderiv)
        k_fft_cols<true><<<cols, f.threads, cols_bytes(f, 1), s>>>(f, a, loss_const, loss, done);
    else
        k_fft_cols<false><<<cols, f.threads, cols_bytes(f, 2), s>>>(f, a, loss_const, loss, done);
    return cudaGetLastError();
}

std::vector<FftClassSet> fft_class_sets(std::vector<FftClass> cls, int col_buffers) {
    auto bytes = [&](const FftClass &c) {
        return col_buffers ? cols_bytes(c.f, col_buffers) : fft_bytes(c.f, c.f.rows);
    };
    // the blocks that take longest first
    std::stable_sort(cls.begin(), cls.end(), [&](const FftClass &a, const FftClass &b) {
        return bytes(a) > bytes(b);
    });
    std::vector<FftClassSet> out;
    for (const FftClass &c : cls) {
        // a class whose blocks need much less shared memory than those that set a launch's residency
        // (below kFftBlocks) starts another launch
        const bool apart = !out.empty() && out.back().smem * kFftBlocks > kFftSmem &&
                           2 * bytes(c) <= out.back().smem;
        const int64_t blocks = (int64_t)c.blocks * c.count;
        if (out.empty() || out.back().n == kFftClasses || apart ||
            out.back().first[out.back().n] + blocks > 2147483647LL) {
            out.emplace_back();
            out.back().smem = bytes(c);
        }
        FftClassSet &q = out.back();
        q.c[q.n] = c;
        q.first[q.n + 1] = (int)(q.first[q.n] + blocks);
        ++q.n;
    }
    for (FftClassSet &q : out)
        q.threads = least_threads([&](int t) {
            double cost = 0.0;
            for (int i = 0; i < q.n; ++i)
                cost += (double)q.c[i].blocks * q.c[i].count *
                        thread_cost(q.c[i].f, q.c[i].f.rows, t);
            return cost;
        });
    return out;
}

cudaError_t fft_rows_forward_b(const FftClassSet &q, const float *grid, float2 *xt,
                               const float2 *tws, cudaStream_t s) {
    k_fft_rows_fwd_b<<<(unsigned)q.first[q.n], q.threads, q.smem, s>>>(q, grid, xt, tws);
    return cudaGetLastError();
}

cudaError_t fft_rows_inverse_b(const FftClassSet &q, const float2 *bt, float *grid,
                               const float2 *tws, cudaStream_t s) {
    k_fft_rows_inv_b<<<(unsigned)q.first[q.n], q.threads, q.smem, s>>>(q, bt, grid, tws);
    return cudaGetLastError();
}

cudaError_t fft_rows_inverse_cb(const FftClassSet &q, const float2 *bt, float2 *g, cudaStream_t s) {
    k_fft_rows_inv_cb<<<(unsigned)q.first[q.n], q.threads, q.smem, s>>>(q, bt, g);
    return cudaGetLastError();
}

cudaError_t fft_cols_mask_b(const FftClassSet &q, const ColsBatch &a, bool kderiv, cudaStream_t s) {
    const unsigned g = (unsigned)q.first[q.n];
    if (kderiv) k_fft_cols_b<true><<<g, q.threads, q.smem, s>>>(q, a);
    else k_fft_cols_b<false><<<g, q.threads, q.smem, s>>>(q, a);
    return cudaGetLastError();
}

cudaError_t fft_cols_spectrum(const FftDesc &f, const float2 *xt, float2 *out, int kx,
                              cudaStream_t s) {
    k_fft_cols_spec<<<(unsigned)(kx + 1), f.threads, fft_bytes(f, 1), s>>>(f, xt, out);
    return cudaGetLastError();
}

}  // namespace fresco
