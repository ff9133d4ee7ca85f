// Repulsive pair term of the hybrid loss (Eq. 6): E = sum_{m<n} U(|r_m - r_n|), minimum image in
// the periodic box, U(r) = (eps / alpha)(1 - r / sigma)^alpha for r < sigma (alpha = 2.5 is the
// Hertzian potential of Eq. 6, alpha = 2 the harmonic soft sphere), evaluated with a cell list:
// cells at least sigma wide, points counting-sorted by cell, each point scanning its own and the
// neighbouring cells (a finite-ranged potential keeps the cost O(N), as the text after Eq. 6 notes).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>

#include "fresco.h"
#include "fresco_internal.h"

namespace {

constexpr int kPairBlocks = 152 * 32;

struct PairGeom {
    int dim;
    int nc[3];          // cells per axis
    int nd[3];          // distinct neighbour offsets per axis: 1 (nc = 1), 2 (nc = 2) or 3
    double box[3];
    int64_t n;
    double sigma, eps, alpha;
};

template <typename T>
__device__ __forceinline__ T wrap_coord(T r, T L) {
    T x = r - L * floor(r / L);
    if (x >= L) x -= L;
    if (x < T(0)) x = T(0);
    return x;
}

template <typename T, int D>
__device__ __forceinline__ int cell_of(const T (&x)[3], const PairGeom &g, int (&c)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c[a] = 0;
        if (a < D) {
            int v = (int)(x[a] * (T)g.nc[a] / (T)g.box[a]);
            c[a] = v < 0 ? 0 : (v >= g.nc[a] ? g.nc[a] - 1 : v);
        }
    }
    return c[0] + g.nc[0] * (c[1] + g.nc[1] * c[2]);
}

// Words per sorted record: 3D records are padded to four words, so that a candidate is one 16-byte
// load (FP32) or two (FP64) instead of three scalar ones.
template <int D>
constexpr int kPairWords = D == 3 ? 4 : 2;

// The fourth word of a 3D record holds the caller index (its bits); 2D plans keep perm.
template <typename T, int D>
__device__ __forceinline__ void store_pair_record(T *__restrict__ sorted, int *__restrict__ perm,
                                                  int64_t q, const T (&x)[3], int j) {
    if constexpr (D == 2) {
        using V = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
        reinterpret_cast<V *>(sorted)[q] = V{x[0], x[1]};
        perm[q] = j;
    } else if constexpr (sizeof(T) == 4) {
        reinterpret_cast<float4 *>(sorted)[q] = make_float4(x[0], x[1], x[2], __int_as_float(j));
    } else {
        reinterpret_cast<double2 *>(sorted)[2 * q] = make_double2(x[0], x[1]);
        reinterpret_cast<double2 *>(sorted)[2 * q + 1] =
            make_double2(x[2], __longlong_as_double((long long)j));
    }
}
template <typename T, int D>
__device__ __forceinline__ int pair_record_index(const T *__restrict__ sorted,
                                                 const int *__restrict__ perm, int64_t q) {
    if constexpr (D == 2) return perm[q];
    else if constexpr (sizeof(T) == 4) return __float_as_int(sorted[4 * q + 3]);
    else return (int)__double_as_longlong(sorted[4 * q + 3]);
}

template <typename T, int D>
__device__ __forceinline__ void load_pair_record(const T *__restrict__ sorted, int64_t q,
                                                 T (&x)[3]) {
    if constexpr (D == 2) {
        using V = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
        const V v = reinterpret_cast<const V *>(sorted)[q];
        x[0] = v.x; x[1] = v.y; x[2] = T(0);
    } else if constexpr (sizeof(T) == 4) {
        const float4 v = reinterpret_cast<const float4 *>(sorted)[q];
        x[0] = v.x; x[1] = v.y; x[2] = v.z;
    } else {
        const double2 v = reinterpret_cast<const double2 *>(sorted)[2 * q];
        x[0] = v.x; x[1] = v.y; x[2] = sorted[4 * q + 2];
    }
}

template <typename T, int D>
__global__ void __launch_bounds__(256) k_cell_bin(PairGeom g, const T *__restrict__ pts,
                                                  int *__restrict__ cnt, int *__restrict__ key,
                                                  int *__restrict__ slot) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < g.n; j += stride) {
        T x[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int a = 0; a < D; ++a) x[a] = wrap_coord<T>(pts[j * D + a], (T)g.box[a]);
        int c[3];
        const int lin = cell_of<T, D>(x, g, c);
        key[j] = lin;
        slot[j] = atomicAdd(&cnt[lin], 1);
    }
}

template <typename T, int D>
__global__ void __launch_bounds__(256) k_cell_scatter(PairGeom g, const T *__restrict__ pts,
                                                      const int *__restrict__ key,
                                                      const int *__restrict__ slot,
                                                      const int *__restrict__ off,
                                                      T *__restrict__ sorted,
                                                      int *__restrict__ perm) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < g.n; j += stride) {
        const int64_t pos = (int64_t)off[key[j]] + slot[j];
        T x[3];
#pragma unroll
        for (int a = 0; a < D; ++a)
            x[a] = wrap_coord<T>(pts[j * D + a], (T)g.box[a]);
        store_pair_record<T, D>(sorted, perm, pos, x, (int)j);
    }
}

// A thread's energy sum, no less exact than adding every term in FP64, which took 446 us on 2^21 points
// in 3D (the whole term) against 380 with three floats. Terms and sums beyond 1e30 go to the FP64 part, a
// word of the thread in shared memory.
template <typename T>
struct EnergySum;
template <>
struct EnergySum<float> {
    fresco::Sum3 s;
    double *d;
    __device__ __forceinline__ explicit EnergySum(double *word) : d(word) { *d = 0.0; }
    __device__ __forceinline__ void add(float x) {
        if (!(s.h + x < 1e30f)) {
            *d += s.value() + (double)x;
            s = fresco::Sum3();
            return;
        }
        s.add(x);
    }
    __device__ __forceinline__ double value() const { return *d + s.value(); }
};
template <>
struct EnergySum<double> {
    double d = 0.0;
    __device__ __forceinline__ explicit EnergySum(double *) {}
    __device__ __forceinline__ void add(double x) { d += x; }
    __device__ __forceinline__ double value() const { return d; }
};

// U and U' of one pair at distance r = sqrt(r2) < sigma: the energy goes to the thread's sum, the force
// along dx to f.
template <typename T, int D>
__device__ __forceinline__ void add_pair(const PairGeom &g, T r2, const T (&dx)[3], T inv_sig,
                                         T eps, T alpha, T eps_alpha, bool harmonic, bool hertz,
                                         EnergySum<T> &e, T (&f)[3]) {
    const T r = sqrt(r2);
    const T u = fmax(T(1) - r * inv_sig, T(0));   // (r2 < sigma^2 may still round to r > sigma)
    T up;   // u^(alpha - 1)
    if (harmonic) up = u;
    else if (hertz) up = u * sqrt(u);
    else up = pow(u, alpha - T(1));
    e.add(eps_alpha * up * u);
    const T coef = -eps * inv_sig * up / r;
#pragma unroll
    for (int a = 0; a < D; ++a) f[a] = fma(coef, dx[a], f[a]);
}

// Cell rows of a point's neighbourhood: 3^(D-1) rows of up to three cells, contiguous in the sorted
// order, plus one wrapped cell per row at the ends of an x row.
template <int D>
constexpr int kPairSegs = D == 3 ? 18 : 6;

// One thread per (sorted) point; every pair is seen from both ends, so each end books half of the
// pair energy and its own force.
//
// ROWS (at least three cells along every axis): the three cells of a row of the neighbourhood are
// one range of the sorted order, and the periodic shift of a candidate follows from its cell. The
// thread first collects the non-empty ranges of its rows in shared memory (all offset loads in
// flight at once), then runs through their points in one flat loop, so the lanes of a warp wait
// for the largest total (about 1.6 times the mean at 14 candidates) and not for the largest count
// of every cell in turn. What bounds it is that imbalance and the instructions per candidate (a
// prefetch of the next candidate's record changed nothing). 2^21 points in 3D, sigma = 0.8
// spacings, FP32, GB300, the whole term: 741 -> 378 us against one loop per cell with a division per
// candidate and axis and an FP64 addition per pair. With two cells along an axis (sigma above a
// third of the box) a candidate's shift is not known from its cell: the general form scans the
// distinct cells one by one and rounds to the nearest image.
template <typename T, int D, bool ROWS>
__global__ void __launch_bounds__(128) k_pair(PairGeom g, const T *__restrict__ sorted,
                                              const int *__restrict__ perm,
                                              const int *__restrict__ off, int accumulate,
                                              T *__restrict__ grad, double *__restrict__ partial) {
    constexpr int BS = 128;
    __shared__ double ws[BS / 32];
    __shared__ int2 seg[ROWS ? kPairSegs<D> : 1][BS];
    __shared__ unsigned char seg_shift[ROWS ? kPairSegs<D> : 1][BS];
    __shared__ double s_big[sizeof(T) == 4 ? BS : 1];
    EnergySum<T> es(s_big + (sizeof(T) == 4 ? threadIdx.x : 0));
    const T sig = (T)g.sigma, inv_sig = T(1) / sig, sig2 = sig * sig;
    const T eps = (T)g.eps, alpha = (T)g.alpha, eps_alpha = eps / alpha;
    const bool harmonic = g.alpha == 2.0, hertz = g.alpha == 2.5;
    const T L[3] = {(T)g.box[0], (T)g.box[1], (T)g.box[2]};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += stride) {
        T x[3];
        load_pair_record<T, D>(sorted, i, x);
        int c[3];
        cell_of<T, D>(x, g, c);
        T f[3] = {T(0), T(0), T(0)};
        if constexpr (ROWS) {
            constexpr int NR = D == 3 ? 9 : 3;
            const int lo = max(c[0] - 1, 0), hi = min(c[0] + 1, g.nc[0] - 1);
            const int edge = c[0] == 0 ? -1 : (c[0] == g.nc[0] - 1 ? 1 : 0);   // x shift of the
            const int wx = edge < 0 ? g.nc[0] - 1 : 0;                         // wrapped cell
            int q0[NR], q1[NR], row[NR], code[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int o[3] = {0, r % 3 - 1, D == 3 ? r / 3 - 1 : 0};
                int base = 0, sh = 1;   // shift code: (sx + 1) + 3 (sy + 1) + 9 (sz + 1)
#pragma unroll
                for (int a = D - 1; a >= 1; --a) {
                    int v = c[a] + o[a], w = 0;
                    if (v < 0) { v += g.nc[a]; w = -1; }
                    else if (v >= g.nc[a]) { v -= g.nc[a]; w = 1; }
                    base = (base + v) * g.nc[a - 1];
                    sh += (w + 1) * (a == 1 ? 3 : 9);
                }
                row[r] = base;
                code[r] = sh + (D == 2 ? 9 : 0);
                q0[r] = off[base + lo];
                q1[r] = off[base + hi + 1];
            }
            int ns = 0;
#pragma unroll
            for (int r = 0; r < NR; ++r)
                if (q1[r] > q0[r]) {
                    seg[ns][threadIdx.x] = make_int2(q0[r], q1[r]);
                    seg_shift[ns++][threadIdx.x] = (unsigned char)code[r];
                }
            if (edge)
                for (int r = 0; r < NR; ++r) {
                    const int a0 = off[row[r] + wx], a1 = off[row[r] + wx + 1];
                    if (a1 > a0) {
                        seg[ns][threadIdx.x] = make_int2(a0, a1);
                        seg_shift[ns++][threadIdx.x] = (unsigned char)(code[r] + edge);
                    }
                }
            // (the point's own cell is never empty: ns >= 1)
            int s = 0, q = seg[0][threadIdx.x].x, qe = seg[0][threadIdx.x].y;
            int sh = seg_shift[0][threadIdx.x];
            T S[3] = {L[0] * (T)(sh % 3 - 1), L[1] * (T)((sh / 3) % 3 - 1), L[2] * (T)(sh / 9 - 1)};
            while (true) {
                if (q == qe) {
                    if (++s == ns) break;
                    const int2 n = seg[s][threadIdx.x];
                    q = n.x;
                    qe = n.y;
                    sh = seg_shift[s][threadIdx.x];
                    S[0] = L[0] * (T)(sh % 3 - 1);
                    S[1] = L[1] * (T)((sh / 3) % 3 - 1);
                    S[2] = L[2] * (T)(sh / 9 - 1);
                }
                T y[3], dx[3], r2 = T(0);
                load_pair_record<T, D>(sorted, q, y);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    dx[a] = a < D ? (x[a] - y[a]) - S[a] : T(0);
                    r2 = fma(dx[a], dx[a], r2);
                }
                // (the point itself, and coincident points, have r2 = 0)
                if (r2 < sig2 && r2 > T(0))
                    add_pair<T, D>(g, r2, dx, inv_sig, eps, alpha, eps_alpha, harmonic, hertz, es,
                                   f);
                ++q;
            }
        } else {
            const int zl = D == 3 ? g.nd[2] : 1;
            for (int oz = 0; oz < zl; ++oz)
                for (int oy = 0; oy < g.nd[1]; ++oy)
                    for (int ox = 0; ox < g.nd[0]; ++ox) {
                        const int o[3] = {ox, oy, oz};
                        int cc[3];
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            if (a >= D) { cc[a] = 0; continue; }
                            // offsets -1, 0, +1 (only the distinct ones when nc < 3)
                            int d = g.nd[a] == 1 ? 0 : (g.nd[a] == 2 ? o[a] : o[a] - 1);
                            int v = c[a] + d;
                            v += v < 0 ? g.nc[a] : (v >= g.nc[a] ? -g.nc[a] : 0);
                            cc[a] = v;
                        }
                        const int lin = cc[0] + g.nc[0] * (cc[1] + g.nc[1] * cc[2]);
                        const int q0 = off[lin], q1 = off[lin + 1];
                        for (int q = q0; q < q1; ++q) {
                            T y[3], dx[3] = {T(0), T(0), T(0)}, r2 = T(0);
                            load_pair_record<T, D>(sorted, q, y);
#pragma unroll
                            for (int a = 0; a < D; ++a) {
                                T v = x[a] - y[a];
                                v -= L[a] * rint(v / L[a]);
                                dx[a] = v;
                                r2 = fma(v, v, r2);
                            }
                            if (r2 < sig2 && r2 > T(0))
                                add_pair<T, D>(g, r2, dx, inv_sig, eps, alpha, eps_alpha, harmonic,
                                               hertz, es, f);
                        }
                    }
        }
        const int64_t j = pair_record_index<T, D>(sorted, perm, i);
#pragma unroll
        for (int a = 0; a < D; ++a) {
            if (accumulate) grad[j * D + a] += f[a];
            else grad[j * D + a] = f[a];
        }
    }
    double e = 0.5 * es.value();   // (each pair is booked at both ends)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < BS / 32; ++w) s += ws[w];
        partial[blockIdx.x] = s;
    }
}

__global__ void __launch_bounds__(256) k_pair_final(const double *__restrict__ partial, int nb,
                                                    int accumulate, double *__restrict__ energy) {
    __shared__ double sm[256];
    double v = 0.0;
    for (int i = threadIdx.x; i < nb; i += 256) v += partial[i];
    sm[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *energy = accumulate ? *energy + sm[0] : sm[0];
}

}  // namespace

struct fresco_pair_s {
    PairGeom g{};
    int precision = FRESCO_F32;
    size_t es = 4;
    cudaStream_t stream = nullptr;
    int64_t ncell = 0;
    int *cnt = nullptr, *off = nullptr, *bsum = nullptr, *key = nullptr, *slot = nullptr;
    int *perm = nullptr;
    void *sorted = nullptr;
    double *partial = nullptr;
    int n_blocks = 0;
};

namespace {

void pair_free(fresco_pair_s *p) {
    if (!p) return;
    if (p->stream) cudaStreamSynchronize(p->stream);
    void *b[] = {p->cnt, p->off, p->bsum, p->key, p->slot, p->perm, p->sorted, p->partial};
    for (void *x : b)
        if (x) cudaFree(x);
    delete p;
}

template <typename T>
fresco_status pair_eval(fresco_pair_s *p, const void *pts, double *energy, void *grad,
                        int accumulate) {
    const PairGeom &g = p->g;
    cudaStream_t s = p->stream;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((g.n + 255) / 256, 152 * 16));
    if (cudaMemsetAsync(p->cnt, 0, sizeof(int) * (size_t)p->ncell, s) != cudaSuccess)
        return FRESCO_ERR_CUDA;
    if (g.dim == 2)
        k_cell_bin<T, 2><<<grid, 256, 0, s>>>(g, (const T *)pts, p->cnt, p->key, p->slot);
    else
        k_cell_bin<T, 3><<<grid, 256, 0, s>>>(g, (const T *)pts, p->cnt, p->key, p->slot);
    int nl = 0;
    if (fresco::Launch<float>::scan(p->cnt, p->off, p->bsum, p->ncell, s, &nl) != cudaSuccess)
        return FRESCO_ERR_CUDA;
    const bool rows = g.nc[0] >= 3 && g.nc[1] >= 3 && (g.dim == 2 || g.nc[2] >= 3);
    const T *sorted = (const T *)p->sorted;
    T *gr = (T *)grad;
    if (g.dim == 2) {
        k_cell_scatter<T, 2><<<grid, 256, 0, s>>>(g, (const T *)pts, p->key, p->slot, p->off,
                                                  (T *)p->sorted, p->perm);
        const auto kern = rows ? k_pair<T, 2, true> : k_pair<T, 2, false>;
        kern<<<p->n_blocks, 128, 0, s>>>(g, sorted, p->perm, p->off, accumulate, gr, p->partial);
    } else {
        k_cell_scatter<T, 3><<<grid, 256, 0, s>>>(g, (const T *)pts, p->key, p->slot, p->off,
                                                  (T *)p->sorted, p->perm);
        const auto kern = rows ? k_pair<T, 3, true> : k_pair<T, 3, false>;
        kern<<<p->n_blocks, 128, 0, s>>>(g, sorted, p->perm, p->off, accumulate, gr, p->partial);
    }
    k_pair_final<<<1, 256, 0, s>>>(p->partial, p->n_blocks, accumulate, energy);
    return cudaGetLastError() == cudaSuccess ? FRESCO_OK : FRESCO_ERR_CUDA;
}

}  // namespace

extern "C" {

fresco_status fresco_pair_plan(fresco_pair_t *out, int dim, const double *box, int64_t n_points,
                               double sigma, double eps, double alpha, int precision,
                               void *stream) {
    if (!out) return FRESCO_ERR_ARG;
    *out = nullptr;
    if ((dim != 2 && dim != 3) || !box || n_points < 1 || n_points > 2147483647LL ||
        !(sigma > 0.0) || !(eps >= 0.0) || !(alpha > 1.0) || !std::isfinite(alpha) ||
        (precision != FRESCO_F32 && precision != FRESCO_F64))
        return FRESCO_ERR_ARG;
    PairGeom g{};
    g.dim = dim;
    g.n = n_points;
    g.sigma = sigma;
    g.eps = eps;
    g.alpha = alpha;
    int64_t ncell = 1;
    for (int a = 0; a < 3; ++a) {
        if (a < dim) {
            if (!(box[a] > 0.0) || !std::isfinite(box[a])) return FRESCO_ERR_ARG;
            if (!(sigma < 0.5 * box[a])) return FRESCO_ERR_UNSUPPORTED;   // minimum image
            double nc = std::floor(box[a] / sigma);
            if (nc > 4096.0) nc = 4096.0;
            g.nc[a] = (int)nc;
            g.nd[a] = g.nc[a] >= 3 ? 3 : g.nc[a];
            g.box[a] = box[a];
        } else {
            g.nc[a] = 1;
            g.nd[a] = 1;
            g.box[a] = 1.0;
        }
        ncell *= g.nc[a];
    }
    if (ncell >= 2147483647LL) return FRESCO_ERR_UNSUPPORTED;
    fresco_pair_s *p = new (std::nothrow) fresco_pair_s();
    if (!p) return FRESCO_ERR_OOM;
    p->g = g;
    p->precision = precision;
    p->es = precision == FRESCO_F64 ? 8 : 4;
    p->stream = (cudaStream_t)stream;
    p->ncell = ncell;
    p->n_blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n_points + 127) / 128, kPairBlocks));
    auto A = [](void **q, size_t b) {
        if (cudaMalloc(q, b) != cudaSuccess) {
            cudaGetLastError();
            *q = nullptr;
            return false;
        }
        return true;
    };
    const size_t N = (size_t)n_points;
    bool ok = A((void **)&p->cnt, sizeof(int) * ncell) &&
              A((void **)&p->off, sizeof(int) * (ncell + 1)) &&
              A((void **)&p->bsum, sizeof(int) * ((ncell + 1023) / 1024 + 1)) &&
              A((void **)&p->key, sizeof(int) * N) && A((void **)&p->slot, sizeof(int) * N) &&
              (dim == 3 || A((void **)&p->perm, sizeof(int) * N)) &&
              A(&p->sorted, p->es * N * (dim == 3 ? kPairWords<3> : kPairWords<2>)) &&
              A((void **)&p->partial, sizeof(double) * p->n_blocks);
    if (!ok) {
        pair_free(p);
        return FRESCO_ERR_OOM;
    }
    *out = p;
    return FRESCO_OK;
}

fresco_status fresco_pair_energy_grad(fresco_pair_t p, const void *d_points, double *d_energy,
                                      void *d_grad, int accumulate) {
    fresco::clear_pending_error();
    if (!p || !d_points || !d_energy || !d_grad) return FRESCO_ERR_ARG;
    if (p->precision == FRESCO_F64) return pair_eval<double>(p, d_points, d_energy, d_grad, accumulate);
    return pair_eval<float>(p, d_points, d_energy, d_grad, accumulate);
}

fresco_status fresco_pair_set_stream(fresco_pair_t p, void *stream) {
    if (!p) return FRESCO_ERR_ARG;
    p->stream = (cudaStream_t)stream;
    return FRESCO_OK;
}

fresco_status fresco_pair_destroy(fresco_pair_t p) {
    pair_free(p);
    return FRESCO_OK;
}

}  // extern "C"
