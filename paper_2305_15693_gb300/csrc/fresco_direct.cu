// Direct sums for small single plans: rho(n) and the gradient by separable phases instead of the
// nonuniform FFT.
//
// A small problem's evaluation by NUFFT is some twenty launches of nearly empty kernels. Its direct
// sums cost less than those launches: with A_j[n] = exp(+2 pi i n x_j / L_x) and B_j[m] the phase of
// a column m of the mask (a pair +-(n_y[, n_z]), the half with n_y > 0 or n_y = 0 and n_z >= 0),
//   rho(n, +m) = conj sum_j A_j[n] B_j[m],   rho(n, -m) = conj sum_j A_j[n] conj B_j[m]
// come from the same four real sums (Ar Br, Ai Bi, Ar Bi, Ai Br): two fused multiply-adds per point
// and wavevector; and with D(n, +-m) = E rho, E = 4 W' (S - S0') / N (Eq. 4),
//   dL/dr_j = -sum_n k Im[A_j[n] (sum_m D+ B_j[m] + D- conj B_j[m])],
// where the sums over m with and without the factors n_y, n_z share their loads. Three launches:
//   k_direct_rho   one block per chunk of points: phases (kept for the gradient), then the sums of
//                  its points for every quad of four n at one column; blocks leave partial sums;
//   k_direct_mask  adds the partial sums in a fixed order, forms S, the loss (FP64) and D; the last
//                  block to finish adds the loss partials in a fixed order;
//   k_direct_grad  threads over (point, n), the block's points' B in shared memory.
// Columns are sorted by their number of quads, so quad row q (n = 4 q .. 4 q + 3) holds columns
// 0 .. cnt[q] - 1 and cell (n, m) is (qbase[n / 4] + m) * 4 + n % 4, without tables per column.
// FP32 phases keep the point's position as a float pair and reduce n x modulo 1 exactly, so each is
// within an ulp or two; FP64 likewise. Errors against 64 bits are those of the arithmetic alone
// (the NUFFT adds its kernel's truncation).
//
// What bounds it: FP64 the FP64 pipe; FP32 shared-memory loads; at the smallest sizes the three
// launches; with few points the gradient's walk over all cells, which every block makes for its
// eight points. The line between the two forms (kDirectWork, kDirectCost) lies where they measured
// equal on GB300; see direct_build.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <initializer_list>
#include <new>
#include <type_traits>
#include <vector>

#include "fresco.h"
#include "fresco_internal.h"

namespace fresco {

namespace {

// dynamic shared memory the kernels may take (the same limits for every plan: the attribute belongs
// to the kernel, not to the plan)
constexpr int kDirectRhoSmem = 100 * 1024, kDirectGradSmem = 200 * 1024;
constexpr int kDirectStage = 64 * 1024;   // gradient: bytes of staged coefficients

template <typename T>
using Cx = typename std::conditional<sizeof(T) == 4, float2, double2>::type;

struct DirectGeom {
    int dim;
    int n_points;
    int kx, ky, kz;      // largest |n| per axis
    int nx4;             // kx + 1 rounded up to a multiple of 4
    int n_col, n_quad;   // columns, quads
    int chunk, n_blk;    // points per block of the forward sums, blocks
    int groups;          // thread groups that split a block's points
    double s_hi[3], s_lo[3];   // 1 / L as s_hi + s_lo (s_hi exact in the working precision)
    double kscale[3];          // 2 pi / L
    double inv_n;
    double loss_const;
};

__device__ __forceinline__ void cispi(float t, float &c, float &s) { sincospif(2.f * t, &s, &c); }
__device__ __forceinline__ void cispi(double t, double &c, double &s) { sincospi(2.0 * t, &s, &c); }

// exp(2 pi i n (hi + lo)), the product reduced modulo 1 exactly before the trigonometric call
template <typename T>
__device__ __forceinline__ Cx<T> phase(int n, T hi, T lo) {
    const T q = (T)n * hi;
    const T e = fma((T)n, hi, -q) + (T)n * lo;
    Cx<T> v;
    cispi((q - rint(q)) + e, v.x, v.y);
    return v;
}

template <typename T>
__host__ __device__ size_t direct_rho_smem(const DirectGeom &g, int chunk) {
    const size_t per = (size_t)(g.nx4 + g.n_col + (g.dim == 3 ? g.ky + g.kz + 2 : 0)) * 2 + 6;
    return per * sizeof(T) * chunk;
}

constexpr int kRhoThreads = 512;

template <typename T, int D>
__global__ void __launch_bounds__(kRhoThreads) k_direct_rho(DirectGeom g, const T *__restrict__ pts,
                                                    const int2 *__restrict__ cols,
                                                    const int2 *__restrict__ quads,
                                                    Cx<T> *__restrict__ tab, T *__restrict__ part,
                                                    int *__restrict__ err) {
    using C = Cx<T>;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    C *sa = reinterpret_cast<C *>(sm_raw);          // [chunk][nx4]
    C *sb = sa + (size_t)g.chunk * g.nx4;           // [chunk][n_col]
    C *ty = sb + (size_t)g.chunk * g.n_col;         // 3D: [chunk][ky + 1], [chunk][kz + 1]
    C *tz = ty + (D == 3 ? (size_t)g.chunk * (g.ky + 1) : 0);
    T *sf = reinterpret_cast<T *>(tz + (D == 3 ? (size_t)g.chunk * (g.kz + 1) : 0));   // [chunk][6]
    const int j0 = blockIdx.x * g.chunk;
    const int n = min(g.chunk, g.n_points - j0);
    bool ok = true;
    for (int t = threadIdx.x; t < n * D; t += blockDim.x) {
        const int j = t / D, a = t - j * D;
        T r = pts[(int64_t)(j0 + j) * D + a];
        if (!isfinite(r)) {
            ok = false;
            r = T(0);
        }
        const T sh = (T)g.s_hi[a];
        const T p = r * sh;
        sf[j * 6 + 2 * a] = p - rint(p);
        sf[j * 6 + 2 * a + 1] = fma(r, (T)g.s_lo[a], fma(r, sh, -p));
    }
    if (!ok) atomicOr(err, 1);
    __syncthreads();
    for (int t = threadIdx.x; t < n * g.nx4; t += blockDim.x) {
        const int j = t / g.nx4, k = t - j * g.nx4;
        sa[t] = k <= g.kx ? phase<T>(k, sf[j * 6], sf[j * 6 + 1]) : C{T(0), T(0)};
    }
    if constexpr (D == 2) {
        for (int t = threadIdx.x; t < n * g.n_col; t += blockDim.x) {
            const int j = t / g.n_col, m = t - j * g.n_col;
            sb[t] = phase<T>(cols[m].x, sf[j * 6 + 2], sf[j * 6 + 3]);
        }
    } else {
        for (int t = threadIdx.x; t < n * (g.ky + 1); t += blockDim.x) {
            const int j = t / (g.ky + 1), k = t - j * (g.ky + 1);
            ty[t] = phase<T>(k, sf[j * 6 + 2], sf[j * 6 + 3]);
        }
        for (int t = threadIdx.x; t < n * (g.kz + 1); t += blockDim.x) {
            const int j = t / (g.kz + 1), k = t - j * (g.kz + 1);
            tz[t] = phase<T>(k, sf[j * 6 + 4], sf[j * 6 + 5]);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < n * g.n_col; t += blockDim.x) {
            const int j = t / g.n_col, m = t - j * g.n_col;
            const int2 c = cols[m];   // n_y >= 0, n_z of either sign
            const C y = ty[j * (g.ky + 1) + c.x];
            C z = tz[j * (g.kz + 1) + (c.y < 0 ? -c.y : c.y)];
            if (c.y < 0) z.y = -z.y;
            sb[t] = C{y.x * z.x - y.y * z.y, fma(y.x, z.y, y.y * z.x)};
        }
    }
    __syncthreads();
    // the phases for the gradient, [nx4 + n_col][n_points]
    for (int t = threadIdx.x; t < n * (g.nx4 + g.n_col); t += blockDim.x) {
        const int i = t / n, j = t - i * n;
        tab[(int64_t)i * g.n_points + j0 + j] =
            i < g.nx4 ? sa[j * g.nx4 + i] : sb[j * g.n_col + i - g.nx4];
    }
    const int gt = blockDim.x / g.groups, grp = threadIdx.x / gt;
    const int64_t cells = 4 * (int64_t)g.n_quad;
    T *out = part + (int64_t)blockIdx.x * 4 * cells;
    // (several groups: a group has a thread for every quad, so the loop runs once)
    for (int q = threadIdx.x - grp * gt; q < g.n_quad || g.groups > 1; q += gt) {
        T rr[4] = {}, ii[4] = {}, ri[4] = {}, ir[4] = {};
        const bool in = q < g.n_quad;
        const int2 qm = in ? quads[q] : make_int2(0, 0);
        const C *a = sa + 4 * qm.x, *b = sb + qm.y;
#pragma unroll 4
        for (int j = in ? grp : n; j < n; j += g.groups) {
            const C v = b[j * g.n_col];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const C u = a[j * g.nx4 + k];
                rr[k] = fma(u.x, v.x, rr[k]);
                ii[k] = fma(u.y, v.y, ii[k]);
                ri[k] = fma(u.x, v.y, ri[k]);
                ir[k] = fma(u.y, v.x, ir[k]);
            }
        }
        if (g.groups > 1) {
            // the groups' sums through shared memory, added in order by the first one
            __syncthreads();
            T *red = reinterpret_cast<T *>(sm_raw);
            if (grp && in)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    T *o = red + (size_t)((grp - 1) * 16 + 4 * k) * gt + q;
                    o[0] = rr[k];
                    o[gt] = ii[k];
                    o[2 * gt] = ri[k];
                    o[3 * gt] = ir[k];
                }
            __syncthreads();
            if (grp || !in) return;
            for (int h = 0; h < g.groups - 1; ++h)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const T *o = red + (size_t)(h * 16 + 4 * k) * gt + q;
                    rr[k] += o[0];
                    ii[k] += o[gt];
                    ri[k] += o[2 * gt];
                    ir[k] += o[3 * gt];
                }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            out[4 * (int64_t)q + k] = rr[k];
            out[cells + 4 * (int64_t)q + k] = ii[k];
            out[2 * cells + 4 * (int64_t)q + k] = ri[k];
            out[3 * cells + 4 * (int64_t)q + k] = ir[k];
        }
        if (g.groups > 1) return;
    }
}

// kMaskCells cells per block: 32 threads per cell take every 32nd partial sum, then one warp per
// cell adds their results. Few cells per block spread a small problem over the SMs: 1024 FP64 points
// took 40 us with 32 cells a block, 15 with 8 and 18 with 4.
constexpr int kMaskCells = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kMaskCells) k_direct_mask(DirectGeom g, int n_part,
                                                     const T *__restrict__ part,
                                                     const T *__restrict__ cell_s0,
                                                     const T *__restrict__ cell_w,
                                                     Cx<T> *__restrict__ rho, T *__restrict__ dco,
                                                     double *__restrict__ lpart,
                                                     unsigned *__restrict__ done,
                                                     double *__restrict__ loss) {
    using C = Cx<T>;
    __shared__ T sm[4][32][kMaskCells + 1];
    __shared__ double sl[kMaskCells];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t cells = 4 * (int64_t)g.n_quad;
    {
        const int cl = threadIdx.x % kMaskCells, sp = threadIdx.x / kMaskCells;
        const int64_t c = (int64_t)blockIdx.x * kMaskCells + cl;
        T v[4] = {T(0), T(0), T(0), T(0)};
        if (c < cells) {
#pragma unroll 4
            for (int s = sp; s < n_part; s += 32) {
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] += part[((int64_t)s * 4 + k) * cells + c];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) sm[k][sp][cl] = v[k];
    }
    __syncthreads();
    T v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = sm[k][lane][wid];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
    const int64_t c = (int64_t)blockIdx.x * kMaskCells + wid;
    if (lane < 2) {   // lane 0 the wavevector at +m, lane 1 the one at -m
        double l = 0.0;
        C d{T(0), T(0)};
        if (c < cells) {
            const T inv_n = (T)g.inv_n;
            C r;
            r.x = lane ? v[0] + v[1] : v[0] - v[1];
            r.y = lane ? v[2] - v[3] : -(v[2] + v[3]);
            rho[2 * c + lane] = r;
            const T w = cell_w[2 * c + lane], s0 = cell_s0[2 * c + lane];
            if (w > T(0)) {
                const T S = (r.x * r.x + r.y * r.y) * inv_n;
                const double dv = (double)S - (double)s0;
                l = (double)w * dv * dv;
                const T e = T(4) * w * (T)dv * inv_n;
                d = C{e * r.x, e * r.y};
            }
        }
        const T ox = __shfl_xor_sync(3u, d.x, 1), oy = __shfl_xor_sync(3u, d.y, 1);
        l += __shfl_xor_sync(3u, l, 1);
        if (c < cells) {   // D+ + D-, then D+ - D-
            dco[4 * c + 2 * lane] = lane ? ox - d.x : d.x + ox;
            dco[4 * c + 2 * lane + 1] = lane ? oy - d.y : d.y + oy;
        }
        if (lane == 0) sl[wid] = l;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kMaskCells; ++w) s += sl[w];
        lpart[blockIdx.x] = s;
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (wid == 0) {
        double s = 0.0;
        for (int i = lane; i < (int)gridDim.x; i += 32) s += __ldcg(lpart + i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            *loss = s + g.loss_const;
            *done = 0;
        }
    }
}

// PJ points per block; thread t takes point t % PJ and every (NT / PJ)-th n from t / PJ.
template <int PJ>
constexpr int kGradThreads = PJ == 32 ? 512 : 256;

template <typename T, int D, int PJ>
__global__ void __launch_bounds__(kGradThreads<PJ>) k_direct_grad(DirectGeom g, const int2 *__restrict__ cols,
                                                     const int *__restrict__ qbase,
                                                     const Cx<T> *__restrict__ tab,
                                                     const T *__restrict__ dco,
                                                     const double *__restrict__ grad_out,
                                                     T *__restrict__ grad, int stage) {
    using C = Cx<T>;
    constexpr int NT = kGradThreads<PJ>, NL = NT / PJ;
    // FP64, 2D: n_y B is staged too, which saves two of the ten operations per (n, column)
    constexpr bool kScaled = sizeof(T) == 8 && D == 2;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T *sd = reinterpret_cast<T *>(sm_raw);                      // [stage] quads of 16
    C *sb = reinterpret_cast<C *>(sd + 16 * stage);             // [n_col][PJ]
    C *sn = sb + (size_t)g.n_col * PJ;                          // [n_col] (n_y, n_z), or n_y B
    __shared__ T red[D][NL][PJ];
    const int j0 = blockIdx.x * PJ;
    const int jj = threadIdx.x % PJ, nl = threadIdx.x / PJ;
    for (int t = threadIdx.x; t < g.n_col * PJ; t += NT) {
        const int m = t / PJ, j = t - m * PJ;
        const C b = j0 + j < g.n_points ? tab[(int64_t)(g.nx4 + m) * g.n_points + j0 + j]
                                        : C{T(0), T(0)};
        sb[t] = b;
        if (kScaled) sn[t] = C{(T)cols[m].x * b.x, (T)cols[m].x * b.y};
    }
    if (!kScaled)
        for (int m = threadIdx.x; m < g.n_col; m += NT) {
            const int2 c = cols[m];
            sn[m] = C{(T)c.x, (T)c.y};
        }
    T gr[3] = {T(0), T(0), T(0)};
    const bool in = j0 + jj < g.n_points;
    const int nq = g.nx4 / 4;
    // the coefficients pass through shared memory, `stage` quads (whole quad rows) at a time: read
    // from global memory in the loop below they cost an L2 round trip per few columns
    for (int qa = 0; qa < nq;) {
        const int b0 = qbase[qa];
        int qe = qa + 1;
        while (qe < nq && qbase[qe + 1] - b0 <= stage) ++qe;
        __syncthreads();
        {
            // a quad is 4 cells of 4 coefficients: 16 sizeof(T) bytes, sizeof(T) float4s
            const int words = (qbase[qe] - b0) * (int)sizeof(T);
            const float4 *src = reinterpret_cast<const float4 *>(dco + 16 * (int64_t)b0);
            for (int i = threadIdx.x; i < words; i += NT) reinterpret_cast<float4 *>(sd)[i] = src[i];
        }
        __syncthreads();
        const int ke = min(4 * qe, g.kx + 1);
        for (int k = 4 * qa + nl; k < ke; k += NL) {
            const int qb = qbase[k >> 2], cnt = qbase[(k >> 2) + 1] - qb;
            const T *d = sd + 16 * (qb - b0) + 4 * (k & 3);
            T ur = T(0), ui = T(0), yr = T(0), yi = T(0), zr = T(0), zi = T(0);
#pragma unroll 4
            for (int m = 0; m < cnt; ++m) {
                T pr, pi, mr, mi;   // D+ + D-, D+ - D-
                if constexpr (sizeof(T) == 4) {
                    const float4 q = *reinterpret_cast<const float4 *>(d + 16 * m);
                    pr = q.x; pi = q.y; mr = q.z; mi = q.w;
                } else {
                    const double2 q0 = *reinterpret_cast<const double2 *>(d + 16 * m);
                    const double2 q1 = *reinterpret_cast<const double2 *>(d + 16 * m + 2);
                    pr = q0.x; pi = q0.y; mr = q1.x; mi = q1.y;
                }
                const C b = sb[m * PJ + jj];
                ur = fma(pr, b.x, fma(-mi, b.y, ur));
                ui = fma(pi, b.x, fma(mr, b.y, ui));
                if constexpr (kScaled) {
                    const C c = sn[m * PJ + jj];
                    yr = fma(mr, c.x, fma(-pi, c.y, yr));
                    yi = fma(mi, c.x, fma(pr, c.y, yi));
                    continue;
                }
                const C nn = sn[m];
                const T tr = fma(mr, b.x, -(pi * b.y)), ti = fma(mi, b.x, pr * b.y);
                yr = fma(nn.x, tr, yr);
                yi = fma(nn.x, ti, yi);
                if (D == 3) {
                    zr = fma(nn.y, tr, zr);
                    zi = fma(nn.y, ti, zi);
                }
            }
            if (in) {
                const C a = tab[(int64_t)k * g.n_points + j0 + jj];
                gr[0] = fma((T)k, fma(a.x, ui, a.y * ur), gr[0]);
                gr[1] += fma(a.x, yi, a.y * yr);
                if (D == 3) gr[2] += fma(a.x, zi, a.y * zr);
            }
        }
        qa = qe;
    }
#pragma unroll
    for (int a = 0; a < D; ++a) red[a][nl][jj] = gr[a];
    __syncthreads();
    const T sc = grad_out ? (T)(*grad_out) : T(1);
    for (int t = threadIdx.x; t < PJ * D; t += NT) {
        const int j = t / D, a = t - j * D;
        if (j0 + j >= g.n_points) continue;
        T s = T(0);
        for (int i = 0; i < NL; ++i) s += red[a][i][j];
        grad[(int64_t)(j0 + j) * D + a] = -sc * (T)g.kscale[a] * s;
    }
}

// rho and S of the mask rows: row q reads cell entry idx[q] = 2 * cell + sign, conjugated (and the
// wavevector negated) where neg[q] is set
template <typename T>
__global__ void k_direct_rho_s(int64_t n_k, const int *__restrict__ idx, const Cx<T> *__restrict__ r,
                               T inv_n, T *__restrict__ rho, T *__restrict__ S) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n_k) return;
    const int i = idx[q];
    const Cx<T> v = r[i < 0 ? -(i + 1) : i];
    if (rho) {
        rho[2 * q] = v.x;
        rho[2 * q + 1] = i < 0 ? -v.y : v.y;
    }
    if (S) S[q] = (v.x * v.x + v.y * v.y) * inv_n;
}

// Quads of coefficients the gradient stages at once (at least a whole quad row, which has no more
// than n_col), and its dynamic shared memory: those, the block's B and the columns.
int direct_stage(const DirectGeom &g, size_t es) {
    return std::max(g.n_col, std::min(g.n_quad, (int)(kDirectStage / (16 * es))));
}
size_t direct_grad_smem(const DirectGeom &g, int pj, int stage, size_t es) {
    return 16 * es * (size_t)stage +
           2 * es * (size_t)g.n_col * (es == 8 && g.dim == 2 ? 2 * pj : pj + 1);
}

// Blocks and threads of the forward sums: points per block so that every SM has one, and their
// phases fit in half of an SM's shared memory
template <typename T>
void size_chunks(DirectGeom &g) {
    g.chunk = std::max(1, (g.n_points + 151) / 152);
    while (g.chunk > 1 && direct_rho_smem<T>(g, g.chunk) > kDirectRhoSmem) --g.chunk;
    g.n_blk = (g.n_points + g.chunk - 1) / g.chunk;
    g.groups = 1;   // a power of two, so that it divides the block
    while (g.groups < 16 && kRhoThreads / (2 * g.groups) >= ((g.n_quad + 31) / 32) * 32 &&
           2 * g.groups <= g.chunk)
        g.groups *= 2;
}

// dynamic shared memory of k_direct_rho: the phases, or the groups' sums after them
template <typename T>
size_t direct_rho_bytes(const DirectGeom &g) {
    const size_t red = (size_t)(g.groups - 1) * 16 * (kRhoThreads / g.groups) * sizeof(T);
    return std::max(direct_rho_smem<T>(g, g.chunk), red);
}

}  // namespace

struct DirectPlan {
    DirectGeom g{};
    std::vector<void *> allocs;
    int2 *cols = nullptr, *quads = nullptr;
    int *qbase = nullptr;
    void *cell_s0 = nullptr, *cell_w = nullptr, *part = nullptr, *dco = nullptr, *rho = nullptr;
    void *tab = nullptr;
    double *lpart = nullptr;
    unsigned *done = nullptr;
    int *row_idx = nullptr;            // [n_k] mask rows -> cell entries (fresco_get_rho_S)
    int64_t n_k = 0;
    int n_mask_blk = 0;
    int64_t bytes = 0;
};

// Points x wavevectors (two per cell: +m and -m) up to which a plan takes the direct sums. Measured
// on GB300, loss and gradient, NUFFT against direct sums (us): FP32, 2D, 3.1e5: 78 / 25, 7.2e6: 89 /
// 29, 3.0e7: 82 / 46, 6.0e7: 91 / 67; 3D, 1.7e7: 123 / 41, 4.6e7: 134 / 99. FP64, 2D, 3.2e6: 206 /
// 81, 4.9e6: 279 / 111, 1.3e7: 200 / 252; 3D, 6.1e6: 391 / 198.
static constexpr double kDirectWork[2] = {4.0e7, 9.0e6};   // FP32, FP64
// With few points most SMs idle, the time is that of one block and the wavevectors alone decide;
// the product above does not see it (100 points and K = 500 took 1226 us, the NUFFT 185). Estimates
// of both forms in us, [precision][dimension - 2]. Fitted to 170 pairs of plans of 1 to 8000 points with
// disks, balls, strips and sparse masks of |n| up to 4000, and to 1380 of 30 to 10^6 points with disks and
// balls, on both sides of the line. Direct sums / NUFFT: 2D FP32, 300 points, K = 60 31 / 55, 100 55 / 57,
// 130 75 / 58, 200 160 / 70; 120000 points, K = 10 62 / 91; 10 points, 30 wavevectors of |n| up to 2000
// 170 / 1315, a strip of 4000 x 1 163 / 94; 2D FP64, 300 points, K = 60 100 / 142, 80 156 / 136; K = 50
// and 1000 points 100 / 130, 2000 points 157 / 134; K = 10 and 3000 points 48 / 1295, 30000 157 / 12123;
// 3D, K = 18 and 3000 points 109 / 139; FP64, K = 10 and 1000 points 114 / 212, 3000 189 / 284.
struct DirectCost {
    double fixed, quad, row;         // launches; a quad, a quad row of one block's walk
    double turn;                     // points from which on an SM's blocks wait for its FP64 pipe
    double pt_quad, pt_phase;        // a point's share of the sums over a quad, of one phase
    double nufft, nufft_cell;        // the NUFFT's launches, 10^6 cells of its fine grid
    double nufft_pt;                 // a point (FP64: few enough tiles that all of them count)
    double nufft_dense, crowd;       // more than a point a cell; points per 10^6 cells (few tiles)
};
static constexpr DirectCost kDirectCost[2][2] = {
    {{18.0, 0.0152, 0.11, 0.0, 2.0e-6, 1.4e-5, 55.0, 20.0, 0.0, 30.0, 1.5e-7},
     {15.0, 0.029, 0.11, 0.0, 3.0e-6, 1.0e-5, 100.0, 100.0, 0.0, 0.0, 1.5e-7}},
    {{22.0, 0.097, 0.15, 1216.0, 3.4e-5, 6.0e-5, 122.0, 250.0, 0.0, 0.0, 3.3e-4},
     {25.0, 0.27, 0.15, 2000.0, 1.0e-5, 3.0e-5, 180.0, 900.0, 0.035, 0.0, 1.5e-4}}};
// Tolerances the plan may ask for: the direct sums carry the working precision, so a plan that
// states a looser tolerance keeps the NUFFT whose error it expects (and its speed at that width).
static constexpr double kDirectTol[2] = {1.0e-5, 1.0e-9};

void direct_free(DirectPlan *d) {
    if (!d) return;
    for (void *p : d->allocs) cudaFree(p);
    delete d;
}

int64_t direct_bytes(const DirectPlan *d) { return d->bytes; }

bool direct_wanted(const int64_t n_points, const fresco_opts &o, int precision, double tol) {
    if (o.width_override || o.tile[0] || o.tile[1] || o.tile[2]) return false;
    return tol <= kDirectTol[precision == FRESCO_F64] && n_points <= (1 << 20);
}

template <typename T>
static fresco_status build_t(DirectPlan *d, const std::vector<int2> &cols,
                             const std::vector<int2> &quads, const std::vector<int> &qbase,
                             const std::vector<double> &s0, const std::vector<double> &w,
                             const std::vector<int> &row_idx) {
    DirectGeom &g = d->g;
    d->n_k = (int64_t)row_idx.size();
    size_chunks<T>(g);
    const size_t cells = 4 * (size_t)g.n_quad;
    const size_t n_part = (size_t)g.n_blk;
    d->n_mask_blk = (int)((cells + kMaskCells - 1) / kMaskCells);
    auto A = [&](void **p, size_t b) {
        if (cudaMalloc(p, std::max<size_t>(b, 16)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        d->allocs.push_back(*p);
        d->bytes += (int64_t)b;
        return true;
    };
    if (!(A((void **)&d->cols, sizeof(int2) * cols.size()) &&
          A((void **)&d->quads, sizeof(int2) * quads.size()) &&
          A((void **)&d->qbase, sizeof(int) * qbase.size()) &&
          A((void **)&d->row_idx, sizeof(int) * row_idx.size()) &&
          A(&d->cell_s0, sizeof(T) * 2 * cells) && A(&d->cell_w, sizeof(T) * 2 * cells) &&
          A(&d->part, sizeof(T) * 4 * cells * n_part) && A(&d->dco, sizeof(T) * 4 * cells) &&
          A(&d->rho, sizeof(T) * 4 * cells) &&
          A(&d->tab, sizeof(T) * 2 * (size_t)(g.nx4 + g.n_col) * (size_t)g.n_points) &&
          A((void **)&d->lpart, sizeof(double) * d->n_mask_blk) &&
          A((void **)&d->done, sizeof(unsigned))))
        return FRESCO_ERR_OOM;
    std::vector<T> ts(2 * cells), tw(2 * cells);
    for (size_t i = 0; i < 2 * cells; ++i) {
        ts[i] = (T)s0[i];
        tw[i] = (T)w[i];
    }
    bool ok = cudaMemcpy(d->cols, cols.data(), sizeof(int2) * cols.size(),
                         cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(d->quads, quads.data(), sizeof(int2) * quads.size(),
                         cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(d->qbase, qbase.data(), sizeof(int) * qbase.size(),
                         cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(d->row_idx, row_idx.data(), sizeof(int) * row_idx.size(),
                         cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemcpy(d->cell_s0, ts.data(), sizeof(T) * ts.size(), cudaMemcpyHostToDevice) ==
                  cudaSuccess &&
              cudaMemcpy(d->cell_w, tw.data(), sizeof(T) * tw.size(), cudaMemcpyHostToDevice) ==
                  cudaSuccess &&
              cudaMemset(d->done, 0, sizeof(unsigned)) == cudaSuccess;
    const auto kern = g.dim == 2 ? k_direct_rho<T, 2> : k_direct_rho<T, 3>;
    ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    kDirectRhoSmem) == cudaSuccess;
    const auto g8 = g.dim == 2 ? k_direct_grad<T, 2, 8> : k_direct_grad<T, 3, 8>;
    const auto g32 = g.dim == 2 ? k_direct_grad<T, 2, 32> : k_direct_grad<T, 3, 32>;
    for (const auto k : {g8, g32})
        ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        kDirectGradSmem) == cudaSuccess;
    return ok ? FRESCO_OK : FRESCO_ERR_CUDA;
}

// Builds the direct form of a plan, or leaves *out null where the NUFFT is the better one. mask:
// the caller's rows; rep_n, rep_s0, rep_w: the folded representatives (n_x >= 0 half); fine_cells:
// cells of the fine grid the NUFFT would use.
fresco_status direct_build(DirectPlan **out, int dim, int64_t n_points, const double *box,
                           int precision, double fine_cells, const int32_t *mask, int64_t n_k,
                           const std::vector<int32_t> &rep_n, const std::vector<double> &rep_s0,
                           const std::vector<double> &rep_w, double loss_const) {
    *out = nullptr;
    const double work = kDirectWork[precision == FRESCO_F64];
    if ((double)n_k * 0.5 * (double)n_points > work) return FRESCO_OK;
    // columns +-(n_y, n_z) of the mask's n_x >= 0 half, and the largest n_x of each
    DirectGeom g{};
    g.dim = dim;
    g.n_points = (int)n_points;
    struct Entry {
        int nx, ny, nz;
        bool minus, neg;
    };
    auto entry = [&](const int32_t *r) {
        Entry e{r[0], r[1], dim == 3 ? r[2] : 0, false, false};
        const bool canon = e.nx != 0 ? e.nx > 0 : (e.ny != 0 ? e.ny > 0 : e.nz > 0);
        if (!canon) {
            e = Entry{-e.nx, -e.ny, -e.nz, false, true};
        }
        if (e.ny < 0 || (e.ny == 0 && e.nz < 0)) {
            e.ny = -e.ny;
            e.nz = -e.nz;
            e.minus = true;
        }
        return e;
    };
    int64_t kx = 0, ky = 0, kz = 0;
    for (int64_t q = 0; q < n_k; ++q) {
        const int32_t *r = mask + q * dim;
        kx = std::max<int64_t>(kx, std::abs(r[0]));
        ky = std::max<int64_t>(ky, std::abs(r[1]));
        if (dim == 3) kz = std::max<int64_t>(kz, std::abs(r[2]));
    }
    const int64_t plane = (ky + 1) * (2 * kz + 1);
    if (kx > 4096 || plane > (1 << 16)) return FRESCO_OK;
    g.kx = (int)kx;
    g.ky = (int)ky;
    g.kz = (int)kz;
    g.nx4 = ((int)kx + 4) / 4 * 4;
    std::vector<int> top((size_t)plane, -1);
    for (int64_t q = 0; q < n_k; ++q) {
        const Entry e = entry(mask + q * dim);
        int &t = top[(size_t)(e.ny * (2 * kz + 1) + e.nz + kz)];
        t = std::max(t, e.nx);
    }
    std::vector<int> order;
    for (int64_t i = 0; i < plane; ++i)
        if (top[(size_t)i] >= 0) order.push_back((int)i);
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return top[(size_t)a] / 4 > top[(size_t)b] / 4; });
    std::vector<int2> cols;
    std::vector<int> col_of((size_t)plane, -1), cnt((size_t)g.nx4 / 4, 0), qbase;
    for (int i : order) {
        col_of[(size_t)i] = (int)cols.size();
        cols.push_back(make_int2(i / (int)(2 * kz + 1), i % (int)(2 * kz + 1) - (int)kz));
        for (int q = 0; q <= top[(size_t)i] / 4; ++q) ++cnt[(size_t)q];
    }
    qbase.push_back(0);
    std::vector<int2> quads;
    for (int q = 0; q < g.nx4 / 4; ++q) {
        for (int m = 0; m < cnt[(size_t)q]; ++m) quads.push_back(make_int2(q, m));
        qbase.push_back((int)quads.size());
    }
    g.n_col = (int)cols.size();
    g.n_quad = (int)quads.size();
    if (8.0 * g.n_quad * (double)n_points > 1.25 * work) return FRESCO_OK;
    const DirectCost &c = kDirectCost[precision == FRESCO_F64][dim - 2];
    const double n = (double)n_points, mcells = fine_cells * 1e-6;
    const double turns = c.turn > 0.0 ? std::max(1.0, n / c.turn) : 1.0;
    const double sums = c.fixed + c.quad * g.n_quad * turns + c.row * (g.nx4 / 4) +
                        n * (c.pt_quad * g.n_quad + c.pt_phase * (g.nx4 + g.n_col));
    const double nufft = c.nufft + c.nufft_cell * mcells + c.nufft_pt * n +
                         (n > fine_cells ? c.nufft_dense : 0.0) + c.crowd * n / mcells;
    if (sums > nufft) return FRESCO_OK;
    // one point's phases must fit the shared memory of both kernels
    const size_t es = precision == FRESCO_F64 ? 8 : 4;
    if ((precision == FRESCO_F64 ? direct_rho_smem<double>(g, 1) : direct_rho_smem<float>(g, 1)) >
            kDirectRhoSmem ||
        direct_grad_smem(g, 32, direct_stage(g, es), es) > (size_t)kDirectGradSmem)
        return FRESCO_OK;
    for (int a = 0; a < dim; ++a) {
        const double s = 1.0 / box[a];
        g.s_hi[a] = es == 4 ? (double)(float)s : s;
        g.s_lo[a] = (double)(1.0L / (long double)box[a] - (long double)g.s_hi[a]);
        g.kscale[a] = 2.0 * M_PI / box[a];
    }
    g.inv_n = 1.0 / (double)n_points;
    g.loss_const = loss_const;
    auto cell = [&](const Entry &e) {
        const int m = col_of[(size_t)(e.ny * (2 * kz + 1) + e.nz + kz)];
        return 2 * (4 * (qbase[(size_t)(e.nx / 4)] + m) + e.nx % 4) + (e.minus ? 1 : 0);
    };
    std::vector<double> s0(8 * (size_t)g.n_quad, 0.0), w(8 * (size_t)g.n_quad, 0.0);
    for (size_t r = 0; r < rep_s0.size(); ++r) {
        const int c = cell(entry(rep_n.data() + r * dim));
        s0[(size_t)c] = rep_s0[r];
        w[(size_t)c] = rep_w[r];
    }
    DirectPlan *d = new (std::nothrow) DirectPlan();
    if (!d) return FRESCO_ERR_OOM;
    d->g = g;
    std::vector<int> row_idx((size_t)n_k);
    for (int64_t q = 0; q < n_k; ++q) {
        const Entry e = entry(mask + q * dim);
        const int c = cell(e);
        row_idx[(size_t)q] = e.neg ? -(c + 1) : c;
    }
    const fresco_status st = precision == FRESCO_F64
                                 ? build_t<double>(d, cols, quads, qbase, s0, w, row_idx)
                                 : build_t<float>(d, cols, quads, qbase, s0, w, row_idx);
    if (st) {
        direct_free(d);
        return st;
    }
    *out = d;
    return FRESCO_OK;
}

template <typename T>
cudaError_t direct_rho(DirectPlan *d, const T *pts, int *err, cudaStream_t s) {
    const DirectGeom &g = d->g;
    const size_t smem = direct_rho_bytes<T>(g);
    const auto kern = g.dim == 2 ? k_direct_rho<T, 2> : k_direct_rho<T, 3>;
    kern<<<g.n_blk, kRhoThreads, smem, s>>>(g, pts, d->cols, d->quads, (Cx<T> *)d->tab, (T *)d->part, err);
    return cudaGetLastError();
}

template <typename T>
cudaError_t direct_mask(DirectPlan *d, double *loss, cudaStream_t s) {
    const DirectGeom &g = d->g;
    k_direct_mask<T><<<d->n_mask_blk, 32 * kMaskCells, 0, s>>>(
        g, g.n_blk, (const T *)d->part, (const T *)d->cell_s0, (const T *)d->cell_w,
        (Cx<T> *)d->rho, (T *)d->dco, d->lpart, d->done, loss);
    return cudaGetLastError();
}

template <typename T>
cudaError_t direct_grad(DirectPlan *d, const double *grad_out, T *grad, cudaStream_t s) {
    const DirectGeom &g = d->g;
    // eight points per block until 32 fill every SM
    const int pj = g.n_points >= 152 * 32 ? 32 : 8;
    const int stage = direct_stage(g, sizeof(T));
    const size_t smem = direct_grad_smem(g, pj, stage, sizeof(T));
    const auto kern = g.dim == 2 ? (pj == 8 ? k_direct_grad<T, 2, 8> : k_direct_grad<T, 2, 32>)
                                 : (pj == 8 ? k_direct_grad<T, 3, 8> : k_direct_grad<T, 3, 32>);
    const int nt = pj == 32 ? kGradThreads<32> : kGradThreads<8>;
    kern<<<(g.n_points + pj - 1) / pj, nt, smem, s>>>(g, d->cols, d->qbase, (const Cx<T> *)d->tab,
                                                       (const T *)d->dco, grad_out, grad, stage);
    return cudaGetLastError();
}

template <typename T>
cudaError_t direct_rho_s(DirectPlan *d, T *rho, T *S, cudaStream_t s) {
    k_direct_rho_s<T><<<(unsigned)((d->n_k + 255) / 256), 256, 0, s>>>(
        d->n_k, d->row_idx, (const Cx<T> *)d->rho, (T)d->g.inv_n, rho, S);
    return cudaGetLastError();
}

#define FRESCO_INST_DIRECT(T)                                                                   \
    template cudaError_t direct_rho<T>(DirectPlan *, const T *, int *, cudaStream_t);           \
    template cudaError_t direct_mask<T>(DirectPlan *, double *, cudaStream_t);                  \
    template cudaError_t direct_grad<T>(DirectPlan *, const double *, T *, cudaStream_t);       \
    template cudaError_t direct_rho_s<T>(DirectPlan *, T *, T *, cudaStream_t);
FRESCO_INST_DIRECT(float)
FRESCO_INST_DIRECT(double)

}  // namespace fresco
