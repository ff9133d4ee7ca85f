// Device-resident L-BFGS minimisation of the FReSCo loss (the optimiser of the main text after
// Eq. 4: L-BFGS with a maximal step size and a backtracking line search).
//
// All vectors (positions, gradients, search direction, the m (s, y) history pairs) stay on the
// device in the plan's precision; every inner product keeps FP64 accuracy (per thread a float
// pair for FP32 vectors, fresco::DotAcc) and is reduced in FP64 in a fixed order. The two-loop
// recursion, the step bound and the first trial point are one launch (or one per pair and
// direction on long vectors), the trial's pair and its products another; the host reads the
// scalars once per trial and decides.
//
// Algorithm (Nocedal & Wright, Numerical Optimization, Alg. 7.4 / 7.5):
//   d = -H g by the two-loop recursion over the stored pairs, H0 = (s.y)/(y.y) I;
//   if g.d >= 0 the history is dropped and d = -g;
//   t0 = min(1, max_step / max_j |d_j|)        (no coordinate moves more than max_step);
//   t = t0, t0/2, ... until L(x + t d) <= L(x) + c1 t g.d (at most max_backtrack halvings);
//   s = t d, y = g(x + t d) - g(x); the pair is stored only if s.y > 0.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "fresco.h"
#include "fresco_internal.h"

namespace {

constexpr int kRedBlocks = 1024;
constexpr int kRedThreads = 256;

// Device scalars; the first SL_READ of them are what the host reads, in one copy per trial.
enum Slot {
    SL_GD = 0,      // g.d
    SL_DMAX,        // max |d_j|
    SL_GMAX,        // max |d_j| of d = -g, where g.d is not below 0
    SL_LOSS,        // loss at the trial point
    SL_SY,          // s.y of the candidate pair
    SL_YY,          // y.y of the candidate pair
    SL_GG,          // g.g at the trial point (or at the start point)
    SL_READ,
    SL_BETA = SL_READ,
    SL_GAMMA,       // s.y / y.y of the newest stored pair at SL_GAMMA + slot; then, likewise per
                    // slot, rho = 1 / s.y and alpha (slots() entries each)
};

// Block sums (or maxima) of NV values; results in thread 0
template <int NV, int NT>
__device__ __forceinline__ void block_reduce(double (&v)[NV], bool is_max) {
    __shared__ double ws[NV][NT / 32];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_xor_sync(0xffffffffu, v[k], o);
            v[k] = is_max ? fmax(v[k], u) : v[k] + u;
        }
        if ((threadIdx.x & 31) == 0) ws[k][threadIdx.x >> 5] = v[k];
    }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double r = ws[k][0];
            for (int w = 1; w < NT / 32; ++w) r = is_max ? fmax(r, ws[k][w]) : r + ws[k][w];
            v[k] = r;
        }
}

// Grid sums (or maxima) of NV values: every block leaves its own, the block that finishes last adds
// them in block order (so the result repeats) and returns true in its thread 0, with the totals in
// v. done is zero before the launch and after it.
template <int NV>
__device__ __forceinline__ bool grid_reduce(double (&v)[NV], bool is_max,
                                            double *__restrict__ part,
                                            unsigned *__restrict__ done) {
    __shared__ bool s_last;
    block_reduce<NV, kRedThreads>(v, is_max);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) part[(int64_t)k * gridDim.x + blockIdx.x] = v[k];
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double r = 0.0;   // (maxima are of absolute values)
        for (int i = threadIdx.x; i < (int)gridDim.x; i += kRedThreads) {
            const double u = __ldcg(part + (int64_t)k * gridDim.x + i);
            r = is_max ? fmax(r, u) : r + u;
        }
        v[k] = r;
    }
    block_reduce<NV, kRedThreads>(v, is_max);
    if (threadIdx.x == 0) *done = 0;
    return threadIdx.x == 0;
}

// *out = a.b
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_dot(const T *__restrict__ a,
                                                     const T *__restrict__ b, int64_t n,
                                                     double *__restrict__ part,
                                                     unsigned *__restrict__ done,
                                                     double *__restrict__ out) {
    fresco::DotAcc<T> acc;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        acc.add(a[i], b[i]);
    double v[1] = {acc.value()};
    if (grid_reduce<1>(v, false, part, done)) *out = v[0];
}

template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_absmax(const T *__restrict__ a, int64_t n,
                                                        double *__restrict__ part,
                                                        unsigned *__restrict__ done,
                                                        double *__restrict__ out) {
    T m = T(0);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(a[i]));
    double v[1] = {(double)m};
    if (grid_reduce<1>(v, true, part, done)) *out = v[0];
}

// The candidate pair of a trial point: s = xt - x, y = gt - g, with s.y, y.y and gt.gt in the same
// pass, and 1 / s.y, s.y / y.y for the slot it would take.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_candidate(
    T *__restrict__ s, T *__restrict__ y, const T *__restrict__ xt, const T *__restrict__ x,
    const T *__restrict__ gt, const T *__restrict__ g, int64_t n, double *__restrict__ part,
    unsigned *__restrict__ done, double *__restrict__ sc, double *__restrict__ gamma,
    double *__restrict__ rho) {
    fresco::DotAcc<T> sy, yy, gg;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const T gi = gt[i];
        const T si = fma(T(-1), x[i], xt[i]), yi = fma(T(-1), g[i], gi);
        s[i] = si;
        y[i] = yi;
        sy.add(si, yi);
        yy.add(yi, yi);
        gg.add(gi, gi);
    }
    double v[3] = {sy.value(), yy.value(), gg.value()};
    if (grid_reduce<3>(v, false, part, done)) {
        sc[SL_SY] = v[0];
        sc[SL_YY] = v[1];
        sc[SL_GG] = v[2];
        // (non-positive products give scale 1; the pair is stored only if s.y > 0)
        *gamma = (v[1] > 0.0 && v[0] > 0.0) ? v[0] / v[1] : 1.0;
        *rho = 1.0 / v[0];
    }
}

// The stored pairs, newest first, passed by value; gamma, rho and alpha lie in the device scalars.
constexpr int kMaxHistory = 64;
struct History {
    int count;
    int slot[kMaxHistory];
    const void *s[kMaxHistory], *y[kMaxHistory];
};

// Two-loop recursion, d = -H g, with g.d, max |d|, and the first trial point xt = x + t d,
// t = min(1, max_step / max |d|); where d is not a descent direction (g.d >= 0, or not a number after
// a pair whose s.y is next to nothing), d = -g instead: a trial runs before the host has seen g.d, and
// must not run on points along a direction that is dropped. For vectors that fit the registers of one cluster: kTlBlocks
// blocks of kTlThreads threads with up to E elements each. Every dot product is a sum per warp and
// one exchange of these over the cluster's shared memory. A launch per vector operation costs more than these
// operations up to about 3e4 elements (20 points of history: 60 launches, 190 us, against one of
// 25 us at 2048 FP64 elements); beyond, k_two_loop_step does one launch per pair and direction.
constexpr int kTlBlocks = 8, kTlThreads = 256;

template <typename T, int E>
__global__ void __cluster_dims__(kTlBlocks, 1, 1) __launch_bounds__(kTlThreads)
    k_two_loop(const __grid_constant__ History hist, const T *__restrict__ g,
               const T *__restrict__ x, T *__restrict__ d, T *__restrict__ xt, int64_t n,
               double max_step, double *__restrict__ sc, const double *__restrict__ gamma,
               const double *__restrict__ rho) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    constexpr int NW = kTlThreads / 32;
    __shared__ double slot[2][NW];
    __shared__ double alpha[kMaxHistory];
    const int64_t i0 = (int64_t)blockIdx.x * kTlThreads + threadIdx.x;
    constexpr int64_t ST = kTlBlocks * kTlThreads;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int phase = 0;
    // sums (or maxima) over the cluster of one value per thread, the same in every thread: every warp
    // leaves its own, and after one cluster barrier every warp adds all of them in the same tree
    // (with block sums first a stored pair's two products took 6.4 us at 2048 FP64 elements, now 4.7)
    auto total = [&](double v, bool is_max) -> double {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_xor_sync(0xffffffffu, v, o);
            v = is_max ? fmax(v, u) : v + u;
        }
        if (lane == 0) slot[phase][wid] = v;
        cl.sync();
        static_assert(kTlBlocks * NW == 64, "two values per lane");
        const double a = *cl.map_shared_rank(&slot[phase][lane & (NW - 1)], lane / NW);
        const double b = *cl.map_shared_rank(&slot[phase][lane & (NW - 1)], lane / NW + 32 / NW);
        v = is_max ? fmax(a, b) : a + b;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_xor_sync(0xffffffffu, v, o);
            v = is_max ? fmax(v, u) : v + u;
        }
        phase ^= 1;   // the other buffer next: a block writes this one again only after the next
        return v;     // exchange, which every block reaches after this read
    };
    // Vectors are loaded one product ahead, so that a product does not begin with a wait for memory
    // (and the pairs' scalars once): a stored pair 4.7 us without, now 3.9.
    __shared__ double srho[kMaxHistory];
    auto load = [&](T (&b)[E], const void *src) {
#pragma unroll
        for (int e = 0; e < E; ++e)
            b[e] = i0 + e * ST < n ? ((const T *)src)[i0 + e * ST] : T(0);
    };
    auto part = [&](const T (&v)[E], const T (&b)[E]) -> double {
        fresco::DotAcc<T> acc;
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (i0 + e * ST < n) acc.add(b[e], v[e]);
        return acc.value();
    };
    auto axpy = [&](T (&v)[E], const T (&b)[E], double c) {
        const T ct = (T)c;
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (i0 + e * ST < n) v[e] = fma(ct, b[e], v[e]);
    };
    const int m = hist.count;
    T v[E], bs[E], by[E], nx[E];
    load(v, g);
    if (m) {
        load(bs, hist.s[0]);
        load(by, hist.y[0]);
    }
    if (threadIdx.x < m) srho[threadIdx.x] = rho[hist.slot[threadIdx.x]];
    const T gm = m ? (T)gamma[hist.slot[0]] : T(1);
    __syncthreads();
    for (int k = 0; k < m; ++k) {              // newest to oldest
        const double p = part(v, bs);
        if (k + 1 < m) {
            load(bs, hist.s[k + 1]);
            load(nx, hist.y[k + 1]);
        }
        const double a = total(p, false) * srho[k];
        if (threadIdx.x == 0) alpha[k] = a;
        axpy(v, by, -a);
        if (k + 1 < m)
#pragma unroll
            for (int e = 0; e < E; ++e) by[e] = nx[e];
    }
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = gm * v[e];
    __syncthreads();
    for (int k = m - 1; k >= 0; --k) {         // oldest to newest (bs, by hold the oldest pair)
        const double p = part(v, by);
        if (k) {
            load(by, hist.y[k - 1]);
            load(nx, hist.s[k - 1]);
        }
        const double b = total(p, false) * srho[k];
        axpy(v, bs, alpha[k] - b);
        if (k)
#pragma unroll
            for (int e = 0; e < E; ++e) bs[e] = nx[e];
    }
    T mx = T(0), gx = T(0);
    fresco::DotAcc<T> acc;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e] = T(-1) * v[e];
        if (i0 + e * ST < n) {
            const T ge = g[i0 + e * ST];
            acc.add(ge, v[e]);
            mx = fmax(mx, fabs(v[e]));
            gx = fmax(gx, fabs(ge));
        }
    }
    const double gd = total(acc.value(), false);
    if (!(gd < 0.0))
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = i0 + e * ST < n ? T(-1) * g[i0 + e * ST] : T(0);
    const double dmax = total((double)(gd < 0.0 ? mx : gx), true);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc[SL_GD] = gd;
        sc[SL_DMAX] = sc[SL_GMAX] = dmax;
    }
    const T t = (T)fmin(1.0, max_step / dmax);
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (i0 + e * ST < n) {
            d[i0 + e * ST] = v[e];
            xt[i0 + e * ST] = fma(t, v[e], x[i0 + e * ST]);
        }
    cl.sync();   // no block leaves while another may still read its shared memory
}

// One step of the recursion over a vector of any length: v = in (+ c a), c = sign (*c0 - *c1),
// times *scale, negated if neg; then, in the same pass, v.b times *mul into *out and, if out_max,
// max |v| and max |b| into its two entries. Null pointers leave their part out.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_two_loop_step(
    T *__restrict__ v, const T *in, const T *__restrict__ a, const double *__restrict__ c0,
    const double *__restrict__ c1, double sign, const double *__restrict__ scale, int neg,
    const T *__restrict__ b, const double *__restrict__ mul, int64_t n, double *__restrict__ part,
    unsigned *__restrict__ done, double *__restrict__ out, double *__restrict__ out_max) {
    const T c = a ? (T)(sign * (*c0 - (c1 ? *c1 : 0.0))) : T(0);
    const T st = scale ? (T)*scale : T(1);
    fresco::DotAcc<T> acc;
    T mx = T(0), bx = T(0);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        T u = in[i];
        if (a) u = fma(c, a[i], u);
        if (scale) u = st * u;
        if (neg) u = T(-1) * u;
        v[i] = u;
        if (b) acc.add(b[i], u);
        mx = fmax(mx, fabs(u));
        if (out_max) bx = fmax(bx, fabs(b[i]));
    }
    double r[1] = {acc.value()};
    if (b && grid_reduce<1>(r, false, part, done)) *out = r[0] * (mul ? *mul : 1.0);
    if (!out_max) return;
    // (a second pass over the blocks' counters: the sum's is zero again only once its last block
    // is done, so the maxima have their own)
    double q[2] = {(double)mx, (double)bx};
    if (grid_reduce<2>(q, true, part + gridDim.x, done + 1)) {
        out_max[0] = q[0];
        out_max[1] = q[1];
    }
}

// z = x + min(1, max_step / max |d|) d; d = -g first where it is not a descent direction (k_two_loop
// has the reason). sc: the device scalars
template <typename T>
__global__ void k_first_trial(T *__restrict__ z, const T *__restrict__ x, T *__restrict__ d,
                              const T *__restrict__ g, int64_t n, double max_step,
                              const double *__restrict__ sc) {
    const bool steepest = !(sc[SL_GD] < 0.0);
    const T tt = (T)fmin(1.0, max_step / (steepest ? sc[SL_GMAX] : sc[SL_DMAX]));
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        T u;
        if (steepest) d[i] = u = T(-1) * g[i];
        else u = d[i];
        z[i] = fma(tt, u, x[i]);
    }
}

// z = a + t * b
template <typename T>
__global__ void k_lincomb(T *__restrict__ z, const T *__restrict__ a, const T *__restrict__ b,
                          int64_t n, double t) {
    const T tt = (T)t;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        z[i] = fma(tt, b[i], a[i]);
}

}  // namespace

struct fresco_lbfgs_s {
    fresco_plan_t plan = nullptr;
    fresco_pair_t pair = nullptr;
    fresco_lbfgs_opts opts{};
    int64_t n = 0;          // N * dim
    size_t es = 4;
    cudaStream_t stream = nullptr;
    int *order = nullptr;   // tile_order: solver position i holds caller point order[i]
    int *tpre = nullptr;    // tile_order: first solver position of every tile's points
    void *xs = nullptr;     // tile_order: the points in solver order
    bool have_order = false;
    void *g = nullptr, *d = nullptr, *xt = nullptr, *gt = nullptr;
    std::vector<void *> S, Y;
    double *scal = nullptr;   // device scalars (Slot)
    double *part = nullptr;   // reduction partials
    unsigned *done = nullptr; // blocks finished in the running reductions
    double *h_scal = nullptr; // pinned host copy of the first SL_READ scalars
    // stored pairs; head is the slot the next candidate pair is written to. There is one slot more
    // than the history holds, so a candidate that is not accepted overwrites no stored pair
    int count = 0, head = 0;
    int64_t evals = 0, iters = 0;
};

namespace {

template <typename T>
struct Ops {
    fresco_lbfgs_s *s;
    int grid() const {
        int64_t b = (s->n + kRedThreads - 1) / kRedThreads;
        return (int)std::max<int64_t>(1, std::min<int64_t>(b, kRedBlocks));
    }
    void dot(const void *a, const void *b, double *out) {
        k_dot<T><<<grid(), kRedThreads, 0, s->stream>>>((const T *)a, (const T *)b, s->n, s->part,
                                                        s->done, out);
    }
    void absmax(const void *a, double *out) {
        k_absmax<T><<<grid(), kRedThreads, 0, s->stream>>>((const T *)a, s->n, s->part, s->done,
                                                           out);
    }
    int slots() const { return s->opts.history + 1; }
    double *gamma() const { return s->scal + SL_GAMMA; }
    double *rho() const { return gamma() + slots(); }
    double *alpha() const { return rho() + slots(); }
    // d = -H g (or -g), g.d, max |d| and the first trial point xt
    void direction(const void *x) {
        History h;
        h.count = s->count;
        for (int k = 0; k < s->count; ++k) {
            h.slot[k] = (s->head - 1 - k + slots()) % slots();
            h.s[k] = s->S[h.slot[k]];
            h.y[k] = s->Y[h.slot[k]];
        }
        const T *g = (const T *)s->g, *xp = (const T *)x;
        T *d = (T *)s->d, *xt = (T *)s->xt;
        constexpr int64_t per = kTlBlocks * kTlThreads;
        if (s->n <= 16 * per) {
            const auto kern = s->n <= 4 * per ? k_two_loop<T, 4> : k_two_loop<T, 16>;
            kern<<<kTlBlocks, kTlThreads, 0, s->stream>>>(h, g, xp, d, xt, s->n, s->opts.max_step,
                                                          s->scal, gamma(), rho());
            return;
        }
        const int m = h.count;
        auto step = [&](const T *in, const T *a, const double *c0, const double *c1, double sign,
                        const double *scale, int neg, const T *b, const double *mul, double *out,
                        double *out_max) {
            k_two_loop_step<T><<<grid(), kRedThreads, 0, s->stream>>>(
                d, in, a, c0, c1, sign, scale, neg, b, mul, s->n, s->part, s->done, out, out_max);
        };
        double *sc = s->scal;
        if (!m) {
            step(g, nullptr, nullptr, nullptr, 1.0, nullptr, 1, g, nullptr, sc + SL_GD,
                 sc + SL_DMAX);
        } else {
            // q = g, with the newest pair's alpha; then q -= alpha y, each with the next product
            step(g, nullptr, nullptr, nullptr, 1.0, nullptr, 0, (const T *)h.s[0],
                 rho() + h.slot[0], alpha(), nullptr);
            for (int k = 0; k < m; ++k) {
                const bool last = k + 1 == m;
                step(d, (const T *)h.y[k], alpha() + k, nullptr, -1.0,
                     last ? gamma() + h.slot[0] : nullptr, 0,
                     (const T *)(last ? h.y[k] : h.s[k + 1]), rho() + h.slot[last ? k : k + 1],
                     last ? sc + SL_BETA : alpha() + k + 1, nullptr);
            }
            for (int k = m - 1; k >= 0; --k) {
                // beta of the next pair goes to the other of two words: this step still reads its own
                double *beta = sc + SL_BETA, *spare = alpha() + slots();
                double *now = (m - 1 - k) & 1 ? spare : beta, *next = (m - 1 - k) & 1 ? beta : spare;
                if (k)
                    step(d, (const T *)h.s[k], alpha() + k, now, 1.0, nullptr, 0,
                         (const T *)h.y[k - 1], rho() + h.slot[k - 1], next, nullptr);
                else
                    step(d, (const T *)h.s[k], alpha() + k, now, 1.0, nullptr, 1, g, nullptr,
                         sc + SL_GD, sc + SL_DMAX);
            }
        }
        k_first_trial<T><<<grid(), kRedThreads, 0, s->stream>>>(xt, xp, d, g, s->n,
                                                                s->opts.max_step, sc);
    }
    // the trial point's candidate pair, in the free slot
    void candidate(const void *x) {
        const int h = s->head;
        k_candidate<T><<<grid(), kRedThreads, 0, s->stream>>>(
            (T *)s->S[h], (T *)s->Y[h], (const T *)s->xt, (const T *)x, (const T *)s->gt,
            (const T *)s->g, s->n, s->part, s->done, s->scal, gamma() + h, rho() + h);
    }
    void lincomb(void *z, const void *a, const void *b, double t) {
        k_lincomb<T><<<grid(), kRedThreads, 0, s->stream>>>((T *)z, (const T *)a, (const T *)b,
                                                            s->n, t);
    }
};

// Solver positions of the tiles: pre[t] = points of tiles 0 .. t-1 (the tiles' record ranges tr
// may have gaps between them), one block scanning the counts 1024 tiles at a time.
__global__ void __launch_bounds__(1024) k_tile_prefix(const int2 *__restrict__ tr, int64_t n_tiles,
                                                      int *__restrict__ pre) {
    __shared__ int warp_tot[32];
    __shared__ int carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t base = 0; base < n_tiles; base += 1024) {
        const int64_t t = base + threadIdx.x;
        const int v = t < n_tiles ? tr[t].y - tr[t].x : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_tot[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int w = warp_tot[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            warp_tot[lane] = w;
        }
        __syncthreads();
        const int incl = x + (wid > 0 ? warp_tot[wid - 1] : 0);
        if (t < n_tiles) pre[t] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry += incl;
        __syncthreads();
    }
}

// order[pre[t] + k] = caller index of the k-th record of tile t (the index a float record
// carries, or the double plans' separate permutation); one warp per tile
template <typename T>
__global__ void __launch_bounds__(256) k_order_from_plan(const void *__restrict__ sorted,
                                                         const int *__restrict__ perm,
                                                         const int2 *__restrict__ tr,
                                                         const int *__restrict__ pre,
                                                         int64_t n_tiles, int *__restrict__ order) {
    const int lane = threadIdx.x & 31;
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < n_tiles;
         t += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int2 r = tr[t];
        const int o = pre[t] - r.x;
        for (int i = r.x + lane; i < r.y; i += 32)
            order[o + i] = sizeof(T) == 4 ? (int)reinterpret_cast<const uint4 *>(sorted)[i].w
                                          : perm[i];
    }
}

// to_solver: y[i] = x[order[i]]; else x[order[i]] = y[i] (points of dim coordinates)
template <typename T>
__global__ void __launch_bounds__(256) k_permute(const int *__restrict__ order, int64_t n,
                                                 int dim, T *__restrict__ x, T *__restrict__ y,
                                                 int to_solver) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = order[i];
        for (int a = 0; a < dim; ++a) {
            if (to_solver) y[i * dim + a] = x[j * dim + a];
            else x[j * dim + a] = y[i * dim + a];
        }
    }
}

fresco_status cerr(cudaError_t e) {
    if (e == cudaSuccess) return FRESCO_OK;
    return e == cudaErrorMemoryAllocation ? FRESCO_ERR_OOM : FRESCO_ERR_CUDA;
}

// The scalars a trial leaves for the host (one copy, one wait).
const double *read_scalars(fresco_lbfgs_s *s) {
    cudaMemcpyAsync(s->h_scal, s->scal, sizeof(double) * SL_READ, cudaMemcpyDeviceToHost,
                    s->stream);
    cudaStreamSynchronize(s->stream);
    return s->h_scal;
}

// loss and gradient of the minimised function: the structure-factor loss, plus the pair term
fresco_status evaluate(fresco_lbfgs_s *s, const void *x, double *loss, void *grad) {
    fresco_status st = fresco_loss_grad(s->plan, x, loss, grad);
    if (st || !s->pair) return st;
    return fresco_pair_energy_grad(s->pair, x, loss, grad, 1);
}

template <typename T>
fresco_status run_impl(fresco_lbfgs_s *s, void *x_caller, int64_t max_iter,
                       fresco_lbfgs_report *rep) {
    Ops<T> op{s};
    const int m = s->opts.history;
    double *sc = s->scal;
    fresco_status st;
    const int dim = s->plan->dim;
    const int64_t np = s->n / dim;
    const unsigned pb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((np + 255) / 256, 152 * 8));
    void *x = x_caller;
    // loss and gradient at the start point
    if (s->opts.tile_order && !s->have_order) {
        // evaluate in caller order once; its tile order becomes the solver's order
        if ((st = evaluate(s, x_caller, sc + SL_LOSS, s->gt))) return st;
        const int64_t nt = s->plan->geom.n_tiles;
        k_tile_prefix<<<1, 1024, 0, s->stream>>>(s->plan->d_tr, nt, s->tpre);
        k_order_from_plan<T><<<pb, 256, 0, s->stream>>>(s->plan->d_sorted, s->plan->d_perm,
                                                         s->plan->d_tr, s->tpre, nt, s->order);
        k_permute<T><<<pb, 256, 0, s->stream>>>(s->order, np, dim, (T *)x_caller, (T *)s->xs, 1);
        k_permute<T><<<pb, 256, 0, s->stream>>>(s->order, np, dim, (T *)s->gt, (T *)s->g, 1);
        s->have_order = true;
        x = s->xs;
    } else if (s->opts.tile_order) {
        k_permute<T><<<pb, 256, 0, s->stream>>>(s->order, np, dim, (T *)x_caller, (T *)s->xs, 1);
        x = s->xs;
        if ((st = evaluate(s, x, sc + SL_LOSS, s->g))) return st;
    } else {
        if ((st = evaluate(s, x, sc + SL_LOSS, s->g))) return st;
    }
    ++s->evals;
    op.dot(s->g, s->g, sc + SL_GG);
    const double *hs = read_scalars(s);
    double fx = hs[SL_LOSS], gg = hs[SL_GG];
    int status = 0;
    // One trial: the loss and gradient at xt and, ahead of the decision on it, the pair it would
    // give, so that the host waits once per trial.
    auto trial = [&]() -> fresco_status {
        const fresco_status e = evaluate(s, s->xt, sc + SL_LOSS, s->gt);
        if (e) return e;
        op.candidate(x);
        read_scalars(s);
        return FRESCO_OK;
    };
    for (int64_t it = 0; it < max_iter; ++it) {
        const double grms = std::sqrt(gg / (double)s->n);
        if (s->opts.gtol > 0.0 && grms < s->opts.gtol) { status = 1; break; }
        if (s->opts.ftol > 0.0 && fx < s->opts.ftol) { status = 2; break; }
        if (!(gg > 0.0)) {   // (a gradient of zeros: no direction, and nothing to evaluate)
            op.absmax(s->g, sc + SL_GMAX);
            if (!(read_scalars(s)[SL_GMAX] > 0.0)) {
                s->count = 0;
                status = 1;
                break;
            }
        }
        op.direction(x);   // two-loop recursion, and xt at the first step length
        if ((st = trial())) return st;
        double gd = hs[SL_GD], dmax = hs[SL_DMAX];
        if (!(gd < 0.0)) {   // not a descent direction: the device has taken the steepest descent
            s->count = 0;
            gd = -gg;
            dmax = hs[SL_GMAX];
        }
        if (!(dmax > 0.0)) { status = 1; break; }
        double t = std::min(1.0, s->opts.max_step / dmax);
        bool accepted = false;
        double ft = fx;
        for (int k = 0;; ++k) {
            ++s->evals;
            ft = hs[SL_LOSS];
            if (std::isfinite(ft) && ft <= fx + s->opts.c1 * t * gd) {
                accepted = true;
                break;
            }
            if (k == s->opts.max_backtrack) break;
            t *= 0.5;
            op.lincomb(s->xt, x, s->d, t);
            if ((st = trial())) return st;
        }
        if (cudaGetLastError() != cudaSuccess) return FRESCO_ERR_CUDA;
        if (!accepted) { status = 4; break; }
        if (hs[SL_SY] > 0.0) {   // store the candidate pair
            s->head = (s->head + 1) % (m + 1);
            s->count = std::min(s->count + 1, m);
        } else if (s->count == m) {
            s->count = m - 1;   // a rejected pair takes the place of the oldest one
        }
        // accept: x = xt, g = gt
        if (cudaMemcpyAsync(x, s->xt, s->es * (size_t)s->n, cudaMemcpyDeviceToDevice,
                            s->stream) != cudaSuccess)
            return FRESCO_ERR_CUDA;
        std::swap(s->g, s->gt);
        fx = ft;
        gg = hs[SL_GG];
        ++s->iters;
        if (it + 1 == max_iter) status = 3;
    }
    if (s->opts.tile_order)   // the result back in caller order
        k_permute<T><<<pb, 256, 0, s->stream>>>(s->order, np, dim, (T *)x_caller, (T *)x, 0);
    if (rep) {
        rep->iterations = s->iters;
        rep->evaluations = s->evals;
        rep->loss = fx;
        rep->grad_rms = std::sqrt(gg / (double)s->n);
        rep->status = status;
    }
    return cerr(cudaGetLastError());
}

void lbfgs_free(fresco_lbfgs_s *s) {
    if (!s) return;
    if (s->stream) cudaStreamSynchronize(s->stream);
    if (s->h_scal) cudaFreeHost(s->h_scal);
    void *bufs[] = {s->g, s->d, s->xt, s->gt, s->scal, s->part, s->done,
                    s->order, s->tpre, s->xs};
    for (void *b : bufs)
        if (b) cudaFree(b);
    for (void *b : s->S)
        if (b) cudaFree(b);
    for (void *b : s->Y)
        if (b) cudaFree(b);
    delete s;
}

}  // namespace

extern "C" {

void fresco_lbfgs_opts_default(fresco_lbfgs_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->history = 10;
    o->max_step = 0.0;
    o->c1 = 1e-4;
    o->max_backtrack = 20;
}

fresco_status fresco_lbfgs_create(fresco_lbfgs_t *out, fresco_plan_t plan,
                                  const fresco_lbfgs_opts *opts) {
    if (!out || !plan) return FRESCO_ERR_ARG;
    *out = nullptr;
    fresco_lbfgs_opts o;
    fresco_lbfgs_opts_default(&o);
    if (opts) o = *opts;
    for (int i = 0; i < 3; ++i)
        if (o.reserved[i]) return FRESCO_ERR_ARG;
    if (o.tile_order != 0 && o.tile_order != 1) return FRESCO_ERR_ARG;
    if (o.history < 1 || o.history > 64 || o.max_backtrack < 0 || o.max_backtrack > 60 ||
        !(o.c1 > 0.0 && o.c1 < 1.0) || o.max_step < 0.0 || o.gtol < 0.0 || o.ftol < 0.0)
        return FRESCO_ERR_ARG;
    fresco_info info;
    fresco_status st = fresco_get_info(plan, &info);
    if (st) return st;
    if (o.max_step == 0.0) {   // a tenth of the mean spacing along the shortest box side
        double lmin = 1e300;
        for (int a = 0; a < info.dim; ++a) lmin = std::min(lmin, plan->box[a]);
        o.max_step = 0.1 * lmin * std::pow((double)info.n_points, -1.0 / info.dim);
    }
    fresco_lbfgs_s *s = new (std::nothrow) fresco_lbfgs_s();
    if (!s) return FRESCO_ERR_OOM;
    if (plan->direct) o.tile_order = 0;   // direct sums have no tiles: the caller's order is as good
    s->plan = plan;
    s->opts = o;
    s->n = info.n_points * info.dim;
    s->es = info.precision == FRESCO_F64 ? 8 : 4;
    s->stream = plan->stream;
    const size_t vb = s->es * (size_t)s->n;
    auto alloc = [&](void **p, size_t bytes) -> bool {
        if (cudaMalloc(p, bytes) != cudaSuccess) {
            cudaGetLastError();
            *p = nullptr;
            return false;
        }
        return true;
    };
    const size_t n_scal = SL_GAMMA + 3 * (size_t)(o.history + 1) + 1;   // (the last: a spare beta)
    bool ok = alloc(&s->g, vb) && alloc(&s->d, vb) && alloc(&s->xt, vb) && alloc(&s->gt, vb) &&
              alloc((void **)&s->scal, sizeof(double) * n_scal) &&
              alloc((void **)&s->part, sizeof(double) * 4 * kRedBlocks) &&
              alloc((void **)&s->done, sizeof(unsigned) * 2) &&
              cudaMallocHost((void **)&s->h_scal, sizeof(double) * SL_READ) == cudaSuccess;
    s->S.assign(o.history + 1, nullptr);
    s->Y.assign(o.history + 1, nullptr);
    for (int i = 0; ok && i <= o.history; ++i) ok = alloc(&s->S[i], vb) && alloc(&s->Y[i], vb);
    if (ok && o.tile_order)
        ok = alloc((void **)&s->order, sizeof(int) * (size_t)info.n_points) && alloc(&s->xs, vb) &&
             alloc((void **)&s->tpre, sizeof(int) * (size_t)plan->geom.n_tiles);
    if (!ok) {
        lbfgs_free(s);
        return FRESCO_ERR_OOM;
    }
    cudaMemsetAsync(s->scal, 0, sizeof(double) * n_scal, s->stream);
    cudaMemsetAsync(s->done, 0, sizeof(unsigned) * 2, s->stream);
    *out = s;
    return FRESCO_OK;
}

fresco_status fresco_lbfgs_run(fresco_lbfgs_t s, void *d_points, int64_t max_iter,
                               fresco_lbfgs_report *report) {
    fresco::clear_pending_error();
    if (!s || !d_points || max_iter < 0) return FRESCO_ERR_ARG;
    s->stream = s->plan->stream;
    if (s->es == 8) return run_impl<double>(s, d_points, max_iter, report);
    return run_impl<float>(s, d_points, max_iter, report);
}

fresco_status fresco_lbfgs_set_pair(fresco_lbfgs_t s, fresco_pair_t p) {
    if (!s) return FRESCO_ERR_ARG;
    s->pair = p;
    return FRESCO_OK;
}

fresco_status fresco_lbfgs_reset(fresco_lbfgs_t s) {
    if (!s) return FRESCO_ERR_ARG;
    s->have_order = false;
    s->count = 0;
    s->head = 0;
    s->iters = 0;
    s->evals = 0;
    return FRESCO_OK;
}

fresco_status fresco_lbfgs_destroy(fresco_lbfgs_t s) {
    lbfgs_free(s);
    return FRESCO_OK;
}

}  // extern "C"
