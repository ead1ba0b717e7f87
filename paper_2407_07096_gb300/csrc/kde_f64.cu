// FP64 form of exact KDE (Sec. 3: K(q) = sum_i k(||q - x_i||)) for FP64 data: direct
// differences and the kernel function in double precision throughout.
//
// What bounds it: the FP64 pipe. GB300 executes about two FP64 FMAs per SM and clock, so a
// warp's FP64 instruction holds the pipe for 16 clocks; every load, integer operation and
// shared-memory access hides behind it, and the only ways to go faster are to use every SM
// and to spend fewer FP64 instructions per pair. Hence:
//  * work split: a block takes ql queries (the power of two at or above m, at most 32) and
//    a contiguous range of point tiles; its 128 threads are ql queries x 128/ql point
//    lanes, each thread summing up to four points per tile, so a single query still fills
//    whole warps. The point set is split into enough ranges for about eight blocks per
//    SM. (One thread per query over all points, as before, left all but 8 SMs idle at
//    n = m = 1000.)
//  * exp: table-driven (P. T. P. Tang, "Table-driven implementation of the exponential
//    function in IEEE floating-point arithmetic", ACM TOMS 15(2), 1989): 64 powers
//    2^(j/64) in shared memory and a degree-5 Taylor polynomial on |r| <= ln2/128
//    (truncation r^6/720 < 4e-17), 11 FP64 instructions beside the squared distance.
//    Measured below 1 ulp against exp; arguments below -708 (and NaN) take the library's
//    exp, below -745.2 the result is 0 in double.
//  * the last block of a query tile to finish (an atomic ticket that wraps to zero by
//    itself) adds the tile's partial sums in range order, so there is no combine launch.
//  * a query under stream capture takes all ranges in one block per query tile (kOwn): its
//    replays may overlap other queries of the handle, so it uses no shared partial sums.
// Measured, n = m = 1000, d = 2: host call 933 us before (902 us of it the kernel), 70 us
// now; on the device 901 -> 48 us, a replayed capture 900 -> 193 us. n = 1e5, m = 1, d = 8:
// 124.8 ms -> 19 us, replayed 1.60 ms.
// Sums: per thread in index order, then a fixed tree over the point lanes, then the ranges
// in order: bitwise reproducible.
#include <math.h>

#include <algorithm>

#include "internal.h"

namespace stagkde {

namespace {

constexpr int kThreads = 128;
constexpr int kKC = 8;             // coordinates per staged chunk
constexpr int kXS = kKC + 1;       // row stride of the staged points (doubles): odd, so that 16
                                   // lanes on 16 rows hit 16 different bank pairs
constexpr int kMaxQl = 32;         // queries per block at most
constexpr int kMaxPts = 128;       // points per tile at most
constexpr int kTab = 64;
constexpr double kInvL = 0x1.71547652b82fep+6;    // 64 / ln 2
constexpr double kLHi = 0x1.62e42fefa39efp-7;     // ln 2 / 64, and the rest of it below
constexpr double kLLo = 0x1.abc9e3b39803fp-62;

// exp(x) for x <= 0 (the slow branch also takes NaN).
__device__ __forceinline__ double exp_neg(double x, const double *tab) {
    if (!(x > -708.0)) return x < -745.2 ? 0.0 : exp(x);
    const double t = fma(x, kInvL, 0x1.8p52);
    const int n = __double2loint(t);
    const double nf = t - 0x1.8p52;
    const double r = fma(nf, -kLLo, fma(nf, -kLHi, x));
    double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    const double p = fma(q, r * r, r);
    const double T = tab[n & (kTab - 1)];
    const double v = fma(T, p, T);
    return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

template <int KERN>
__device__ __forceinline__ double term64(double a, double d2, const double *tab) {
    if constexpr (KERN == STAG_KDE_KERNEL_GAUSSIAN) {
        return exp_neg(-a * d2, tab);
    } else {
        const double x = a * sqrt(d2);
        if constexpr (KERN == STAG_KDE_KERNEL_EXPONENTIAL)
            return exp_neg(-x, tab);
        else
            return 4.0 / (2.0 + exp(x) + exp(-x));
    }
}

// Sum over the point lanes of each query: lanes of a warp that hold the same query (lane
// distance ql, 2 ql, ...), then the four warps. Every thread calls; the result is valid
// for threads below ql.
__device__ __forceinline__ double reduce_lanes(double s, int ql, double *red) {
    for (int o = 16; o >= ql; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane < ql) red[warp * kMaxQl + lane] = s;
    __syncthreads();
    return threadIdx.x < ql ? (red[threadIdx.x] + red[kMaxQl + threadIdx.x]) +
                                  (red[2 * kMaxQl + threadIdx.x] + red[3 * kMaxQl + threadIdx.x])
                            : 0.0;
}

// R points per thread and tile; ql = 1 << qlog. kOwn: the block takes every range of points
// of its queries in turn and combines them itself, in the order in which the last block of
// the split form does (the same bits), without the handle's partial sums.
template <int KERN, int R, bool kOwn>
__global__ void __launch_bounds__(kThreads)
kde_f64_kernel(const double *__restrict__ X, int64_t n, const double *__restrict__ Q, int64_t m, int d, double a,
               double scale, int qlog, int64_t tiles_per_split, double *part, unsigned *ticket,
               double *__restrict__ out, int *flag) {
    __shared__ double sx[2][kMaxPts * kXS];
    __shared__ double sq[2][kKC * kMaxQl];
    __shared__ double tab[kTab];
    __shared__ double red[4 * kMaxQl];
    __shared__ double own[kOwn ? kMaxQl : 1];
    __shared__ bool last;
    const int ql = 1 << qlog, pl = kThreads >> qlog, pts = pl * R;
    const int tid = threadIdx.x, j = tid & (ql - 1), p = tid >> qlog;
    const int64_t q0 = (int64_t)blockIdx.x * ql;
    const int rows = (int)min((int64_t)ql, m - q0);
    if (tid < kTab) tab[tid] = exp2((double)tid / kTab);
    if (flag && blockIdx.y == 0) {
        // the input check: bit 0 if a query is not finite or beyond 1e15
        int bad = 0;
        for (int64_t e = tid; e < (int64_t)rows * d; e += kThreads) bad |= !(fabs(Q[q0 * d + e]) <= 1e15);
        if (bad) atomicOr(flag, 1);
    }
    const int64_t tiles = (n + pts - 1) / pts;
    const int64_t t0 = kOwn ? 0 : blockIdx.y * tiles_per_split, t1 = kOwn ? tiles : min(tiles, t0 + tiles_per_split);
    const int nch = (d + kKC - 1) / kKC;

    // chunk ch of point tile t, and (unless it is there already) of the queries
    auto load = [&](int st, int64_t t, int ch) {
        const int k0 = ch * kKC, kl = min(kKC, d - k0);
        const int cnt = (int)min((int64_t)pts, n - t * pts);
        const double *src = X + t * pts * (int64_t)d + k0;
        for (int e = tid; e < cnt * kl; e += kThreads) {
            const int r = e / kl, k = e - r * kl;
            const unsigned s = (unsigned)__cvta_generic_to_shared(&sx[st][r * kXS + k]);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src + (int64_t)r * d + k));
        }
        if (nch > 1 || t == t0) {
            // (one chunk: both stages' query halves are filled once, at the first tile)
            for (int e = tid; e < rows * kl; e += kThreads) {
                const int r = e / kl, k = e - r * kl;
                const double *g = Q + (q0 + r) * (int64_t)d + k0 + k;
                const unsigned s = (unsigned)__cvta_generic_to_shared(&sq[st][k * kMaxQl + r]);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(g));
                if (nch == 1) {
                    const unsigned s1 = (unsigned)__cvta_generic_to_shared(&sq[st ^ 1][k * kMaxQl + r]);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s1), "l"(g));
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };

    double s = 0.0, d2[R];
    double acc = 0.0;        // kOwn: the ranges whose number is p modulo pl
    int64_t range = 0, in_range = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) d2[r] = 0.0;
    if (t0 < t1) load(0, t0, 0);
    int st = 0, ch = 0;
    for (int64_t t = t0; t < t1;) {
        const int64_t tn = ch + 1 < nch ? t : t + 1;
        const int cn = ch + 1 < nch ? ch + 1 : 0;
        if (tn < t1) {
            load(st ^ 1, tn, cn);
            asm volatile("cp.async.wait_group 1;\n" ::);
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::);
        }
        __syncthreads();
        const int kl = min(kKC, d - ch * kKC);
        for (int k = 0; k < kl; ++k) {
            const double q = sq[st][k * kMaxQl + j];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const double df = q - sx[st][(p + r * pl) * kXS + k];
                d2[r] = fma(df, df, d2[r]);
            }
        }
        if (cn == 0) {
            const int64_t left = n - t * pts;  // points of the tile
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (p + r * pl < left && j < rows) s += term64<KERN>(a, d2[r], tab);
                d2[r] = 0.0;
            }
            if constexpr (kOwn) {
                if (++in_range == tiles_per_split || t + 1 == t1) {
                    const double v = reduce_lanes(s, ql, red);
                    if (tid < ql) own[tid] = v;
                    __syncthreads();
                    if (p == (range & (pl - 1)) && j < rows) acc += own[j];
                    s = 0.0;
                    in_range = 0;
                    ++range;
                }
            }
        }
        __syncthreads();  // the stage may be refilled
        st ^= 1;
        t = tn;
        ch = cn;
    }
    s = reduce_lanes(kOwn ? acc : s, ql, red);
    if (kOwn || gridDim.y == 1) {
        if (tid < rows) out[q0 + tid] = s * scale;
        return;
    }
    if (tid < rows) part[blockIdx.y * m + q0 + tid] = s;
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicInc(&ticket[blockIdx.x], gridDim.y - 1) == gridDim.y - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    s = 0.0;
    if (j < rows)
        for (int64_t k = p; k < gridDim.y; k += pl) s += __ldcg(&part[k * m + q0 + j]);
    s = reduce_lanes(s, ql, red);
    if (tid < rows) out[q0 + tid] = s * scale;
}

struct Split64 {
    int qlog, r;
    int64_t q_tiles, tps, splits;
};

// ql = the power of two at or above m, at most 32; four points per thread where that
// leaves tiles of at most 128 points. About eight blocks per SM (about as many as are
// resident), each of at least two tiles.
Split64 split64(const stag_kde *h, int64_t m) {
    Split64 s;
    s.qlog = 0;
    while ((1 << s.qlog) < kMaxQl && (1 << s.qlog) < m) ++s.qlog;
    s.r = (kThreads >> s.qlog) * 4 <= kMaxPts ? 4 : 1;
    const int64_t pts = (int64_t)(kThreads >> s.qlog) * s.r;
    s.q_tiles = ceil_div(m, (int64_t)1 << s.qlog);
    const int64_t tiles = ceil_div(h->n, pts);
    const int64_t want = std::max<int64_t>(1, ceil_div((int64_t)h->sm_count * 8, s.q_tiles));
    s.tps = std::max<int64_t>(2, ceil_div(tiles, std::min<int64_t>(want, 65535)));
    s.splits = ceil_div(tiles, s.tps);
    return s;
}

template <int KERN, bool kOwn>
void launch64(const stag_kde *h, const Split64 &sp, const double *dQ, int64_t m, double *dOut, int *dflag,
              cudaStream_t s) {
    const dim3 grid((unsigned)sp.q_tiles, kOwn ? 1u : (unsigned)sp.splits);
    const double scale = h->normalise ? 1.0 / (double)h->n : 1.0;
    if (sp.r == 4)
        kde_f64_kernel<KERN, 4, kOwn><<<grid, kThreads, 0, s>>>(h->x64, h->n, dQ, m, (int)h->d, h->a, scale, sp.qlog,
                                                                sp.tps, h->f64_part, h->tickets, dOut, dflag);
    else
        kde_f64_kernel<KERN, 1, kOwn><<<grid, kThreads, 0, s>>>(h->x64, h->n, dQ, m, (int)h->d, h->a, scale, sp.qlog,
                                                                sp.tps, h->f64_part, h->tickets, dOut, dflag);
}

template <bool kOwn>
void launch64(const stag_kde *h, const Split64 &sp, const double *dQ, int64_t m, double *dOut, int *dflag,
              cudaStream_t s) {
    switch (h->kernel) {
        case STAG_KDE_KERNEL_EXPONENTIAL:
            return launch64<STAG_KDE_KERNEL_EXPONENTIAL, kOwn>(h, sp, dQ, m, dOut, dflag, s);
        case STAG_KDE_KERNEL_LOGISTIC:
            return launch64<STAG_KDE_KERNEL_LOGISTIC, kOwn>(h, sp, dQ, m, dOut, dflag, s);
        default:
            return launch64<STAG_KDE_KERNEL_GAUSSIAN, kOwn>(h, sp, dQ, m, dOut, dflag, s);
    }
}

}  // namespace

// Scratch for every m: more than one range of points only while the query tiles are fewer
// than 8 per SM, and then at most 8 per SM + query tiles blocks, each with at most 32
// partial sums. Held from creation on, so that a query never allocates.
static int64_t f64_partials(const stag_kde *h) { return 2 * (int64_t)h->sm_count * 8 * kMaxQl; }

size_t f64_scratch_bytes(const stag_kde *h) {
    return (size_t)f64_partials(h) * sizeof(double) + (size_t)h->sm_count * 8 * sizeof(unsigned);
}

int f64_set_scratch(stag_kde *h, void *p) {
    h->f64_part = static_cast<double *>(p);
    h->tickets = reinterpret_cast<unsigned *>(h->f64_part + f64_partials(h));
    STAG_CUDA_TRY(cudaMemsetAsync(h->tickets, 0, (size_t)h->sm_count * 8 * sizeof(unsigned), h->stream));
    STAG_CUDA_TRY(cudaEventCreateWithFlags(&h->f64_done, cudaEventDisableTiming));
    return 0;
}

int f64_query(stag_kde *h, const double *dQ, int64_t m, double *dOut, cudaStream_t s, int *dflag) {
    if (h->d > kF64MaxD) return fail(STAG_KDE_EUNSUPPORTED, "FP64 form: d too large");
    const Split64 sp = split64(h, m);
    if (sp.q_tiles > 0x7fffffff) return fail(STAG_KDE_EINVAL, "query batch too large");
    // Queries of one handle queued on several streams share the partial sums: each waits for
    // the one before it. A captured query may be replayed beside any other and cannot wait
    // for it: its blocks combine their own ranges.
    bool own = false;
    if (sp.splits > 1) {
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        STAG_CUDA_TRY(cudaStreamIsCapturing(s, &st));
        own = st != cudaStreamCaptureStatusNone;
    }
    const bool ordered = sp.splits > 1 && !own;
    if (ordered) STAG_CUDA_TRY(cudaStreamWaitEvent(s, h->f64_done, 0));
    count_launch();
    prof_start(h, s);
    if (own)
        launch64<true>(h, sp, dQ, m, dOut, dflag, s);
    else
        launch64<false>(h, sp, dQ, m, dOut, dflag, s);
    prof_stop(h, s, (double)m * (double)h->n);
    STAG_CUDA_TRY(cudaGetLastError());
    if (ordered) STAG_CUDA_TRY(cudaEventRecord(h->f64_done, s));
    return 0;
}

}  // namespace stagkde
