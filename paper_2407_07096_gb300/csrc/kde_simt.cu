// Plain CUDA-core FP32 form of exact KDE (Sec. 3: K(q) = sum_i k(||q - x_i||), by default the
// Gaussian kernel k(r) = exp(-a r^2); also the exponential and logistic kernels of Sec. 3),
// evaluated over every data point, the "naive" exact method of Sec. 3 / Sec. 6.1.
//
//  * kde_simt_f32_kernel: FP32 direct differences sum_k (q_k - x_k)^2, register-tiled
//    8 queries x 4 points per thread, 64 x 64 pairs per 128-thread block, shared-memory
//    chunks of 32 coordinates fed by cp.async; the exp and the row sum are fused, so no
//    m x n matrix is ever written.
//
// Exponent arithmetic (FP32 form). With c = a log2(e), every term is evaluated as
//     e = 2^(-c d2 - s)      (one fused multiply-add, then ex2.approx)
// where s is a per-row integer shift, so that terms near the row maximum are computed
// with a small argument (accurate) and rows whose every term is below FP32's range
// (a d2 > 87, e.g. d = 128, a = 1) are still represented. s starts at -2^100, which
// forces the first tile through the rescale path; a tile whose FP32 sum exceeds 2^64
// (or is not finite) recomputes with s = ceil(max of its exponents) after rescaling
// the row's accumulators by the exact power of two 2^(s_old - s_new). Terms more than
// 2^-126 below the shift flush to zero (relative contribution < n 2^-126).
//
// Other kernel functions (Sec. 3): the exponential and logistic kernels of r = sqrt(d2),
// in the same shifted form (kernel_fn.cuh).
//
// Squared distances: FP32 FMA chains over blocks of 16 coordinates, block sums added
// (about half the rounding error of a single chain at d >= 32).
// Summation: per thread, FP32 over 16 tiles (64 terms), then FP64; the 16 threads that
// share a row are combined in FP64 with a fixed shuffle pattern; splits of the point set
// are combined in FP64 by kde_combine.cu. Every order is fixed, so results are
// bitwise reproducible.
#include <math.h>

#include "internal.h"
#include "simt_item.cuh"

namespace stagkde {

namespace {

using namespace simt;

// One block per (query tile, contiguous range of point tiles); the partials of query q of
// range s go to part_sum[s * m + q].
template <bool kQResident, bool kOneBlock, int KERN>
__global__ void __launch_bounds__(kThreads, 3)
kde_simt_f32_kernel(const float *__restrict__ xt, int64_t n, int64_t n_tiles, const float *__restrict__ qt, int64_t m,
                    int d_pad, float negc, int64_t tiles_per_split, double *__restrict__ part_sum,
                    float *__restrict__ part_shift) {
    extern __shared__ __align__(16) float smem[];
    const int64_t qtile = blockIdx.x, split = blockIdx.y;
    const int64_t t0 = split * tiles_per_split;
    const int64_t t1 = min(n_tiles, t0 + tiles_per_split);
    const int64_t off = split * m + qtile * kSimtTile;
    simt_item<kQResident, kOneBlock, KERN, false>(
        smem, xt, n, qt + qtile * (int64_t)d_pad * (2 * kSimtTile), d_pad, negc, max((int64_t)0, t1 - t0),
        [t0](int64_t i) { return t0 + i; }, m - qtile * kSimtTile, part_sum + off, part_shift + off);
}

// Row-major n x d -> tile-transposed [tile][d_pad][64], zero padded. kDup: every value
// twice, [tile][d_pad][64][2] (queries). Sets bit 0 of *flag (or NULL) if a value is not
// finite or exceeds 1e15 in magnitude.
template <typename T, bool kDup>
__global__ void to_tiles_kernel(const T *__restrict__ src, int64_t rows, int64_t d, int d_pad,
                                int64_t n_tiles, float *__restrict__ dst, int *flag = nullptr) {
    const int64_t total = n_tiles * d_pad * kSimtTile;
    int bad = 0;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(idx % kSimtTile);
        const int64_t rest = idx / kSimtTile;
        const int k = (int)(rest % d_pad);
        const int64_t t = rest / d_pad;
        const int64_t row = t * kSimtTile + r;
        float v = 0.f;
        if (row < rows && k < d) v = (float)src[row * d + k];
        bad |= !(fabsf(v) <= 1e15f);  // (FP32 values: the same as <= 1e15)
        if (kDup)
            reinterpret_cast<float2 *>(dst)[idx] = make_float2(v, v);
        else
            dst[idx] = v;
    }
    if (flag && bad) atomicOr(flag, 1);
}

// ORs `bit` into *flag when a value is not finite or exceeds 1e15 in magnitude.
__global__ void check_finite_kernel(const float *__restrict__ p, int64_t count, int *flag, int bit) {
    int bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = (double)p[i];
        bad |= !(fabs(v) <= 1e15);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, bit);
}

int grid_for(int64_t total, int threads) {
    return (int)std::min<int64_t>(ceil_div(total, threads), 152 * 16);
}

}  // namespace

int ensure_partials(stag_kde *h, int64_t entries) {
    if (h->part.cap >= entries) return 0;
    ++h->scratch_epoch;
    if (h->part.sum) cudaFree(h->part.sum);
    if (h->part.shift) cudaFree(h->part.shift);
    h->part = Partials{};
    STAG_CUDA_TRY(dev_malloc(&h->part.sum, entries * sizeof(double)));
    STAG_CUDA_TRY(dev_malloc(&h->part.shift, entries * sizeof(float)));
    h->part.cap = entries;
    return 0;
}

int ensure_qt(stag_kde *h, int64_t floats) {
    if (h->qt_cap >= floats) return 0;
    ++h->scratch_epoch;
    if (h->qt) cudaFree(h->qt);
    h->qt = nullptr;
    h->qt_cap = 0;
    STAG_CUDA_TRY(dev_malloc(&h->qt, floats * sizeof(float)));
    h->qt_cap = floats;
    return 0;
}

int launch_check_finite_f32(const float *p, int64_t count, int *dflag, cudaStream_t s, int bit) {
    if (count <= 0) return 0;
    count_launch();
    check_finite_kernel<<<grid_for(count, 256), 256, 0, s>>>(p, count, dflag, bit);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int simt_prepare_points(stag_kde *h, const float *dX) {
    h->d_pad = (int)round_up(h->d, 4);
    h->n_tiles = ceil_div(h->n, kSimtTile);
    const int64_t total = h->n_tiles * h->d_pad * kSimtTile;
    STAG_CUDA_TRY(dev_malloc(&h->xt, total * sizeof(float)));
    count_launch();
    to_tiles_kernel<float, false><<<grid_for(total, 256), 256, 0, h->stream>>>(dX, h->n, h->d, h->d_pad,
                                                                        h->n_tiles, h->xt);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

// Launches the FP32 kernel instance for the handle's operand width and kernel function:
// up to 16 coordinates a pair's squared distance is one chain (no second set of totals).
template <bool kQResident, bool kOneBlock, int KERN>
int launch_simt_inst(const stag_kde *h, dim3 grid, cudaStream_t s, int64_t m, float negc, int64_t tps) {
    auto kern = kde_simt_f32_kernel<kQResident, kOneBlock, KERN>;
    static SmemOptIn opt_in;
    STAG_CUDA_TRY(opt_in((const void *)kern, kMaxSmem));
    kern<<<grid, kThreads, simt_smem(h->d_pad), s>>>(h->xt, h->n, h->n_tiles, h->qt, m, h->d_pad, negc, tps,
                                                     h->part.sum, h->part.shift);
    return 0;
}
template <int KERN>
int launch_simt_kern(const stag_kde *h, dim3 grid, cudaStream_t s, int64_t m, float negc, int64_t tps) {
    if (h->d_pad <= kSumBlock) return launch_simt_inst<true, true, KERN>(h, grid, s, m, negc, tps);
    if (h->d_pad <= kSimtResidentMaxD) return launch_simt_inst<true, false, KERN>(h, grid, s, m, negc, tps);
    return launch_simt_inst<false, false, KERN>(h, grid, s, m, negc, tps);
}
int launch_simt(const stag_kde *h, dim3 grid, cudaStream_t s, int64_t m, int64_t tps) {
    const float negc = (float)(-h->a * 1.4426950408889634);  // -a log2(e)
    switch (h->kernel) {
        case STAG_KDE_KERNEL_EXPONENTIAL:
            return launch_simt_kern<STAG_KDE_KERNEL_EXPONENTIAL>(h, grid, s, m, negc, tps);
        case STAG_KDE_KERNEL_LOGISTIC:
            return launch_simt_kern<STAG_KDE_KERNEL_LOGISTIC>(h, grid, s, m, negc, tps);
        default:
            return launch_simt_kern<STAG_KDE_KERNEL_GAUSSIAN>(h, grid, s, m, negc, tps);
    }
}

// Points per split: about 12 blocks per SM in all, four waves of the three resident ones. (The
// last wave may be nearly empty: n = 70000, m = 10000 gives 1884 blocks on 456 slots, 4.13 waves.
// Another count would regroup the FP32 sums.)
static int64_t choose_tiles_per_split(const stag_kde *h, int64_t q_tiles) {
    const int64_t target_blocks = (int64_t)h->sm_count * 2 * 6;
    int64_t splits = std::max<int64_t>(1, ceil_div(target_blocks, q_tiles));
    splits = std::min<int64_t>(splits, h->n_tiles);
    // keep at least 8 tiles (512 points) per split so per-block set-up stays amortised
    splits = std::min<int64_t>(splits, std::max<int64_t>(1, h->n_tiles / 8));
    return ceil_div(h->n_tiles, splits);
}

int simt_query_f32(stag_kde *h, const float *dQ, int64_t m, double *dOut, cudaStream_t s,
                   int *dflag) {
    const int64_t q_tiles = ceil_div(m, kSimtTile);
    int rc = ensure_qt(h, q_tiles * h->d_pad * kSimtTile * 2);
    if (rc) return rc;
    const int64_t total = q_tiles * h->d_pad * kSimtTile;
    count_launch();
    to_tiles_kernel<float, true><<<grid_for(total, 256), 256, 0, s>>>(dQ, m, h->d, h->d_pad, q_tiles, h->qt, dflag);
    STAG_CUDA_TRY(cudaGetLastError());
    const int64_t tps = choose_tiles_per_split(h, q_tiles);
    const int64_t splits = ceil_div(h->n_tiles, tps);
    rc = ensure_partials(h, splits * m);
    if (rc) return rc;
    if (q_tiles > 0x7fffffff || splits > 65535) return fail(STAG_KDE_EINVAL, "query batch too large");
    dim3 grid((unsigned)q_tiles, (unsigned)splits);
    count_launch();
    prof_start(h, s);
    rc = launch_simt(h, grid, s, m, tps);
    prof_stop(h, s, (double)m * (double)h->n);
    if (rc) return rc;
    STAG_CUDA_TRY(cudaGetLastError());
    return launch_combine(h->part.sum, h->part.shift, m, (int)splits, h->normalise ? 1.0 / (double)h->n : 1.0,
                          dOut, s);
}

int simt_reserve(stag_kde *h, int64_t m) {
    const int64_t q_tiles = ceil_div(m, kSimtTile);
    int rc = ensure_qt(h, q_tiles * h->d_pad * kSimtTile * 2);
    if (rc) return rc;
    const int64_t tps = choose_tiles_per_split(h, q_tiles);
    return ensure_partials(h, ceil_div(h->n_tiles, tps) * m);
}

// Tile-transposed [tile][d_pad][64] back to row-major rows of `stride` coordinates (d, or
// d_pad with the padding).
__global__ void tiles_to_rows_kernel(const float *__restrict__ xt, int64_t n, int64_t stride, int d_pad,
                                     float *__restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * stride;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / stride, k = i % stride;
        out[i] = xt[((row / kSimtTile) * d_pad + k) * kSimtTile + row % kSimtTile];
    }
}

__global__ void subtract_one_kernel(double *__restrict__ v, int64_t count, double one) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        v[i] -= one;
}

int simt_points_rows(stag_kde *h, float *out, int64_t stride, cudaStream_t s) {
    count_launch();
    tiles_to_rows_kernel<<<grid_for(h->n * stride, 256), 256, 0, s>>>(h->xt, h->n, stride, h->d_pad, out);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_subtract(double *v, int64_t count, double one, cudaStream_t s) {
    count_launch();
    subtract_one_kernel<<<grid_for(count, 256), 256, 0, s>>>(v, count, one);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int simt_tiles_from_rows(const stag_kde *h, const float *rows, float *out, cudaStream_t s) {
    const int64_t total = h->n_tiles * h->d_pad * kSimtTile;
    count_launch();
    to_tiles_kernel<float, false><<<grid_for(total, 256), 256, 0, s>>>(rows, h->n, h->d, h->d_pad, h->n_tiles, out);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace stagkde
