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

#include "f32x2.cuh"
#include "internal.h"
#include "kernel_fn.cuh"

namespace stagkde {

namespace {

constexpr float kShiftFloor = -0x1p100f;  // initial shift (an exact integer)
constexpr float kOverflowGuard = 0x1p64f;
constexpr int kFlushTiles = 16;
constexpr int kSumBlock = 16;  // coordinates per partial chain of a squared distance
constexpr int kThreads = 128;  // threads per block: 8 row groups x 16 point groups
constexpr int kRows = 8;       // query rows per thread
constexpr int kStages = 3;     // ring of staged chunks

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ int clamp_exp(float e) {
    return (int)fminf(fmaxf(e, -4000.f), 4000.f);
}

// Row state: value = (acc64 + acc32) * 2^shift.
struct RowAcc {
    float shift;
    float acc32;
    double acc64;
};

__device__ __forceinline__ void rescale(RowAcc &r, float s_new) {
    int de = clamp_exp(r.shift - s_new);  // <= 0
    r.acc32 = ldexpf(r.acc32, de);
    r.acc64 = ldexp(r.acc64, de);
    r.shift = s_new;
}

using kfn::term;
using kfn::term_log2;

// Adds the four terms k(r_j) 2^-shift (j < valid) to row r.
template <int KERN>
__device__ __forceinline__ void add_terms(RowAcc &r, const float d2[4], float negc, int valid) {
    float ts = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float e = term<KERN>(negc, d2[j], r.shift);
        ts += (j < valid) ? e : 0.f;
    }
    if (!(ts <= kOverflowGuard)) {
        float mx = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < valid) mx = fmaxf(mx, term_log2<KERN>(negc, d2[j]));
        float s_new = fmaxf(ceilf(mx), kShiftFloor);
        if (s_new > r.shift) rescale(r, s_new);
        ts = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float e = term<KERN>(negc, d2[j], r.shift);
            ts += (j < valid) ? e : 0.f;
        }
    }
    r.acc32 += ts;
}

__device__ __forceinline__ void merge(RowAcc &r, double oacc, float oshift) {
    float sm = fmaxf(r.shift, oshift);
    r.acc64 = ldexp(r.acc64, clamp_exp(r.shift - sm)) + ldexp(oacc, clamp_exp(oshift - sm));
    r.shift = sm;
}

// One work item: a query tile of 64 rows (qbase, tile-transposed with every value stored
// twice) against `ntiles` point tiles, tile_at(i) giving the index of the i-th. Rows at or
// past rows_valid are computed on zero padding and not stored; the partials of row r go
// to out_sum[r] and out_shift[r]. `smem`: the block's dynamic shared memory (simt_smem).
//
// What bounds it: the FP32 pipe, two lane operations per coordinate and pair (a packed
// instruction holds it for two cycles). The register tile of 8 rows x 4 points per thread
// spends, per coordinate, 32 packed instructions on 5 shared-memory loads and nothing
// else: the queries are stored duplicated, (q, q), so that a loaded 64-bit register is the
// broadcast operand (building it took 8 moves per 16 packed instructions in the 4 x 4
// tile before). Six shared-memory wavefronts per 64 pipe cycles. The stages are a ring of three
// with one barrier per chunk: the barrier that publishes chunk i also shows that every
// thread is done with chunk i - 1, whose stage then takes chunk i + 2.
// Measured (before: 4 x 4 pairs per thread, 256 threads, two stages): n = 70000, m = 10000,
// d = 784: 42.7 -> 34.8 ms (78 % of the FP32 pipe counting two operations per coordinate;
// 5 % more is the last wave of blocks); exponential kernel, n = m = 1e5, d = 16: 17.6 ->
// 12.1 ms. Four blocks per SM (128 registers) measured 4 % slower at d = 784, the same at
// d = 16. Of the inner loop's form: a remainder loop beside the unrolled one 41.5 ms, steps
// of 4 coordinates 40.9, of 8 38.5, of 16 36.9, with constant-trip copies 34.8.
// A row's arithmetic depends on its 16 point lanes and the order of the tiles only, not on
// how many rows a thread or a block takes.
template <bool kQResident, bool kOneBlock, int KERN, class TileAt>
__device__ __forceinline__ void simt_item(float *__restrict__ smem, const float *__restrict__ xt, int64_t n,
                                          const float *__restrict__ qbase, int d_pad, float negc, int64_t ntiles,
                                          TileAt tile_at, int64_t rows_valid, double *__restrict__ out_sum,
                                          float *__restrict__ out_shift) {
    const int tid = threadIdx.x;
    const int tx = tid & 15;  // point group: points 4*tx .. 4*tx+3 of the tile
    const int ty = tid >> 4;  // query group: rows 8*ty .. 8*ty+7 of the block
    const int nch = kOneBlock ? 1 : (d_pad + kSimtKC - 1) / kSimtKC;
    constexpr int kXStage = kSimtKC * kSimtTile, kQStage = 2 * kXStage;  // floats
    float *sX = smem, *sQ = smem + kStages * kXStage;

    RowAcc row[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) row[i] = RowAcc{kShiftFloor, 0.f, 0.0};

    const int64_t iters = ntiles * nch;
    // chunk lch of the tile with list index lt is the next one to load, into stage ls
    int64_t lt = 0;
    int lch = 0, ls = 0;
    auto load_next = [&]() {
        if (lt < ntiles) {
            const int k0 = lch * kSimtKC;
            const int nvec = min(kSimtKC, d_pad - k0) * (kSimtTile / 4);
            const float *src = xt + (tile_at(lt) * d_pad + k0) * kSimtTile;
            float *dst = sX + ls * kXStage;
            if (nvec == kSimtKC * (kSimtTile / 4)) {  // a whole chunk: constant trip count
#pragma unroll
                for (int v = 0; v < kSimtKC * (kSimtTile / 4); v += kThreads)
                    cp_async16(dst + (v + tid) * 4, src + (v + tid) * 4);
            } else {
                for (int v = tid; v < nvec; v += kThreads) cp_async16(dst + v * 4, src + v * 4);
            }
            if (!kQResident) {
                const float *qs = qbase + (int64_t)k0 * kSimtTile * 2;
                float *qd = sQ + ls * kQStage;
                if (nvec == kSimtKC * (kSimtTile / 4)) {
#pragma unroll
                    for (int v = 0; v < kSimtKC * (kSimtTile / 2); v += kThreads)
                        cp_async16(qd + (v + tid) * 4, qs + (v + tid) * 4);
                } else {
                    for (int v = tid; v < 2 * nvec; v += kThreads) cp_async16(qd + v * 4, qs + v * 4);
                }
            }
            if (++lch == nch) {
                lch = 0;
                ++lt;
            }
        }
        ls = ls + 1 == kStages ? 0 : ls + 1;
        cp_async_commit();
    };

    if (kQResident) {
        const int nvec = d_pad * (kSimtTile / 2);
        for (int v = tid; v < nvec; v += kThreads) cp_async16(sQ + v * 4, qbase + v * 4);
    }
    load_next();
    load_next();

    // squared distances of the 8 x 4 pairs, as packed column pairs (4*tx+0,1) and (+2,3)
    uint64_t d2p[kRows][2];
#pragma unroll
    for (int i = 0; i < kRows; ++i) d2p[i][0] = d2p[i][1] = 0ull;
    const uint64_t negc2 = f2::pack(negc, negc);

    int group = 0, ch = 0, cs = 0;
    int64_t ct = 0;
    for (int64_t it = 0; it < iters; ++it) {
        cp_async_wait<1>();
        __syncthreads();
        load_next();

        const int klen = min(kSimtKC, d_pad - ch * kSimtKC);
        const float *xs = sX + cs * kXStage + tx * 4;
        const float *qs = (kQResident ? sQ + ch * kQStage : sQ + cs * kQStage) + ty * (2 * kRows);
        // blocks of kSumBlock coordinates: each block's squares are summed in a chain of
        // its own and the block sum is added to the pair's total, which keeps the
        // accumulated rounding error of d2 about half that of one chain over all d
        for (int kb = 0; kb < klen; kb += kSumBlock) {
            const int ke = min(klen, kb + kSumBlock);
            uint64_t b2p[kRows][2];
#pragma unroll
            for (int i = 0; i < kRows; ++i) b2p[i][0] = b2p[i][1] = 0ull;
            auto step = [&](int k) {
                const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(xs + k * kSimtTile);
                uint64_t qq[kRows];
#pragma unroll
                for (int i = 0; i < kRows; i += 2) {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(qs + k * 2 * kSimtTile + i * 2);
                    qq[i] = t.x;
                    qq[i + 1] = t.y;
                }
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    const uint64_t df0 = f2::sub(qq[i], xv.x), df1 = f2::sub(qq[i], xv.y);
                    b2p[i][0] = f2::fma(df0, df0, b2p[i][0]);
                    b2p[i][1] = f2::fma(df1, df1, b2p[i][1]);
                }
            };
            // whole blocks unrolled, the rest in steps of 4 (d_pad is a multiple of 4): no
            // remainder loop, whose copies of the body cost 15 instructions per coordinate
            if (ke - kb == kSumBlock) {
#pragma unroll
                for (int k = 0; k < kSumBlock; ++k) step(kb + k);
            } else {
#pragma unroll 1
                for (int k1 = kb; k1 < ke; k1 += 4) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) step(k1 + k);
                }
            }
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                // (one block in all: its sums are the totals)
                d2p[i][0] = kOneBlock ? b2p[i][0] : f2::add(d2p[i][0], b2p[i][0]);
                d2p[i][1] = kOneBlock ? b2p[i][1] : f2::add(d2p[i][1], b2p[i][1]);
            }
        }
        cs = cs + 1 == kStages ? 0 : cs + 1;

        if (++ch == nch) {
            ch = 0;
            const int64_t col0 = tile_at(ct++) * kSimtTile + tx * 4;
            const int valid = (int)max((int64_t)0, min((int64_t)4, n - col0));
            // the common case, a full tile whose terms fit the rows' shifts: no selects and
            // one branch for all rows
            float ts[kRows];
            bool slow = valid < 4;
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                float e0, e1, e2, e3;
                kfn::term2<KERN>(negc, negc2, d2p[i][0], row[i].shift, e0, e1);
                kfn::term2<KERN>(negc, negc2, d2p[i][1], row[i].shift, e2, e3);
                ts[i] = ((e0 + e1) + e2) + e3;
                slow = slow || !(ts[i] <= kOverflowGuard);
            }
            if (slow) {
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    float d2[4];
                    f2::unpack(d2p[i][0], d2[0], d2[1]);
                    f2::unpack(d2p[i][1], d2[2], d2[3]);
                    add_terms<KERN>(row[i], d2, negc, valid);
                }
            } else {
#pragma unroll
                for (int i = 0; i < kRows; ++i) row[i].acc32 += ts[i];
            }
            if (!kOneBlock) {
#pragma unroll
                for (int i = 0; i < kRows; ++i) d2p[i][0] = d2p[i][1] = 0ull;
            }
            if (++group == kFlushTiles) {
                group = 0;
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    row[i].acc64 += (double)row[i].acc32;
                    row[i].acc32 = 0.f;
                }
            }
        }
    }
    cp_async_wait<0>();

#pragma unroll
    for (int i = 0; i < kRows; ++i) {
        row[i].acc64 += (double)row[i].acc32;
        row[i].acc32 = 0.f;
    }
    // Combine the 16 threads of the half-warp that share rows 8*ty..8*ty+7.
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const double oa = __shfl_xor_sync(0xffffffffu, row[i].acc64, off);
            const float os = __shfl_xor_sync(0xffffffffu, row[i].shift, off);
            merge(row[i], oa, os);
        }
    }
    if (tx == 0) {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int r = ty * kRows + i;
            if (r < rows_valid) {
                out_sum[r] = row[i].acc64;
                out_shift[r] = row[i].shift;
            }
        }
    }
}

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
    simt_item<kQResident, kOneBlock, KERN>(
        smem, xt, n, qt + qtile * (int64_t)d_pad * (2 * kSimtTile), d_pad, negc, max((int64_t)0, t1 - t0),
        [t0](int64_t i) { return t0 + i; }, m - qtile * kSimtTile, part_sum + off, part_shift + off);
}

// The grouped recompute of the tensor-core form's flagged queries (kde_tc.cu): work item
// w belongs to query group g (item_off[g] <= w < item_off[g + 1]; groups = *n_groups) and
// covers the group's kept point tiles [s * seg, min(kcount[g], (s + 1) * seg)) of the
// list kept[g * kstride ..], s = w - item_off[g]; each kept tile is `per` consecutive
// 64-point tiles of xt. Query group g is tile g of qt (64 gathered rows). The partials of
// row r go to part_sum[w * 64 + r]. A fixed grid walks the items (counts on the device).
template <bool kQResident, bool kOneBlock, int KERN>
__global__ void __launch_bounds__(kThreads, 3)
kde_simt_f32_list_kernel(const float *__restrict__ xt, int64_t n, int64_t n_tiles, const float *__restrict__ qt,
                         int d_pad, float negc, const int *__restrict__ kept, int64_t kstride,
                         const int *__restrict__ kcount, const int *__restrict__ item_off,
                         const int *__restrict__ n_groups, int seg, int per, double *__restrict__ part_sum,
                         float *__restrict__ part_shift) {
    extern __shared__ __align__(16) float smem[];
    const int G = *n_groups;
    const int total = G > 0 ? item_off[G] : 0;
    for (int w = blockIdx.x; w < total; w += gridDim.x) {
        __syncthreads();  // the previous item's shared-memory reads are done
        int lo = 0, hi = G - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (item_off[mid] <= w)
                lo = mid;
            else
                hi = mid - 1;
        }
        const int g = lo;
        const int k0 = (w - item_off[g]) * seg;
        const int k1 = min(kcount[g], k0 + seg);
        const int *list = kept + (int64_t)g * kstride + k0;
        // the point set's last tile may cover fewer than `per` 64-point tiles; it can only
        // be the list's last entry (the lists ascend), whose tail is enumerated last
        int64_t nt = (int64_t)(k1 - k0) * per;
        if (k1 > k0) nt -= max((int64_t)0, ((int64_t)list[k1 - k0 - 1] + 1) * per - n_tiles);
        simt_item<kQResident, kOneBlock, KERN>(
            smem, xt, n, qt + (int64_t)g * d_pad * (2 * kSimtTile), d_pad, negc, nt,
            [list, per](int64_t i) { return (int64_t)list[i / per] * per + i % per; }, kSimtTile,
            part_sum + (int64_t)w * kSimtTile, part_shift + (int64_t)w * kSimtTile);
    }
}

// Row-major n x d -> tile-transposed [tile][d_pad][64], zero padded. kDup: every value
// twice, [tile][d_pad][64][2] (queries).
template <typename T, bool kDup>
__global__ void to_tiles_kernel(const T *__restrict__ src, int64_t rows, int64_t d, int d_pad,
                                int64_t n_tiles, float *__restrict__ dst) {
    const int64_t total = n_tiles * d_pad * kSimtTile;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(idx % kSimtTile);
        const int64_t rest = idx / kSimtTile;
        const int k = (int)(rest % d_pad);
        const int64_t t = rest / d_pad;
        const int64_t row = t * kSimtTile + r;
        float v = 0.f;
        if (row < rows && k < d) v = (float)src[row * d + k];
        if (kDup)
            reinterpret_cast<float2 *>(dst)[idx] = make_float2(v, v);
        else
            dst[idx] = v;
    }
}

// ORs `bit` into *flag when a value is not finite or exceeds 1e15 in magnitude.
template <typename T>
__global__ void check_finite_kernel(const T *__restrict__ p, int64_t count, int *flag, int bit) {
    int bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double v = (double)p[i];
        bad |= !(fabs(v) <= 1e15);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, bit);
}

// Rows idx[0 .. *count) of the row-major Q, in that order, into the tile-transposed
// query layout (every value twice; rows past *count are zero).
__global__ void gather_rows_tiles_kernel(const float *__restrict__ Q, int64_t d, int d_pad,
                                         const int *__restrict__ idx, const int *__restrict__ count, int64_t m_cap,
                                         float *__restrict__ qt) {
    const int64_t cnt = *count;
    const int64_t total = ((min(cnt, m_cap) + kSimtTile - 1) / kSimtTile) * d_pad * kSimtTile;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e % kSimtTile);
        const int64_t rest = e / kSimtTile;
        const int k = (int)(rest % d_pad);
        const int64_t j = (rest / d_pad) * kSimtTile + r;
        const float v = (j < cnt && k < d) ? Q[(int64_t)idx[j] * d + k] : 0.f;
        reinterpret_cast<float2 *>(qt)[e] = make_float2(v, v);
    }
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
    check_finite_kernel<float><<<grid_for(count, 256), 256, 0, s>>>(p, count, dflag, bit);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int launch_check_finite_f64(const double *p, int64_t count, int *dflag, cudaStream_t s) {
    if (count <= 0) return 0;
    count_launch();
    check_finite_kernel<double><<<grid_for(count, 256), 256, 0, s>>>(p, count, dflag, 1);
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

// Dynamic shared memory of simt_item: the ring of point chunks, and the queries (the whole
// duplicated tile, or a ring of chunks).
constexpr int kChunkBytes = kSimtKC * kSimtTile * 4;
size_t simt_smem(int d_pad) {
    return d_pad <= kSimtResidentMaxD ? kStages * kChunkBytes + (size_t)d_pad * kSimtTile * 8
                                      : (size_t)kStages * 3 * kChunkBytes;
}

template <typename F>
cudaError_t allow_smem(F *kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                std::max<int>(kStages * 3 * kChunkBytes,
                                              kStages * kChunkBytes + kSimtResidentMaxD * kSimtTile * 8));
}

// Launches the FP32 kernel instance for the handle's operand width and kernel function:
// up to 16 coordinates a pair's squared distance is one chain (no second set of totals).
template <bool kQResident, bool kOneBlock, int KERN>
int launch_simt_inst(const stag_kde *h, dim3 grid, cudaStream_t s, int64_t m, float negc, int64_t tps) {
    auto kern = kde_simt_f32_kernel<kQResident, kOneBlock, KERN>;
    // set once per instantiation (before any stream capture can be in progress)
    static const cudaError_t attr = allow_smem(kern);
    STAG_CUDA_TRY(attr);
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

// Number of point-set splits: enough blocks for several waves of 2 blocks per SM.
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
    to_tiles_kernel<float, true><<<grid_for(total, 256), 256, 0, s>>>(dQ, m, h->d, h->d_pad, q_tiles, h->qt);
    STAG_CUDA_TRY(cudaGetLastError());
    if (dflag) {
        rc = launch_check_finite_f32(dQ, m * h->d, dflag, s);
        if (rc) return rc;
    }
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

template <bool kQResident, bool kOneBlock>
static int list_launch_inst(const stag_kde *h, const float *xt, const float *qt, const int *kept, int64_t kstride,
                            const int *kcount, const int *item_off, const int *n_groups, int seg, int per,
                            double *part_sum, float *part_shift, cudaStream_t s) {
    auto kern = kde_simt_f32_list_kernel<kQResident, kOneBlock, STAG_KDE_KERNEL_GAUSSIAN>;
    static const cudaError_t attr = allow_smem(kern);
    STAG_CUDA_TRY(attr);
    const float negc = (float)(-h->a * 1.4426950408889634);  // -a log2(e)
    count_launch();
    kern<<<(unsigned)(h->sm_count * 3), kThreads, simt_smem(h->d_pad), s>>>(
        xt, h->n, h->n_tiles, qt, h->d_pad, negc, kept, kstride, kcount, item_off, n_groups, seg, per, part_sum,
        part_shift);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int simt_list_launch(const stag_kde *h, const float *xt, const float *qt, const int *kept, int64_t kstride,
                     const int *kcount, const int *item_off, const int *n_groups, int seg, int per, double *part_sum,
                     float *part_shift, cudaStream_t s) {
    if (h->d_pad <= kSumBlock)
        return list_launch_inst<true, true>(h, xt, qt, kept, kstride, kcount, item_off, n_groups, seg, per, part_sum,
                                            part_shift, s);
    if (h->d_pad <= kSimtResidentMaxD)
        return list_launch_inst<true, false>(h, xt, qt, kept, kstride, kcount, item_off, n_groups, seg, per,
                                             part_sum, part_shift, s);
    return list_launch_inst<false, false>(h, xt, qt, kept, kstride, kcount, item_off, n_groups, seg, per, part_sum,
                                          part_shift, s);
}

int simt_gather_rows(const stag_kde *h, const float *dQ, const int *idx, const int *count, int64_t m_cap, float *qt,
                     cudaStream_t s) {
    count_launch();
    gather_rows_tiles_kernel<<<grid_for(ceil_div(m_cap, kSimtTile) * h->d_pad * kSimtTile, 256), 256, 0, s>>>(
        dQ, h->d, h->d_pad, idx, count, m_cap, qt);
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
