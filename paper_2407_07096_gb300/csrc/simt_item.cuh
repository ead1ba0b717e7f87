// The plain FP32 form's work item, shared by its own kernel (kde_simt.cu) and by the
// recompute of the tensor-core form's flagged queries (tc_finish.cu): 64 queries against a
// list of 64-point tiles, register-tiled FP32 direct differences with the kernel function
// and the row sums fused.
#pragma once
#include <math.h>

#include "f32x2.cuh"
#include "internal.h"
#include "kernel_fn.cuh"

namespace stagkde {
namespace simt {

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
    r.acc32 = de > -126 ? r.acc32 * __int_as_float((127 + de) << 23) : 0.f;
    r.acc64 = kfn::scale_down(r.acc64, de);
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
    r.acc64 = kfn::scale_down(r.acc64, clamp_exp(r.shift - sm)) + kfn::scale_down(oacc, clamp_exp(oshift - sm));
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
// kListed: tile_at reads a list in global memory (its next entry is fetched ahead).
template <bool kQResident, bool kOneBlock, int KERN, bool kListed, class TileAt>
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
    // chunk lch of the tile with list index lt is the next one to load, into stage ls;
    // kListed: that tile, and the one after it on its way
    int64_t lt = 0, ltile = kListed && ntiles > 0 ? tile_at(0) : 0, ltile1 = kListed && ntiles > 1 ? tile_at(1) : 0;
    int lch = 0, ls = 0;
    auto load_next = [&]() {
        if (lt < ntiles) {
            const int k0 = lch * kSimtKC;
            const int nvec = min(kSimtKC, d_pad - k0) * (kSimtTile / 4);
            const float *src = xt + ((kListed ? ltile : tile_at(lt)) * d_pad + k0) * kSimtTile;
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
                if (kListed) {
                    ltile = ltile1;
                    if (lt + 1 < ntiles) ltile1 = tile_at(lt + 1);
                }
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
            // (only the point set's last tile is ragged, and it is the last of any list)
            const int64_t col0 = ++ct < ntiles && kListed ? 0 : tile_at(ct - 1) * kSimtTile + tx * 4;
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

// Dynamic shared memory of simt_item: the ring of point chunks, and the queries (the whole
// duplicated tile, or a ring of chunks).
constexpr int kChunkBytes = kSimtKC * kSimtTile * 4;
inline size_t simt_smem(int d_pad) {
    return d_pad <= kSimtResidentMaxD ? kStages * kChunkBytes + (size_t)d_pad * kSimtTile * 8
                                      : (size_t)kStages * 3 * kChunkBytes;
}

constexpr int kMaxSmem =
    std::max(kStages * 3 * kChunkBytes, kStages * kChunkBytes + kSimtResidentMaxD * kSimtTile * 8);

}  // namespace simt
}  // namespace stagkde
