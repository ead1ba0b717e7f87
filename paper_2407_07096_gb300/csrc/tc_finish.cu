// The end of a tensor-core query (kde_tc.cu): the FP64 combine of the per-range partial
// sums with the per-query error estimate, and the FP32 recompute of the flagged queries
// over the tiles that can matter.
//
// Two launches, whatever the number of instances:
//   fin_combine_kernel  a group of `lpq` lanes per query adds its ranges' partials (a
//                       single thread per query walks them one latency at a time: 724 us
//                       for 17 queries with 1200 ranges each; 32 lanes with eight loads in
//                       flight each: 30 us, a block per query: 7);
//   fin_fix_kernel      returns at once when no query is flagged. Otherwise its blocks
//                       work through the phases below, taking work items from a counter
//                       per phase and waiting for a phase's last item before the next.
//                       Items of a phase are claimed by running blocks only and never
//                       block, so the waits end however few blocks are resident (and are
//                       bounded all the same). Twelve launches of mostly idle kernels took
//                       about 35 us of every query, and 3328 of them most of a 256-instance
//                       batch's time.
// Phases of the recompute (flagged queries in groups of 64, so that every point load serves
// 64 queries, while the tiles that cannot matter are still skipped):
//   count, compact   the flagged queries in query order, each with the bound LB of its
//                    largest exponent, its threshold LB - 64 and, as sort key, the tile
//                    holding LB;
//   sort             stably by that tile (k-d order: queries near the same points become
//                    neighbours; stable on an ordered input, so the groups are
//                    deterministic): one block per instance up to 4096 of them, else
//                    histogram, scan and scatter items per 4096;
//   keep, gather     per group, the union of its members' kept tiles (ub_t >= threshold for
//                    at least one member), and its 64 queries in the plain form's layout;
//   list             the plain form's work item over `seg` kept tiles of one group;
//   combine          per query, the FP64 sum of its group's segments.
// Two queries of one handle that overlap on the device (different streams, a replayed graph
// beside other calls) share this scratch, so their results are undefined; what must not happen
// is an access out of range or a wait that nobody ends. So each call has counters of its own
// (fin_ctl_slot in kde_tc.cu), reads the number of flagged queries once, and every index that is
// read back from the shared scratch is clamped before it is used as one.
// Per query, from the row terms R_t = c ||q - c_t||^2 and the tiles' max radii rho_t (c = a
// log2 e, exponents in log2 units):
//     ub_t = -(max(0, sqrt(R_t) - sqrt(c) rho_t))^2  >= every exponent -c ||q - x||^2 in tile t
//     lb_t = -(sqrt(R_t) + sqrt(c) rho_t)^2          <= the largest exponent in tile t
// (with a 1e-5 relative slack on sqrt(R_t) for rounding), so LB = max_t lb_t bounds the
// row's largest term from below, and a tile with ub_t < LB - 64 holds only terms below
// 2^-64 of it: all of them together change the sum by less than n 2^-64 relative, and the
// tile is skipped. A member evaluates the other members' tiles too: more terms than its own
// bound needs, never fewer.
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "simt_item.cuh"
#include "sm100_ptx.cuh"
#include "tc_finish.h"

namespace stagkde {

namespace {

constexpr float kPruneLog2 = 64.f;
// Queries whose estimated tensor-core error exceeds this are recomputed with the plain
// FP32 form; the estimate bounds the measured error from above (ratio <= ~0.96), so the
// queries kept stay below ~7.2e-5 against the 1e-4 tolerance.
constexpr double kTcErrThreshold = 7.5e-5;
constexpr int kErrTimeout = 1;
// A phase of the recompute gives up when none of its items is finished for this long. What is
// waited for there is arithmetic, an item at a time (0.7 ms at n = 2e5, d = 128, growing with
// n d: about half a second where the points fill the device's memory), so the handle's limit on
// the pairwise kernel's hand-overs, which may be far shorter, does not apply.
constexpr uint64_t kFixStallNs = 10000000000ull;
constexpr int kFixThreads = simt::kThreads;  // 128: four warps
constexpr int kQBlock = 256;                 // queries per block of the flag count
constexpr int kSortChunk = 4096;             // entries per sort item

__device__ __forceinline__ int cexp(float e) { return (int)fminf(fmaxf(e, -4000.f), 4000.f); }

// The entry of the table that owns number v (begin(i) ascends; entries may own none).
template <class Begin>
__device__ __forceinline__ int find_owner(int n, int v, Begin begin) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (begin(mid) <= v)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// FP64 combine of the per-range partials (as kde_combine.cu) plus the per-query error
// estimate of the tensor-core form,
//     est = a * (sum_t S_t w_t) / (sum_t S_t),   w_t = max(2^-21 ||q - c_g|| r_t, beta rho_t^2),
// S_t the query's sum over tile t, r_t that tile's RMS radius, rho_t its largest radius
// and beta = 2^-23 sqrt(MMA steps). The first term (the split products' error grows with
// ||q - c_g|| |x - c_t|) was calibrated on the whole arithmetic over spatially coherent
// tiles, so it covers their FP32 accumulation error too; the second takes over where the
// accumulation error of a tile's outlying points (it grows with ||x - c_t||^2; see
// tc_tile_radius) exceeds it. The epilogue accumulates sum_t S_t w_t. Queries with
// est above the threshold (or an empty sum) are flagged for the plain FP32 form.
__global__ void __launch_bounds__(256)
fin_combine_kernel(const __grid_constant__ FinInst inst0, const FinInst *__restrict__ table, int n_inst,
                   FinCtl *__restrict__ ctl) {
    const FinInst *tab = table ? table : &inst0;
    const FinInst &I = tab[find_owner(n_inst, blockIdx.x, [&](int i) { return tab[i].cblock_begin; })];
    const int tid = threadIdx.x, lpq = I.lpq, qpb = 256 / lpq;
    if (blockIdx.x == 0 && tid < 32) ctl->claim[tid] = ctl->done[tid] = 0;
    const int64_t m = I.m, q0 = (int64_t)(blockIdx.x - I.cblock_begin) * qpb;
    const int64_t j = q0 + tid / lpq;
    const int sub = tid & (lpq - 1), splits = I.splits;
    bool flag = false;
    // (every range of a query has the same shift: it comes from the query's bound, fixed
    // before the first tile; the sums are in units of 2^shift)
    double tot = 0.0, wt = 0.0;
    if (j < m) {
        const double *ps = I.part_sum + j, *pw = I.part_w + j;
        int k = sub;
        for (; k + 3 * lpq < splits; k += 4 * lpq) {  // eight loads in flight
            double s4[4], w4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                s4[u] = ps[(int64_t)(k + u * lpq) * m];
                w4[u] = pw[(int64_t)(k + u * lpq) * m];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                tot += s4[u];
                wt += w4[u];
            }
        }
        for (; k < splits; k += lpq) {
            tot += ps[(int64_t)k * m];
            wt += pw[(int64_t)k * m];
        }
    }
    for (int o = min(lpq, 32) >> 1; o; o >>= 1) {
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
        wt += __shfl_xor_sync(0xffffffffu, wt, o);
    }
    if (lpq == 256) {  // (one query per block: its eight warps)
        __shared__ double part[2][8];
        if ((tid & 31) == 0) {
            part[0][tid >> 5] = tot;
            part[1][tid >> 5] = wt;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 8; ++w) {
                tot += part[0][w];
                wt += part[1][w];
            }
        }
    }
    if (j < m && sub == 0) {
        I.out[j] = ldexp(tot, cexp(I.part_shift[j])) * I.scale;
        // tot is in units of 2^shift, a bound on every term: below 2^-40 the bound was too
        // loose for the fixed shift (terms under 2^-126 of it were flushed)
        const double est = (tot >= 0x1p-40 && !I.qbad[j]) ? I.a * (wt / tot) : INFINITY;
        flag = est > kTcErrThreshold && I.qflag;
        if (I.qflag) I.qflag[j] = flag ? 1 : 0;
    }
    // the bounds have been used: 0 again for the next call (the last block: padding too)
    const int64_t q1 = q0 + qpb >= m ? I.m_pad : q0 + qpb;
    for (int64_t q = q0 + tid; q < q1; q += 256) I.ub[q] = 0u;
    const int c = __syncthreads_count(flag);
    if (c && tid == 0) atomicAdd(I.fix_count, c);
}

// ------------------------------------------------------------------ recompute
// Block-wide exclusive prefix sum of one value per thread (four warps).
__device__ __forceinline__ int block_scan(int v, int *warp_sums, int *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    __syncthreads();
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    int before = inc - v, all = 0;
#pragma unroll
    for (int w = 0; w < kFixThreads / 32; ++w) {
        if (w < warp) before += warp_sums[w];
        all += warp_sums[w];
    }
    *total = all;
    return before;
}

// off[0..n] = exclusive prefix sums of val(0..n-1) (one block).
template <class Val>
__device__ __forceinline__ void scan_to(int n, Val val, int *off, int *warp_sums) {
    int carry = 0;
    for (int base = 0; base < n; base += kFixThreads) {
        const int i = base + threadIdx.x;
        int total;
        const int before = block_scan(i < n ? val(i) : 0, warp_sums, &total);
        if (i < n) off[i] = carry + before;
        carry += total;
    }
    if (threadIdx.x == 0) off[n] = carry;
}

__device__ __forceinline__ int sort_chunks(int F) { return F > kSortChunk ? (F + kSortChunk - 1) / kSortChunk : 0; }

// Flagged query jq's lower bound of its largest exponent, as the arg-max over tiles
// (ties keep the smaller tile), for whole warps: lanes stride over the tiles.
__device__ __forceinline__ void warp_leading_tile(const FinInst &I, float sqc, int64_t jq, float &best, int &bt) {
    const int lane = threadIdx.x & 31, T = (int)I.T;
    best = -INFINITY;
    bt = INT_MAX;
    for (int t0 = lane; t0 < T; t0 += 4 * 32) {
        float rv[4], rho[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = min(t0 + 32 * u, T - 1);
            rv[u] = I.R[(int64_t)t * I.m_pad + jq];
            rho[u] = I.tinfo[(int64_t)t * 4 + 1];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float h2 = sqrtf(rv[u]) * (1.f + 1e-5f) + sqc * rho[u];
            const float lb = -h2 * h2;
            if (t0 + 32 * u < T && lb > best) {  // a lane's tiles ascend
                best = lb;
                bt = t0 + 32 * u;
            }
        }
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int ot = __shfl_xor_sync(0xffffffffu, bt, off);
        if (ob > best || (ob == best && ot < bt)) {
            best = ob;
            bt = ot;
        }
    }
}

// A row number or a position in the sorted arrays, in range whatever was read.
__device__ __forceinline__ int clamp_row(const FinInst &I, uint32_t i) { return (int)min(i, (uint32_t)I.m - 1u); }

// The flagged queries of block b (256 queries) in query order, from position w0 on.
__device__ __forceinline__ void compact_block(const FinInst &I, int b, int w0, int *wcnt) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float sqc = sqrtf(I.c);
    unsigned mask[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int64_t j = (int64_t)b * kQBlock + h * kFixThreads + threadIdx.x;
        mask[h] = __ballot_sync(0xffffffffu, j < I.m && I.qflag[j]);
        if (lane == 0) wcnt[h * 4 + warp] = __popc(mask[h]);
    }
    __syncthreads();
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const int64_t j0 = (int64_t)b * kQBlock + h * kFixThreads + warp * 32;
        int w = w0;
        for (int k = 0; k < h * 4 + warp; ++k) w += wcnt[k];
        const unsigned mk = mask[h];
        if (__popc(mk) >= 8) {
            // many flagged queries in the warp: each lane walks the tiles of its own query
            // (eight row terms in flight; the loads of the warp's queries coalesce)
            if ((mk >> lane) & 1u) {
                const int64_t j = j0 + lane;
                const int T = (int)I.T;
                float best = -INFINITY;
                int bt = 0;
                constexpr int U = 8;
                for (int t0 = 0; t0 < T; t0 += U) {
                    float rv[U], rho[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int t = min(t0 + u, T - 1);
                        rv[u] = I.R[(int64_t)t * I.m_pad + j];
                        rho[u] = I.tinfo[(int64_t)t * 4 + 1];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float h2 = sqrtf(rv[u]) * (1.f + 1e-5f) + sqc * rho[u];
                        const float lb = -h2 * h2;
                        if (t0 + u < T && lb > best) {  // ties keep the smaller tile
                            best = lb;
                            bt = t0 + u;
                        }
                    }
                }
                const int at = clamp_row(I, w + __popc(mk & ((1u << lane) - 1u)));
                I.key[at] = (uint32_t)bt;
                I.val[at] = (uint32_t)j;
                I.thr[j] = best - kPruneLog2;
            }
        } else {
            // few: the warp takes its flagged queries one at a time
            for (unsigned rem = mk; rem; rem &= rem - 1u, ++w) {
                const int64_t jq = j0 + __ffs(rem) - 1;
                float best;
                int bt;
                warp_leading_tile(I, sqc, jq, best, bt);
                if (lane == 0) {
                    const int at = clamp_row(I, w);
                    I.key[at] = (uint32_t)bt;
                    I.val[at] = (uint32_t)jq;
                    I.thr[jq] = best - kPruneLog2;
                }
            }
        }
    }
}

// One radix pass (digit `shift` bits up) over entries [e0, e1) of (ki, vi) -> (ko, vo): the
// block's four warps take contiguous quarters. count fills cnt[warp][digit]; after base
// has turned it into positions, move writes the entries in order (stable).
struct RadixSmem {
    uint32_t cnt[kFixThreads / 32][256];
};
__device__ __forceinline__ void radix_range(int e0, int e1, int &a, int &b) {
    const int warp = threadIdx.x >> 5, q = (((e1 - e0) + 3) / 4 + 31) / 32 * 32;  // whole rounds of 32
    a = min(e1, e0 + warp * q);
    b = min(e1, a + q);
}
__device__ __forceinline__ void radix_count(RadixSmem &r, const uint32_t *ki, int e0, int e1, int shift) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < 4 * 256; i += kFixThreads) (&r.cnt[0][0])[i] = 0u;
    __syncthreads();
    int a, b;
    radix_range(e0, e1, a, b);
    for (int i = a + lane; i < b; i += 32) atomicAdd(&r.cnt[warp][(ki[i] >> shift) & 255u], 1u);
    __syncthreads();
}
__device__ __forceinline__ void radix_move(const FinInst &I, RadixSmem &r, const uint32_t *ki, const uint32_t *vi,
                                           uint32_t *ko, uint32_t *vo, int e0, int e1, int shift) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int a, b;
    radix_range(e0, e1, a, b);
    for (int r0 = a; r0 < b; r0 += 4 * 32) {
        uint32_t k[4], v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = r0 + u * 32 + lane;
            k[u] = i < b ? ki[i] : 0u;
            v[u] = i < b ? vi[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool in = r0 + u * 32 + lane < b;
            const unsigned act = __ballot_sync(0xffffffffu, in);
            if (in) {
                const uint32_t dg = (k[u] >> shift) & 255u;
                const unsigned peers = __match_any_sync(act, dg);
                const int rank = __popc(peers & ((1u << lane) - 1u));
                const int at = clamp_row(I, r.cnt[warp][dg] + rank);
                ko[at] = k[u];
                vo[at] = v[u];
                __syncwarp(act);
                if (rank == 0) r.cnt[warp][dg] += __popc(peers);
            }
            __syncwarp();
        }
    }
}

// Sorts up to kSortChunk entries by all digits (one block).
__device__ __forceinline__ void sort_small(const FinInst &I, int F, RadixSmem &r, int *warp_sums) {
    for (int p = 0; p < I.passes; ++p) {
        uint32_t *ki = p & 1 ? I.ktmp : I.key, *vi = p & 1 ? I.vtmp : I.val;
        uint32_t *ko = p & 1 ? I.key : I.ktmp, *vo = p & 1 ? I.val : I.vtmp;
        radix_count(r, ki, 0, F, 8 * p);
        // positions: digits ascending, warps within a digit
        const int d0 = 2 * threadIdx.x;
        uint32_t c[8];
        int sum = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            c[u] = r.cnt[u & 3][d0 + (u >> 2)];
            sum += (int)c[u];
        }
        int total;
        uint32_t at = (uint32_t)block_scan(sum, warp_sums, &total);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            r.cnt[u & 3][d0 + (u >> 2)] = at;
            at += c[u];
        }
        __syncthreads();
        radix_move(I, r, ki, vi, ko, vo, 0, F, 8 * p);
        __threadfence_block();
        __syncthreads();
    }
}

// Flagged query j in sorted order.
__device__ __forceinline__ int sorted_query(const FinInst &I, int j) {
    return clamp_row(I, (I.passes & 1 ? I.vtmp : I.val)[j]);
}

// The tiles some member of group g may need, in increasing order; their number and the
// group's segment count.
__device__ __forceinline__ void keep_group(const FinInst &I, int g, int F, int *sq, float *sthr, int *wcnt) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = min(64, F - g * 64);
    const float sqc = sqrtf(I.c);
    if (threadIdx.x < rows) {
        const int q = sorted_query(I, g * 64 + threadIdx.x);
        sq[threadIdx.x] = q;
        sthr[threadIdx.x] = I.thr[q];
    }
    __syncthreads();
    int base = 0;
    for (int64_t t0 = 0; t0 < I.T; t0 += kFixThreads) {
        const int64_t t = t0 + threadIdx.x;
        bool keep = false;
        if (t < I.T) {
            const float rho = sqc * I.tinfo[t * 4 + 1];
            // eight members' row terms in flight at a time
            for (int r0 = 0; r0 < rows && !keep; r0 += 8) {
                float rv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) rv[u] = I.R[t * I.m_pad + sq[min(r0 + u, rows - 1)]];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float gap = fmaxf(0.f, sqrtf(rv[u]) * (1.f - 1e-5f) - rho);
                    keep = keep || (r0 + u < rows && -gap * gap >= sthr[r0 + u]);
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) wcnt[warp] = __popc(mask);
        __syncthreads();
        int off = base;
        for (int w = 0; w < warp; ++w) off += wcnt[w];
        if (keep) I.kept[(int64_t)g * I.T + off + __popc(mask & ((1u << lane) - 1u))] = (int)t;
        for (int w = 0; w < kFixThreads / 32; ++w) base += wcnt[w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        I.kcount[g] = base;
        I.items[g] = (base + I.seg - 1) / I.seg;
    }
}

// Group g's queries, tile-transposed, every value twice (rows past the last are zero).
__device__ __forceinline__ void gather_group(const FinInst &I, int g, int F) {
    float2 *dst = reinterpret_cast<float2 *>(I.qt) + (int64_t)g * I.d_pad * kSimtTile;
    for (int e = threadIdx.x; e < I.d_pad * kSimtTile; e += kFixThreads) {
        const int r = e % kSimtTile, k = e / kSimtTile, j = g * 64 + r;
        const float v = j < F && k < I.d ? I.Q[(int64_t)sorted_query(I, j) * I.d + k] : 0.f;
        dst[e] = make_float2(v, v);
    }
}

// Segments a group can have at most; work items of `groups` groups, from their prefix sum.
__device__ __forceinline__ int max_segments(const FinInst &I) { return ((int)I.T + I.seg - 1) / I.seg; }
__device__ __forceinline__ int items_before(const FinInst &I, int g, int groups) {
    return min(max(I.item_off[g], 0), groups * max_segments(I));
}

// Work item w of the instance: kept tiles [s * seg, min(kcount, (s + 1) * seg)) of its group g.
__device__ __forceinline__ void list_item(const FinInst &I, int g, int w, float *smem) {
    const int k0 = min(max(w - I.item_off[g], 0), max_segments(I) - 1) * I.seg;
    const int k1 = min(min(I.kcount[g], (int)I.T), k0 + I.seg);
    const int *list = I.kept + (int64_t)g * I.T + k0;
    const int per_log = I.per_log, per = 1 << per_log;
    // the point set's last tile may cover fewer than `per` 64-point tiles; it can only be
    // the list's last entry (the lists ascend), whose tail is enumerated last
    int64_t nt = (int64_t)(k1 - k0) * per;
    if (k1 > k0) nt -= max((int64_t)0, ((int64_t)list[k1 - k0 - 1] + 1) * per - I.n_tiles);
    const uint64_t last = (uint64_t)I.n_tiles - 1;
    auto tile_at = [list, per_log, per, last](int64_t i) {
        return (int64_t)min((uint64_t)(((int64_t)list[i >> per_log] << per_log) + (i & (per - 1))), last);
    };
    const float *q = I.qt + (int64_t)g * I.d_pad * (2 * kSimtTile);
    double *ps = I.psum + (int64_t)w * kSimtTile;
    float *ph = I.pshift + (int64_t)w * kSimtTile;
    constexpr int kGauss = STAG_KDE_KERNEL_GAUSSIAN;
    if (I.d_pad <= simt::kSumBlock)
        simt::simt_item<true, true, kGauss, true>(smem, I.xkt, I.n, q, I.d_pad, I.negc, nt, tile_at, kSimtTile, ps, ph);
    else if (I.d_pad <= kSimtResidentMaxD)
        simt::simt_item<true, false, kGauss, true>(smem, I.xkt, I.n, q, I.d_pad, I.negc, nt, tile_at, kSimtTile, ps, ph);
    else
        simt::simt_item<false, false, kGauss, true>(smem, I.xkt, I.n, q, I.d_pad, I.negc, nt, tile_at, kSimtTile, ps, ph);
}

// Group g's results: two lanes per query over the group's segments.
__device__ __forceinline__ void combine_group(const FinInst &I, int g, int F, int groups) {
    const int r = threadIdx.x >> 1, sub = threadIdx.x & 1;
    const int w0 = items_before(I, g, groups), w1 = items_before(I, g + 1, groups);
    float smax = -INFINITY;
    for (int w = w0 + sub; w < w1; w += 2) smax = fmaxf(smax, I.pshift[(int64_t)w * 64 + r]);
    smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, 1));
    double tot = 0.0;
    for (int w = w0 + sub; w < w1; w += 2)
        tot += kfn::scale_down(I.psum[(int64_t)w * 64 + r], cexp(I.pshift[(int64_t)w * 64 + r] - smax));
    tot += __shfl_xor_sync(0xffffffffu, tot, 1);
    const int j = g * 64 + r;
    if (sub == 0 && j < F) I.out[sorted_query(I, j)] = w1 > w0 ? ldexp(tot, cexp(smax)) * I.scale : 0.0;
}

__global__ void __launch_bounds__(kFixThreads, 3)
fin_fix_kernel(const __grid_constant__ FinInst inst0, const FinInst *table, int n_inst, int qblocks, int max_passes,
               FinCtl *ctl, int *err, int sms) {
    extern __shared__ __align__(16) float smem[];
    RadixSmem &radix = *reinterpret_cast<RadixSmem *>(smem);  // (the sort's and the lists' phases take turns)
    __shared__ int s_item, s_ok, wcnt[8], warp_sums[kFixThreads / 32], sq[64];
    __shared__ float sthr[64];
    const FinInst *tab = table ? table : &inst0;
    const int tid = threadIdx.x;
    int any = 0;
    for (int i = tid; i < n_inst; i += kFixThreads) any |= *tab[i].fix_count > 0;
    if (!__syncthreads_or(any)) return;
    int *chunk_begin = reinterpret_cast<int *>(ctl + 1), *group_begin = chunk_begin + n_inst + 1,
        *item_begin = group_begin + n_inst + 1, *flagged = item_begin + n_inst + 1;

    // One phase: its N items, whoever takes them, are done when this returns true. `spread`: blocks
    // are placed on the SMs in turn, and the second and third block of an SM let the first ones
    // claim before them (waiting 3 us at most), so that few items lie on different SMs. Whoever asked
    // first took them before, up to three on one SM: the lists of a batch of 7 instances (90
    // items) 157 us, 80 so; of 200 queries on 20000 points in 128 dimensions (160 items) 114, 81 so.
    int phase = 0;
    auto run = [&](int N, auto body, bool spread = false) -> bool {
        const int ph = phase++;
        if (N <= 0) return true;
        if (spread && tid == 0) {
            const int before = (int)blockIdx.x / sms * sms;
            const uint64_t t0 = ptx::globaltimer();
            while (*reinterpret_cast<volatile int *>(&ctl->claim[ph]) < before && ptx::globaltimer() - t0 < 3000)
                __nanosleep(100);
        }
        while (true) {
            __syncthreads();
            if (tid == 0) s_item = atomicAdd(&ctl->claim[ph], 1);
            __syncthreads();
            const int it = s_item;
            if (it >= N) break;
            body(it);
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                atomicAdd(&ctl->done[ph], 1);
            }
        }
        if (tid == 0) {
            uint64_t t0 = ptx::globaltimer();
            int ok = 1, seen = 0;
            while (true) {
                const int done = *reinterpret_cast<volatile int *>(&ctl->done[ph]);
                if (done >= N) break;
                __nanosleep(100);
                const uint64_t now = ptx::globaltimer();
                if (done != seen) {
                    seen = done;
                    t0 = now;
                } else if (now - t0 > kFixStallNs) {
                    atomicExch(err, kErrTimeout);
                    ok = 0;
                    break;
                }
            }
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        return s_ok != 0;
    };
    auto inst_of_qblock = [&](int b) { return find_owner(n_inst, b, [&](int i) { return tab[i].qblock_begin; }); };

    // flag counts per 256 queries; (one more item) where the instances' chunks and groups lie
    bool ok = run(qblocks + 1, [&](int it) {
        if (it < qblocks) {
            const FinInst &I = tab[inst_of_qblock(it)];
            if (!I.qflag) return;
            const int b = it - I.qblock_begin;
            int c = 0;
            for (int h = 0; h < 2; ++h) {
                const int64_t j = (int64_t)b * kQBlock + h * kFixThreads + tid;
                c += __syncthreads_count(j < I.m && I.qflag[j]);
            }
            if (tid == 0) I.bcnt[b] = c;
        } else {
            // (a thread scans the entries that it has written)
            for (int i = tid; i < n_inst; i += kFixThreads)
                flagged[i] = (int)min((int64_t)max(*tab[i].fix_count, 0), tab[i].m);
            scan_to(n_inst, [&](int i) { return sort_chunks(flagged[i]); }, chunk_begin, warp_sums);
            scan_to(n_inst, [&](int i) { return (flagged[i] + 63) / 64; }, group_begin, warp_sums);
        }
    });
    ok = ok && run(qblocks, [&](int it) {
        const FinInst &I = tab[inst_of_qblock(it)];
        const int b = it - I.qblock_begin;
        if (!I.qflag || I.bcnt[b] == 0) return;
        int c = 0, w0;
        for (int i = tid; i < b; i += kFixThreads) c += I.bcnt[i];
        block_scan(c, warp_sums, &w0);
        compact_block(I, b, w0, wcnt);
    });
    ok = ok && run(n_inst, [&](int i) {
        const int F = flagged[i];
        if (F > 0 && F <= kSortChunk) sort_small(tab[i], F, radix, warp_sums);
    });
    const int chunks = ok ? chunk_begin[n_inst] : 0;
    for (int p = 0; p < max_passes && ok && chunks > 0; ++p) {
        // (instance, chunk) of an item; digit p of an instance that has fewer is left alone
        auto each = [&](int it, auto body) {
            const int i = find_owner(n_inst, it, [&](int k) { return chunk_begin[k]; });
            const FinInst &I = tab[i];
            if (p >= I.passes) return;
            const int F = flagged[i], nb = sort_chunks(F), ch = it - chunk_begin[i];
            body(I, nb, ch, ch * kSortChunk, min(F, (ch + 1) * kSortChunk));
        };
        ok = run(chunks, [&](int it) {
            each(it, [&](const FinInst &I, int nb, int ch, int e0, int e1) {
                radix_count(radix, p & 1 ? I.ktmp : I.key, e0, e1, 8 * p);
                for (int dg = tid; dg < 256; dg += kFixThreads)
                    I.hist[dg * nb + ch] =
                        radix.cnt[0][dg] + radix.cnt[1][dg] + radix.cnt[2][dg] + radix.cnt[3][dg];
            });
        });
        ok = ok && run(n_inst, [&](int i) {
            const FinInst &I = tab[i];
            const int nb = sort_chunks(flagged[i]);
            if (nb == 0 || p >= I.passes) return;
            // exclusive scan in place: each thread a run of two digits' entries
            uint32_t *h = I.hist + (int64_t)tid * 2 * nb;
            int sum = 0, total;
            for (int e = 0; e < 2 * nb; ++e) sum += (int)h[e];
            uint32_t at = (uint32_t)block_scan(sum, warp_sums, &total);
            for (int e = 0; e < 2 * nb; ++e) {
                const uint32_t v = h[e];
                h[e] = at;
                at += v;
            }
        });
        ok = ok && run(chunks, [&](int it) {
            each(it, [&](const FinInst &I, int nb, int ch, int e0, int e1) {
                const uint32_t *ki = p & 1 ? I.ktmp : I.key, *vi = p & 1 ? I.vtmp : I.val;
                radix_count(radix, ki, e0, e1, 8 * p);
                for (int dg = tid; dg < 256; dg += kFixThreads) {
                    uint32_t at = I.hist[dg * nb + ch];
                    for (int w = 0; w < 4; ++w) {
                        const uint32_t v = radix.cnt[w][dg];
                        radix.cnt[w][dg] = at;
                        at += v;
                    }
                }
                __syncthreads();
                radix_move(I, radix, ki, vi, p & 1 ? I.key : I.ktmp, p & 1 ? I.val : I.vtmp, e0, e1, 8 * p);
            });
        });
    }
    phase = 3 + 3 * max_passes;  // (the same numbers whether or not anything was in chunks)
    const int groups = ok ? group_begin[n_inst] : 0;
    auto inst_of_group = [&](int g) { return find_owner(n_inst, g, [&](int i) { return group_begin[i]; }); };
    ok = ok && run(2 * groups, [&](int it) {
        const int gg = it < groups ? it : it - groups, i = inst_of_group(gg);
        const FinInst &I = tab[i];
        if (it < groups)
            keep_group(I, gg - group_begin[i], flagged[i], sq, sthr, wcnt);
        else
            gather_group(I, gg - group_begin[i], flagged[i]);
    });
    ok = ok && run(n_inst, [&](int i) {
        const FinInst &I = tab[i];
        const int G = group_begin[i + 1] - group_begin[i];
        if (G > 0) scan_to(G, [&](int g) { return I.items[g]; }, I.item_off, warp_sums);
    });
    ok = ok && run(1, [&](int) {
        scan_to(n_inst,
                [&](int i) {
                    const int G = group_begin[i + 1] - group_begin[i];
                    return G > 0 ? items_before(tab[i], G, G) : 0;
                },
                item_begin, warp_sums);
    });
    const int items = ok ? item_begin[n_inst] : 0;
    int li = -1, lg = -1;  // instance and group of this block's last item
    ok = ok && run(items, [&](int it) {
        if (li < 0 || it < item_begin[li] || it >= item_begin[li + 1]) {
            li = find_owner(n_inst, it, [&](int k) { return item_begin[k]; });
            lg = -1;
        }
        const FinInst &I = tab[li];
        const int w = it - item_begin[li];
        if (lg < 0 || w < I.item_off[lg] || w >= I.item_off[lg + 1])
            lg = find_owner(group_begin[li + 1] - group_begin[li], w, [&](int k) { return I.item_off[k]; });
        list_item(I, lg, w, smem);
    }, true);
    if (ok)
        run(groups, [&](int gg) {
            const int i = inst_of_group(gg);
            combine_group(tab[i], gg - group_begin[i], flagged[i], group_begin[i + 1] - group_begin[i]);
        });
}

// Kept point tiles per work item: at least eight 64-point tiles (the per-item set-up is
// then amortised), and at most 64 items per group.
int group_seg(int64_t T, int BN) { return (int)std::max<int64_t>(8 * 64 / BN, ceil_div(T, 64)); }

}  // namespace

int64_t fin_scratch_bytes(int64_t m, int64_t T, int BN, FinInst *inst, void *base) {
    const int64_t mm = std::max<int64_t>(m, 1);
    const int64_t G = ceil_div(mm, 64), B = ceil_div(mm, kQBlock);
    const int64_t items = G * ceil_div(T, group_seg(T, BN));
    int64_t off = 0;
    auto take = [&](int64_t bytes) {
        const int64_t o = off;
        off += round_up(bytes, 256);
        return static_cast<char *>(base) + o;
    };
    FinInst f{};
    f.key = (uint32_t *)take(mm * 4);
    f.ktmp = (uint32_t *)take(mm * 4);
    f.val = (uint32_t *)take(mm * 4);
    f.vtmp = (uint32_t *)take(mm * 4);
    f.hist = (uint32_t *)take(256 * ceil_div(mm, kSortChunk) * 4);
    f.thr = (float *)take(mm * 4);
    f.qflag = (int *)take(mm * 4);
    f.bcnt = (int *)take(B * 4);
    f.kept = (int *)take(G * T * 4);
    f.kcount = (int *)take(G * 4);
    f.items = (int *)take(G * 4);
    f.item_off = (int *)take((G + 1) * 4);
    f.psum = (double *)take(items * 64 * 8);
    f.pshift = (float *)take(items * 64 * 4);
    if (inst) {
        inst->key = f.key;
        inst->ktmp = f.ktmp;
        inst->val = f.val;
        inst->vtmp = f.vtmp;
        inst->hist = f.hist;
        inst->thr = f.thr;
        inst->qflag = f.qflag;
        inst->bcnt = f.bcnt;
        inst->kept = f.kept;
        inst->kcount = f.kcount;
        inst->items = f.items;
        inst->item_off = f.item_off;
        inst->psum = f.psum;
        inst->pshift = f.pshift;
        inst->seg = group_seg(T, BN);
        inst->per_log = BN == 128 ? 1 : 2;  // 64-point tiles per tile: 2 or 4
        static_assert(kSimtTile == 64, "tiles of 128 or 256 points");
        inst->passes = 1;
        while (inst->passes < 4 && ((int64_t)1 << (8 * inst->passes)) < T) ++inst->passes;
    }
    return off;
}

void fin_number(FinInst *inst, int sm_count, int cblock, int qblock, int *cblocks, int *qblocks) {
    // more lanes per query while that leaves each at least four ranges and the queries alone
    // do not fill the chip
    int lpq = 1;
    while (lpq < 32 && lpq * 8 <= inst->splits && inst->m * lpq < (int64_t)sm_count * 1024) lpq *= 2;
    // few queries with hundreds of ranges each: a whole block per query (17 queries with 1200
    // ranges: 30 -> 7 us)
    if (lpq == 32 && inst->splits >= 256 && inst->m <= 2 * (int64_t)sm_count) lpq = 256;
    inst->lpq = lpq;
    inst->cblock_begin = cblock;
    inst->qblock_begin = qblock;
    *cblocks = (int)ceil_div(inst->m, 256 / lpq);
    *qblocks = (int)ceil_div(inst->m, kQBlock);
}

int fin_launch(const FinInst &inst0, const FinInst *table, int n_inst, int cblocks, int qblocks, int max_passes,
               int max_d_pad, int64_t max_items, bool recompute, FinCtl *ctl, int *err, int sm_count,
               cudaStream_t s) {
    count_launch();
    fin_combine_kernel<<<(unsigned)cblocks, 256, 0, s>>>(inst0, table, n_inst, ctl);
    STAG_CUDA_TRY(cudaGetLastError());
    if (!recompute) return 0;
    static SmemOptIn opt_in;
    STAG_CUDA_TRY(opt_in((const void *)fin_fix_kernel, simt::kMaxSmem));
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count * 3, max_items));
    count_launch();
    // (the ring's layout follows each instance's d_pad; the widest layout is the streamed one)
    const size_t smem = std::max(simt::simt_smem(std::min(max_d_pad, kSimtResidentMaxD)), simt::simt_smem(max_d_pad));
    fin_fix_kernel<<<grid, kFixThreads, smem, s>>>(inst0, table, n_inst, qblocks, max_passes, ctl, err,
                                                   sm_count);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace stagkde
