// Weighted subset sums: the estimator that random sampling (every point weighted n/s)
// and the CKNS scheme (weights 2^i on hashed candidates) evaluate (Sec. 3.1),
//     out[j] = sum_{p = off[j] .. off[j+1]-1} w[p] k(||q_j - x_{idx[p]}||),
// with each query's own list of (point index, weight) pairs, gather-fed.
//
// Layout and work split: the point set is kept row-major, rows padded to a multiple of
// four coordinates (FP32, built once per handle from the plain form's tiled copy), so a
// list entry is one contiguous, 16-byte aligned row. One warp owns one query at a time
// (grid-stride over queries); each lane takes every 32nd entry of the list, forms d2 by
// direct differences in FP32 and adds w k(r) 2^-s with its own integer shift s
// (kernel_fn.cuh; rescaled exactly by a power of two when a term would exceed 2^64),
// flushing to FP64 every 16 terms. The 32 lanes are merged in FP64 with a fixed shuffle
// order, so results are deterministic.
//
// What bounds it: moving the rows, d*4 bytes per entry from L2 when X fits there (beside 8
// + 4 bytes of index and weight from HBM). A lane that loads its own row touches 32 rows
// with every load instruction, and L1 looks up one line per clock: at d = 16 that alone is
// 128 clocks per 32 entries. So rows of at most 16 coordinates are staged: four lanes copy
// 64 contiguous bytes of one row (cp.async into a per-warp ring of three stages of 32
// rows), which touches eight rows per instruction, and each lane then reads its own row
// from shared memory (16-byte pieces swizzled by row, free of bank conflicts). The stages
// run ahead across queries: indices are loaded one stage before their rows are copied, the
// next query's offsets one query before, so the latencies of the list, the rows and the
// arithmetic of different stages overlap even for lists of a few dozen entries.
#include <math.h>
#include <stddef.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "kernel_fn.cuh"

namespace stagkde {

namespace {

constexpr int kSubsetWarps = 8;  // warps per block
constexpr float kShiftInit = -0x1p100f;
constexpr float kGuard = 0x1p64f;
constexpr int kFlush = 16;
constexpr int64_t kSubsetMaxD = 1536;
constexpr int kSubStages = 3;    // stages of a warp's ring
constexpr int kSubChunk = 16;    // coordinates a stage holds per row (one summation block)

__device__ __forceinline__ int clampe(float e) { return (int)fminf(fmaxf(e, -4000.f), 4000.f); }
__device__ __forceinline__ void copy4(void *smem, const void *g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g));
}

// Any number of coordinates: every lane gathers its own rows, 16 bytes at a time (dp = d
// rounded up to 4, the padding zero), and all of a row's loads are in flight together. From
// 17 coordinates on a row fills more than half a cache line, so staging it in chunks gains
// less (d = 64, 1000 lists of 3000: 537 us, staged 478) than the chunks' serial copies cost
// short lists (d = 100, 6000 lists of 50: 42 us, staged 126). Padded rows make every d a
// whole number of 16-byte loads (d = 30, 100 lists of 2000: 323 -> 136 us).
template <int KERN>
__global__ void __launch_bounds__(32 * kSubsetWarps)
kde_subset_kernel(const float *__restrict__ X, int64_t n, int d, int dp, const float *__restrict__ Q, int64_t m,
                  const int64_t *__restrict__ off, const int64_t *__restrict__ idx, const float *__restrict__ W,
                  float negc, double scale, double *__restrict__ out) {
    extern __shared__ __align__(16) float sq_all[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float *sq = sq_all + warp * dp;
    const int pieces = dp / 4;
    const int64_t warps = (int64_t)gridDim.x * kSubsetWarps;
    for (int64_t j = (int64_t)blockIdx.x * kSubsetWarps + warp; j < m; j += warps) {
        __syncwarp();
        for (int k = lane; k < dp; k += 32) sq[k] = k < d ? Q[j * d + k] : 0.f;
        __syncwarp();
        const int64_t p0 = off[j], p1 = off[j + 1];
        float shift = kShiftInit, acc32 = 0.f;
        double acc64 = 0.0;
        int cnt = 0;
        for (int64_t p = p0 + lane; p < p1; p += 32) {
            const int64_t i = idx[p];
            if (i < 0 || i >= n) continue;  // out-of-range entries contribute nothing
            const float w = W ? W[p] : 1.f;
            const float *x = X + i * dp;
            // FP32 chains over blocks of 16 coordinates, block sums added (the plain
            // form's order and error bound; padding adds (0 - 0)^2)
            float d2 = 0.f;
            const float4 *xv4 = reinterpret_cast<const float4 *>(x);
            const float4 *qv4 = reinterpret_cast<const float4 *>(sq);
            auto add4 = [](float b2, const float4 &qv, const float4 &xv) {
                float t = qv.x - xv.x;
                b2 = fmaf(t, t, b2);
                t = qv.y - xv.y;
                b2 = fmaf(t, t, b2);
                t = qv.z - xv.z;
                b2 = fmaf(t, t, b2);
                t = qv.w - xv.w;
                return fmaf(t, t, b2);
            };
            // (a block's loads are issued before any is used; two blocks' at a time measured 13 %
            // faster on few long lists, and 15 % slower on many short ones, by their registers)
            int v = 0;
#pragma unroll 1
            for (; v + 4 <= pieces; v += 4) {
                float4 xv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) xv[u] = xv4[v + u];
                float b2 = 0.f;
#pragma unroll
                for (int u = 0; u < 4; ++u) b2 = add4(b2, qv4[v + u], xv[u]);
                d2 += b2;
            }
            float b2 = 0.f;
            for (; v < pieces; ++v) b2 = add4(b2, qv4[v], xv4[v]);
            d2 += b2;
            float e = w * kfn::term<KERN>(negc, d2, shift);
            if (!(fabsf(e) <= kGuard)) {
                // first term, or one far above the current shift: move the shift up
                const float s_new = fmaxf(ceilf(kfn::term_log2<KERN>(negc, d2)), kShiftInit);
                if (s_new > shift) {
                    const int de = clampe(shift - s_new);
                    acc32 = de > -126 ? acc32 * __int_as_float((127 + de) << 23) : 0.f;
                    acc64 = kfn::scale_down(acc64, de);
                    shift = s_new;
                }
                e = w * kfn::term<KERN>(negc, d2, shift);
            }
            acc32 += e;
            if (++cnt == kFlush) {
                acc64 += (double)acc32;
                acc32 = 0.f;
                cnt = 0;
            }
        }
        acc64 += (double)acc32;
        // merge the lanes: common shift = the largest, fixed butterfly order
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            const double oa = __shfl_xor_sync(0xffffffffu, acc64, o);
            const float os = __shfl_xor_sync(0xffffffffu, shift, o);
            const float sm = fmaxf(shift, os);
            acc64 = kfn::scale_down(acc64, clampe(shift - sm)) + kfn::scale_down(oa, clampe(os - sm));
            shift = sm;
        }
        if (lane == 0) out[j] = ldexp(acc64, clampe(shift)) * scale;
    }
}

// Rows of at most 16 coordinates, staged. The instructions around the arithmetic decide. The
// query stays in registers, the consumer counts its own groups of 32 entries (a query's first
// stage carries its number and its group count), copies take their size instead of a branch,
// and a lane without an entry computes and adds 0. It copies a row that is its warp's own: with
// row 0 for all of them every warp of the chip met on one line of L2. Without that, 1e5 lists of
// 100 entries, n = 1e6, d = 16: 622 -> 125 us; 1e5 lists of 3, n = 1e5, d = 5: 589 -> 84; 3000
// lists of 700 of which half is out of range, n = 1e6, d = 4: 231 -> 23. (Predicating the copies
// instead is 1 to 2 % faster with weights, 3 % slower on long lists without.)
// Measured, n = 1e6, d = 16, 1e5 lists of 1000 weighted entries: 1417 us with every lane loading
// its own row, 1203 with staged rows, 909 with scale_down in place of ldexp, 822 in this form,
// 782 without the branches, 669 with the idle lanes' own rows. Two stages 50 % slower,
// four (three blocks per SM) 2 % slower, the index load outside a branch (it then sinks
// to its use) twice as slow. X in L2 or not makes no difference: the time goes to L1 (row
// copies, their reads, shuffles) and to issue.
struct __align__(128) SubStage16 {
    float rows[32 * kSubChunk];
    float q[kSubChunk];
    float w[32];
    long long j;  // (first stage of a query)
    int groups;
};
constexpr size_t kSubSmem16 = sizeof(SubStage16) * kSubStages * kSubsetWarps;

// kL1: rows are copied through L1 (see few_lines).
template <int KERN, bool kW, bool kFull, bool kL1>
__global__ void __launch_bounds__(32 * kSubsetWarps, 4)
kde_subset16_kernel(const float *__restrict__ X, int64_t n, int d, int dp, const float *__restrict__ Q, int64_t m,
                    const int64_t *__restrict__ off, const int64_t *__restrict__ idx, const float *__restrict__ W,
                    float negc, double scale, double *__restrict__ out) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int S = kSubStages;
    constexpr unsigned SB = sizeof(SubStage16);
    const int lane = threadIdx.x & 31;
    // (the shuffle lets the compiler see that the warp's control flow is uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    SubStage16 *const ring = reinterpret_cast<SubStage16 *>(smem_raw) + warp * S;
    // the weights (like the indices, __ldcs) are read once: first to leave L2, which holds X
    uint64_t stream_policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
    const unsigned ring_a = (unsigned)__cvta_generic_to_shared(ring);
    const int64_t warps = (int64_t)gridDim.x * kSubsetWarps;
    const unsigned rowq = kFull ? 4u : dp / 4;  // 16-byte pieces per row
    // what a lane without an entry copies: one row for the warp, another for most other warps
    const unsigned idle_row = (unsigned)(((uint64_t)blockIdx.x * kSubsetWarps + warp) % (uint64_t)n) * rowq;
    // this lane copies piece `piece` of rows (lane / 4) + 8 i (a piece past the row's end:
    // zero bytes of it, so that the stage holds zeros there)
    const unsigned piece = lane & 3;
    const int bytes = kFull || piece < rowq ? 16 : 0;
    const float4 *const xp = reinterpret_cast<const float4 *>(X) + (kFull || piece < rowq ? piece : 0);
    const unsigned dst0 = ring_a + ((lane >> 2) * kSubChunk + ((piece ^ ((lane >> 3) & 3)) << 2)) * 4;
    // and reads row `lane`
    const unsigned src0 = lane * kSubChunk;
    const unsigned swz = (lane >> 1) & 3;

    int64_t gj = (int64_t)blockIdx.x * kSubsetWarps + warp - warps, n0 = 0, n1 = 0, gi = -1;
    const int64_t *ip = idx, *iend = idx;
    const float *wp = W;
    int gleft = 1, ngroups = 0;  // groups left of query gj, counting the one gi belongs to
    int total = 0x7fffffff, issued = 0;  // stages in all (known once the queries are exhausted)
    bool fresh = false;
    auto fetch_off = [&](int64_t j) {
        n0 = n1 = 0;
        if (j < m) {
            n0 = off[j];
            n1 = off[j + 1];
        }
    };
    auto advance = [&]() {
        ip += 32;
        if (kW) wp += 32;
        if (--gleft == 0) {
            do {
                gj += warps;
                if (gj >= m) {
                    total = issued;
                    return;
                }
                // (an end before its start counts as an empty list, as in the gather kernel: a
                // negative count would take 2^32 steps to come back to 0)
                ngroups = gleft = (int)((max(n1 - n0, (int64_t)0) + 31) >> 5);
                ip = idx + n0 + lane;
                iend = idx + n1;
                if (kW) wp = W + n0 + lane;
                fetch_off(gj + warps);
                if (gleft == 0 && lane == 0) out[gj] = 0.0;  // an empty list
            } while (gleft == 0);
            fresh = true;
        }
        gi = -1;
        if (ip < iend) gi = __ldcs(ip);
    };
    unsigned counts = 0;  // whether the lane's entry counts, one bit per stage in flight
    unsigned in = 0;      // byte offset of the stage to fill
    auto issue = [&]() {
        const bool ok = (unsigned long long)gi < (unsigned long long)n;
        // (an entry out of range contributes nothing and is not followed)
        const unsigned row = ok ? (unsigned)gi * rowq : idle_row;
        counts = counts + counts + (ok ? 1u : 0u);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned r = __shfl_sync(0xffffffffu, row, (lane >> 2) + 8 * i);
            const unsigned dst = dst0 + in + 8 * i * kSubChunk * 4;
            if (kFull && kL1)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(xp + r));
            else if (kFull)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(xp + r));
            else if (kL1)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(xp + r), "r"(bytes));
            else
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(xp + r), "r"(bytes));
        }
        if (kW)
            asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, %2, %3;\n" ::"r"(
                             ring_a + in + (unsigned)offsetof(SubStage16, w) + lane * 4),
                         "l"(ok ? wp : W), "r"(ok ? 4 : 0), "l"(stream_policy));
        if (fresh) {
            fresh = false;
            SubStage16 &st = *reinterpret_cast<SubStage16 *>(reinterpret_cast<unsigned char *>(ring) + in);
            if (lane < d)
                copy4(&st.q[lane], Q + gj * d + lane);
            else if (lane < kSubChunk)
                st.q[lane] = 0.f;
            if (lane == 0) {
                st.j = gj;
                st.groups = ngroups;
            }
        }
        ++issued;
        in = in == (S - 1) * SB ? 0u : in + SB;
        asm volatile("cp.async.commit_group;\n" ::);
    };

    fetch_off(gj + warps);
    advance();
#pragma unroll 1
    for (int s = 0; s < S - 1; ++s) {
        if (total == 0x7fffffff) {
            issue();
            advance();
        } else {
            counts += counts;
            asm volatile("cp.async.commit_group;\n" ::);
        }
    }
    float shift = kShiftInit, acc32 = 0.f;
    double acc64 = 0.0;
    int cnt = 0, cleft = 0;
    int64_t cj = 0;
    float qr[kSubChunk];
#pragma unroll
    for (int k = 0; k < kSubChunk; ++k) qr[k] = 0.f;
    const SubStage16 *st = ring;
#pragma unroll 1
    for (int done = 0; done < total; ++done) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(S - 2));
        __syncwarp();  // every lane's copies of this stage have landed, the oldest stage is free
        if (total == 0x7fffffff) {
            issue();
            advance();
        } else {
            counts += counts;
            asm volatile("cp.async.commit_group;\n" ::);
        }
        if (cleft == 0) {
            cj = st->j;
            cleft = __shfl_sync(0xffffffffu, st->groups, 0);
#pragma unroll
            for (int k = 0; k < kSubChunk; k += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(&st->q[k]);
                qr[k] = v.x;
                qr[k + 1] = v.y;
                qr[k + 2] = v.z;
                qr[k + 3] = v.w;
            }
        }
        const bool mine = (counts >> (S - 1)) & 1u;
        // one FP32 chain (the plain form's order; unused pieces add (0 - 0)^2). A lane without
        // an entry works on its warp's idle row and adds 0.
        float4 xv[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) xv[v] = *reinterpret_cast<const float4 *>(&st->rows[src0 + ((v ^ swz) << 2)]);
        float d2 = 0.f;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float t = qr[v * 4] - xv[v].x;
            d2 = fmaf(t, t, d2);
            t = qr[v * 4 + 1] - xv[v].y;
            d2 = fmaf(t, t, d2);
            t = qr[v * 4 + 2] - xv[v].z;
            d2 = fmaf(t, t, d2);
            t = qr[v * 4 + 3] - xv[v].w;
            d2 = fmaf(t, t, d2);
        }
        float e = kfn::term<KERN>(negc, d2, shift);
        float w = 1.f;
        if (kW) {
            w = st->w[lane];
            e = w * e;
        }
        e = mine ? e : 0.f;
        const bool high = !(fabsf(e) <= kGuard);
        if (__any_sync(0xffffffffu, high)) {
            // first term, or one far above the current shift: move the shift up
            const float s_new = fmaxf(ceilf(kfn::term_log2<KERN>(negc, d2)), kShiftInit);
            const float s_now = high && s_new > shift ? s_new : shift;
            const int de = clampe(shift - s_now);
            acc32 = de > -126 ? acc32 * __int_as_float((127 + de) << 23) : 0.f;
            acc64 = kfn::scale_down(acc64, de);
            shift = s_now;
            e = high ? w * kfn::term<KERN>(negc, d2, shift) : e;
        }
        acc32 += e;
        cnt += mine ? 1 : 0;
        if (__any_sync(0xffffffffu, cnt == kFlush)) {
            const bool flush = cnt == kFlush;
            acc64 += flush ? (double)acc32 : 0.0;
            acc32 = flush ? 0.f : acc32;
            cnt = flush ? 0 : cnt;
        }
        if (--cleft == 0) {
            acc64 += (double)acc32;
            // merge the lanes: common shift = the largest, fixed butterfly order
#pragma unroll 1
            for (int o = 16; o >= 1; o >>= 1) {
                const double oa = __shfl_xor_sync(0xffffffffu, acc64, o);
                const float os = __shfl_xor_sync(0xffffffffu, shift, o);
                const float sm = fmaxf(shift, os);
                acc64 = kfn::scale_down(acc64, clampe(shift - sm)) + kfn::scale_down(oa, clampe(os - sm));
                shift = sm;
            }
            if (lane == 0) out[cj] = ldexp(acc64, clampe(shift)) * scale;
            shift = kShiftInit;
            acc32 = 0.f;
            acc64 = 0.0;
            cnt = 0;
        }
        st = st == ring + S - 1 ? ring : st + 1;
    }
    asm volatile("cp.async.wait_group 0;\n" ::);
}

template <int KERN, bool kW, bool kFull, bool kL1>
int launch16(const stag_kde *h, const float *dQ, int64_t m, const int64_t *dOff, const int64_t *dIdx, const float *dW,
             float negc, double scale, double *dOut, cudaStream_t s) {
    auto kern = kde_subset16_kernel<KERN, kW, kFull, kL1>;
    static SmemOptIn opt_in;
    STAG_CUDA_TRY(opt_in((const void *)kern, (int)kSubSmem16));
    // four blocks per SM are resident; several times as many even out ragged lists
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(m, kSubsetWarps), (int64_t)h->sm_count * 12));
    kern<<<grid, 32 * kSubsetWarps, kSubSmem16, s>>>(h->xrow, h->n, (int)h->d, h->d_pad, dQ, m, dOff, dIdx, dW, negc,
                                                    scale, dOut);
    return 0;
}

// Point sets of a few L2 lines, which every warp of the chip would ask for at once: their rows
// are copied through L1, larger sets past it. Measured, 6e4 lists of 400, past / through L1, and
// every lane gathering its own row: 32 points of 4 coordinates 3486 / 184 / 317 us, 512 points
// 844 / 190 / 331, 2048 (32 KB) 251 / 228 / 332, 4096 184 / 235 / 332, 65536 181 / 243 / 334. Rows
// of 12 coordinates do not divide a line: 170 points 1881 / 201 / 332, 2730 (128 KB) 369 / 269 /
// 357, 4096 (192 KB) 266 / 272 / 370, 8192 212 / 276 / 391.
bool few_lines(const stag_kde *h) {
    return h->n * h->d_pad * 4 < (h->d_pad == 12 ? (int64_t)192 << 10 : (int64_t)64 << 10);
}

// Rows of at most 16 coordinates are staged (their offsets in 16-byte units must fit 32
// bits); longer ones are gathered by their lanes.
template <int KERN>
int launch_kern(const stag_kde *h, const float *dQ, int64_t m, const int64_t *dOff, const int64_t *dIdx,
                const float *dW, double *dOut, cudaStream_t s) {
    const float negc = (float)(-h->a * 1.4426950408889634);  // -a log2(e)
    const double scale = h->normalise ? 1.0 / (double)h->n : 1.0;
    if (h->d_pad <= kSubChunk && h->n * (h->d_pad / 4) <= 0xffffffffll) {
        const bool full = h->d_pad == kSubChunk, l1 = few_lines(h);
        auto go = [&](auto w, auto f, auto l) {
            return launch16<KERN, decltype(w)::value, decltype(f)::value, decltype(l)::value>(
                h, dQ, m, dOff, dIdx, dW, negc, scale, dOut, s);
        };
        const std::true_type yes{};
        const std::false_type no{};
        auto go_w = [&](auto w) {
            if (full) return l1 ? go(w, yes, yes) : go(w, yes, no);
            return l1 ? go(w, no, yes) : go(w, no, no);
        };
        return dW ? go_w(yes) : go_w(no);
    }
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(m, kSubsetWarps), (int64_t)h->sm_count * 16));
    kde_subset_kernel<KERN><<<grid, 32 * kSubsetWarps, (size_t)kSubsetWarps * h->d_pad * sizeof(float), s>>>(
        h->xrow, h->n, (int)h->d, h->d_pad, dQ, m, dOff, dIdx, dW, negc, scale, dOut);
    return 0;
}

// Flags (bit 0) an index outside [0, n) and (bit 1) a weight that is negative or not
// finite, over the nnz list entries.
__global__ void subset_check_kernel(const int64_t *__restrict__ idx, const float *__restrict__ W, int64_t nnz,
                                    int64_t n, int *flag) {
    int bad = 0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx[p];
        if (i < 0 || i >= n) bad |= 1;
        if (W) {
            const float w = W[p];
            if (!(w >= 0.f) || !isfinite(w)) bad |= 2;
        }
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(flag, bad);
}

}  // namespace

int subset_check_entries(const int64_t *dIdx, const float *dW, int64_t nnz, int64_t n, int *dflag, cudaStream_t s) {
    if (nnz <= 0) return 0;
    count_launch();
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(nnz, 256), 152 * 16));
    subset_check_kernel<<<grid, 256, 0, s>>>(dIdx, dW, nnz, n, dflag);
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

int subset_prepare(stag_kde *h, cudaStream_t s) {
    if (h->xrow) return 0;
    if (h->dtype != STAG_KDE_F32 || !h->xt) return fail(STAG_KDE_EUNSUPPORTED, "subset sums: FP32 handles only");
    if (h->d > kSubsetMaxD)
        return fail(STAG_KDE_EUNSUPPORTED, "subset sums: d too large");
    STAG_CUDA_TRY(dev_malloc(&h->xrow, (size_t)(h->n * h->d_pad) * sizeof(float)));
    int rc = simt_points_rows(h, h->xrow, h->d_pad, s);
    if (rc) return rc;
    // later calls may come on other streams: the copy must be complete before them
    STAG_CUDA_TRY(cudaStreamSynchronize(s));
    return 0;
}

int subset_query(stag_kde *h, const float *dQ, int64_t m, const int64_t *dOff, const int64_t *dIdx, const float *dW,
                 double *dOut, cudaStream_t s, double entries) {
    int rc = subset_prepare(h, s);
    if (rc) return rc;
    count_launch();
    prof_start(h, s);
    switch (h->kernel) {
        case STAG_KDE_KERNEL_EXPONENTIAL:
            rc = launch_kern<STAG_KDE_KERNEL_EXPONENTIAL>(h, dQ, m, dOff, dIdx, dW, dOut, s);
            break;
        case STAG_KDE_KERNEL_LOGISTIC:
            rc = launch_kern<STAG_KDE_KERNEL_LOGISTIC>(h, dQ, m, dOff, dIdx, dW, dOut, s);
            break;
        default:
            rc = launch_kern<STAG_KDE_KERNEL_GAUSSIAN>(h, dQ, m, dOff, dIdx, dW, dOut, s);
    }
    prof_stop(h, s, entries);
    if (rc) return rc;
    STAG_CUDA_TRY(cudaGetLastError());
    return 0;
}

}  // namespace stagkde
