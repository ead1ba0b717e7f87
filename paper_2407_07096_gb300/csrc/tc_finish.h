// What follows the tensor-core kernel: the FP64 combine of the partial sums with the
// per-query error estimate, and the FP32 recompute of the queries it flags (tc_finish.cu).
#pragma once
#include "internal.h"

namespace stagkde {

// One instance as the two kernels see it (a launch serves a table of instances; a single
// query passes its one entry in kernel-parameter space).
struct FinInst {
    // combine
    const double *part_sum, *part_w;
    const float *part_shift;
    const int *qbad;
    unsigned *ub;   // per-query exponent bounds, set back to 0 for the next call
    double *out;
    int *qflag;     // per-query flags, or NULL: no estimate, nothing is recomputed
    int *fix_count; // number of flagged queries
    int64_t m, m_pad;
    double scale, a;
    int splits, lpq;  // ranges of points; lanes that share a query's ranges (a power of two)
    // recompute
    const float *Q, *R, *tinfo, *xkt;
    int64_t n, n_tiles, T;
    int d, d_pad, seg, per_log, passes;  // passes: 8-bit digits of a tile index
    float c, negc;
    uint32_t *key, *ktmp, *val, *vtmp, *hist;
    float *thr, *qt, *pshift;
    int *bcnt, *kept, *kcount, *items, *item_off;
    double *psum;
    // numbering inside the launch
    int cblock_begin;  // first combine block
    int qblock_begin;  // first block of 256 queries
};

// Counters of the recompute kernel's phases: work items claimed and done.
struct FinCtl {
    int claim[32], done[32];
};
// (behind it: three arrays of n_inst + 1 prefix sums, and the instances' flag counts)
inline size_t fin_ctl_bytes(int64_t n_inst) { return sizeof(FinCtl) + (4 * (size_t)n_inst + 3) * sizeof(int); }

// Bytes of an instance's recompute scratch for up to m queries; with inst, also sets its
// scratch pointers into base.
int64_t fin_scratch_bytes(int64_t m, int64_t T, int BN, FinInst *inst, void *base);
// Numbers the instance (combine blocks from cblock, 256-query blocks from qblock) and
// returns how many of each it has.
void fin_number(FinInst *inst, int sm_count, int cblock, int qblock, int *cblocks, int *qblocks);
// Queues both kernels: table (device) of n_inst instances, or the single inst0 if table is
// NULL. recompute = false leaves the second out (no instance checks its results).
int fin_launch(const FinInst &inst0, const FinInst *table, int n_inst, int cblocks, int qblocks, int max_passes,
               int max_d_pad, int64_t max_items, bool recompute, FinCtl *ctl, int *err, int sm_count,
               cudaStream_t s);

}  // namespace stagkde
