// caq_launch.h -- the arguments of the quantize kernels' launches, shared by
// the lane-per-vector kernels (k_caq1.cu) and the scan (k_caq_scan.cu).
#pragma once

#include "saq_internal.h"

namespace saq {

constexpr int kMaxSeg = 64;

struct Seg {
    int off, len, bits, words, fidx;
    long long code_off;
};
struct SegTable {
    Seg s[kMaxSeg];
    int order[kMaxSeg];  // segments by decreasing length: long work starts first
};
// One model's rows of a launch: its interleaved projected rows, byte-code
// scratch, v_max and outputs.
struct CaqGroup {
    const float *Oi;
    int64_t n;
    int dk, nseg, rounds, nf;
    uint8_t *cs;
    const float *vmax;
    uint8_t *codes;
    int64_t code_stride;
    float *factors;
    SegTable t;
};
// A launch over G models: global warp w belongs to the group g with
// warp_start[g] <= w < warp_start[g + 1] (ngroups <= G).
template <int G> struct CaqBatch {
    int ngroups;
    int64_t warp_start[G + 1];
    CaqGroup g[G];
};

// The kernel arguments of job j (k_caq1.cu).
saq_status make_group(const CaqJob &j, CaqGroup *g);

// The scan (k_caq_scan.cu): launch_caq_scan runs the jobs if it is the better
// kernel for them and sets *ran, else it does nothing.
saq_status launch_caq_scan(const CaqJob *jobs, int njobs, cudaStream_t s, bool *ran);

}  // namespace saq
