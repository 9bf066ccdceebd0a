// k_caq_scan.cu -- quantize, adjust and pack with one WARP per vector-segment,
// for the batches that leave the lane-per-vector kernels of k_caq1.cu without
// parallelism (one vector, a request, a small collection).
//
// Algorithm 1 is a sequential scan, but most of its trials fail: at d = 960,
// 4 b/dim about 170 of a vector's 4,621 trials move a code.  The 32 lanes of a
// warp try 32 consecutive coordinates against the current state at once; a
// ballot finds the first that moves, its state is broadcast, and the lanes
// after it try again.  Every decision is taken from the state the sequential
// scan has at that coordinate, with the same operations, so the codes are the
// same; the lane-per-vector kernel takes ~54 cycles a coordinate and round
// when a warp has an SM to itself (448 coordinates: 82 us).
//
// A block takes R rows of one kept segment (R = its warps).  The rows are
// staged in shared memory (R + 1 floats per coordinate: conflict-free for
// lanes along rows and for lanes along coordinates), all threads form the
// initial codes, and the sums <u, o>, |o|^2 and |u|^2, which the decisions and
// factors take in coordinate order, run with one lane per row in a warp each.
#include <algorithm>

#include "caq_launch.h"

namespace saq {

namespace {

constexpr size_t kScanSmemMax = 225 * 1024;

// Shared memory of a block: x and u (R + 1 floats per coordinate), and per
// row I, |o|^2, S and v_max.
__host__ __device__ constexpr size_t scan_smem(int len, int R) {
    return (size_t)len * (R + 1) * 8 + (size_t)4 * R * 4;
}

template <int G, int R>
__global__ void __launch_bounds__(R * 32)
k_caq_scan(const __grid_constant__ CaqBatch<G> batch) {
    extern __shared__ float sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the block's segment and rows: warp_start counts blocks here
    int gi = 0;
    const int64_t item = blockIdx.x;
    if constexpr (G > 1)
        while (gi + 1 < batch.ngroups && item >= batch.warp_start[gi + 1]) ++gi;
    const CaqGroup &P = batch.g[gi];
    const int64_t local = item - batch.warp_start[gi];
    const int64_t rgs = (P.n + R - 1) / R;
    const int si = P.t.order[local / rgs];
    const Seg &sg = P.t.s[si];
    const int64_t r0 = local % rgs * R;
    const int nv = (int)min((int64_t)R, P.n - r0);
    const int len = sg.len, B = sg.bits, cmax = (1 << B) - 1;
    const float cmaxf = (float)cmax;
    constexpr int RS = R + 1;
    float *xs = sm, *us = xs + (size_t)len * RS, *st = us + (size_t)len * RS;  // st: I, n2, S, vmax

    const int64_t g32 = r0 >> 5;
    const int sub = (int)(r0 & 31);
    // rows into shared memory and the initial codes (Eq. find_nearest_code)
    {
        const int rr = tid % R;
        if (rr < nv) {
            constexpr int kB = 8;
            const float *src = P.Oi + ((g32 * P.dk + sg.off) << 5) + sub + rr;
            const float vmax = __ldg(P.vmax + ((g32 * P.nseg + si) << 5) + sub + rr);
            float inv_delta = 0.f, off_c = 0.f;
            for (int i0 = tid / R; i0 < len; i0 += 32 * kB) {
                float x[kB];
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int i = i0 + 32 * k;
                    x[k] = i < len ? __ldg(src + ((int64_t)i << 5)) : 0.f;
                }
                if (i0 == tid / R) {  // v_max has come with the first rows
                    inv_delta = vmax > 0.f ? (float)(1 << (B - 1)) / vmax : 0.f;
                    off_c = vmax * inv_delta;
                    if (tid < R) st[3 * R + tid] = vmax;
                }
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    const int i = i0 + 32 * k;
                    if (i >= len) break;
                    const float v = vmax > 0.f ? x[k] : 0.f;
                    const float cf = fminf(fmaxf(floorf(fmaf(v, inv_delta, off_c)), 0.f), cmaxf);
                    xs[i * RS + rr] = v;
                    us[i * RS + rr] = fmaf(2.f, cf, -cmaxf);
                }
            }
        }
    }
    __syncthreads();
    // the three sums in coordinate order, a warp each, a lane per row
    if (warp < 3 && lane < nv) {
        float a = 0.f;
        // <u, x>, <x, x>, <u, u>
        const float *p = (warp == 1 ? xs : us) + lane, *q = (warp == 2 ? us : xs) + lane;
#pragma unroll 8
        for (int i = 0; i < len; ++i) a = fmaf(p[i * RS], q[i * RS], a);
        st[warp * R + lane] = a;
    }
    __syncthreads();
    if (warp >= nv) return;

    // ---- the rounds: warp `warp` scans row r0 + warp
    const int64_t v = r0 + warp;
    float I = st[warp], S = st[2 * R + warp];
    const float n2 = st[R + warp];
    const bool live = st[3 * R + warp] > 0.f;
    float I2 = I * I;
    const int nb = (len + 31) >> 5;
    const float *xr = xs + warp;
    float *ur = us + warp;
    for (int r = 0; r < P.rounds && live; ++r) {
        bool moved = false;
        for (int b = 0; b < nb; ++b) {
            const int i = b * 32 + lane;
            const bool in = i < len;
            const float x = in ? xr[i * RS] : 0.f;
            float u = in ? ur[i * RS] : 0.f;
            uint32_t left = __ballot_sync(0xffffffffu, in);
            bool mine = false;
            for (;;) {
                const float xS = x * S;
                const float T = fmaf(-u, I, xS);
                const uint32_t sgn = __float_as_uint(T) & 0x80000000u;
                const float su = __uint_as_float(__float_as_uint(u) ^ sgn);
                const bool ok = su < cmaxf && fmaf(fabsf(T), I, x * xS) > I2;
                const float In = fmaf(__uint_as_float(0x40000000u | sgn), x, I);
                const float Sn = fmaf(4.f, su, S + 4.f);
                const uint32_t m = __ballot_sync(0xffffffffu, ok) & left;
                if (m == 0u) break;
                const int f = __ffs((int)m) - 1;
                I = __shfl_sync(0xffffffffu, In, f);
                S = __shfl_sync(0xffffffffu, Sn, f);
                I2 = I * I;
                if (lane == f) {
                    u += __uint_as_float(0x40000000u | sgn);
                    mine = true;
                }
                left = f == 31 ? 0u : 0xffffffffu << (f + 1) & left;
                moved = true;
            }
            if (mine) ur[i * RS] = u;
        }
        if (!moved) break;
    }
    __syncwarp();
    // bit-planes (a ballot per plane and 32 coordinates) and |u|^2, exactly
    uint32_t *cout = reinterpret_cast<uint32_t *>(P.codes + v * P.code_stride + sg.code_off);
    int Si = 0;
    for (int b = 0; b < 2 * sg.words; ++b) {
        const int i = b * 32 + lane;
        const bool in = i < len;
        const int u = in && live ? (int)ur[i * RS] : -cmax;
        const int c = (u + cmax) >> 1;
        if (in) Si += u * u;
        uint32_t mine = 0u;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            if (p >= B) break;  // uniform
            const uint32_t w = __ballot_sync(0xffffffffu, (c >> (B - 1 - p)) & 1);
            if (lane == p) mine = w;
        }
        if (lane < B) cout[lane * sg.words * 2 + b] = mine;
    }
    Si = __reduce_add_sync(0xffffffffu, Si);
    if (lane == 0) {
        float *fo = P.factors + v * P.nf + sg.fidx;
        const float nrm = sqrtf(n2);
        // all-zero segment (the paper is silent): codes 0, |o| = 0, cos = 1
        fo[0] = live ? nrm : 0.f;
        fo[1] = live ? I / (sqrtf((float)Si) * nrm) : 1.f;
    }
}

template <int G, int R>
saq_status launch_form(CaqBatch<G> &b, const CaqJob *jobs, int njobs, int maxlen, cudaStream_t s) {
    b.ngroups = 0;
    b.warp_start[0] = 0;
    for (int i = 0; i < njobs; ++i) {
        if (jobs[i].n <= 0 || jobs[i].m->kept.empty()) continue;
        saq_status st = make_group(jobs[i], &b.g[b.ngroups]);
        if (st != SAQ_OK) return st;
        b.warp_start[b.ngroups + 1] =
            b.warp_start[b.ngroups] + (jobs[i].n + R - 1) / R * (int64_t)b.g[b.ngroups].nseg;
        ++b.ngroups;
    }
    const int64_t blocks = b.warp_start[b.ngroups];
    const size_t smem = scan_smem(maxlen, R);
    SAQ_CUDA_CHECK(cudaFuncSetAttribute(k_caq_scan<G, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kScanSmemMax));
    {
        LaunchTimer lt_(kKindQuantize, s);
        k_caq_scan<G, R><<<(unsigned)blocks, R * 32, smem, s>>>(b);
    }
    note_launches();
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

}  // namespace

saq_status launch_caq_scan(const CaqJob *jobs, int njobs, cudaStream_t s, bool *ran) {
    *ran = false;
    int64_t coords = 0;
    int maxlen = 0, chain = 0, used = 0;
    for (int i = 0; i < njobs; ++i) {
        if (jobs[i].n <= 0 || jobs[i].m->kept.empty()) continue;
        ++used;
        coords += jobs[i].n * jobs[i].m->dk;
        for (const KeptSeg &k : jobs[i].m->kept) {
            maxlen = std::max(maxlen, (int)k.len);
            chain = std::max(chain, (int)(k.bits == 1 ? (k.len + 3) / 4 : k.len));
        }
    }
    if (used == 0 || scan_smem(maxlen, 8) > kScanSmemMax) return SAQ_OK;
    // 16 rows per block where their rows fit three blocks to an SM
    const bool r16 = scan_smem(maxlen, 16) <= 75 * 1024;
    // The lane-per-vector kernel takes at least its longest segment's chain of
    // steps (0.18 us a coordinate at 6 rounds, a quarter of it at 1 bit, where
    // the first round moves nothing); the scan takes 12-16 ns per 1,000
    // coordinates, 21-32 where one block fills an SM's shared memory.  Either
    // side of the line, scan and lane-per-vector: d = 960 (448-long, 4 b/dim)
    // 5,500 rows 87.6 us, 5,700 82.1; d = 128 (64-long) 5,900 18.0, 6,100 18.0;
    // d = 1536 (704-long) 5,400 114, 5,600 125; d = 3072 at 1 b/dim 1,150 59,
    // 1,190 79, at 8 b/dim 5,900 584, 6,100 555.
    const bool shared = r16 || scan_smem(maxlen, 8) <= 75 * 1024;
    if (coords > (int64_t)(shared ? 12000 : 6000) * chain) return SAQ_OK;
    *ran = true;
    if (used == 1) {
        CaqBatch<1> b;
        return r16 ? launch_form<1, 16>(b, jobs, njobs, maxlen, s)
                   : launch_form<1, 8>(b, jobs, njobs, maxlen, s);
    }
    CaqBatch<kMaxGroups> b;
    return r16 ? launch_form<kMaxGroups, 16>(b, jobs, njobs, maxlen, s)
               : launch_form<kMaxGroups, 8>(b, jobs, njobs, maxlen, s);
}

}  // namespace saq
