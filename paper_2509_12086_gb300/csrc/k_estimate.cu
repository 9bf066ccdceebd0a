// k_estimate.cu -- distance estimation from codes (Sec. 2.2 Eq. 3, Sec. 3.2
// Eq. estimator_inner_product, progressive prefixes of Sec. 3.2).
//
// Per kept segment s of vector v and query q (q_s = W_s (q_r - c)):
//   est_s = |o_s| <u_s, q_s> / (|u_s| cos_s),   u_s = 2 c - (2^b - 1)
// i.e. <o_bar_a, q> / <o_bar_a, o> |o|^2 with o_bar_a proportional to u_s
// (Delta <c, q> + q_sum (Delta/2 - v_max) = (Delta/2) <u, q>).
// d2 = |o_r - c|^2 + |q_r - c|^2 - 2 sum_s est_s.
// With a b-bit prefix the code is floor(c / 2^(B-b)) = the first b planes.
//
// Multi-stage estimation (Sec. 4.3): the kept segments are taken in plan
// order (decreasing variance); after t stages the first t contribute est_s
// and each remaining one its Chebyshev bound m * sigma_Seg(q), where
// sigma_Seg(q)^2 = sum_{i in Seg} sigma_i^2 (v_i . (q_r - c))^2 is the
// variance of <o_seg, q_seg> over the data:
//   lb_t = |o_r - c|^2 + |q_r - c|^2 - 2 (sum_{s<t} est_s + m sum_{s>=t} sigma_s).
//
// <c_s, q_s> of 16 vectors and 4 queries at a time is a matrix product on the
// tensor cores (mma.sync m16n8k16, FP16 operands, FP32 accumulators).  A code's
// bits are its A operand as they stand: read as a subnormal FP16 number they
// are c 2^-24, so decoding is the bit-plane transposition, a shift and a mask.
// Each query coordinate, times a power of two of its own (query, segment), is
// a pair hi + lo / 4096 in two columns of B: hi an integer, lo the FP16 value
// of what it leaves (at least 23 bits below the larger of hi and 2048).
//
// The tensor core truncates its sums, so those of hi, which carry the result's
// leading bits, are kept exact: the accumulator starts at -2^(b-1) sum hi and
// holds <c - 2^(b-1), hi> at the end, and while
//     2^(b-1) sum |hi| <= 2^24
// every partial sum is an integer (times 2^-24) that FP32 represents.  The
// scale is the largest power of two for which that holds, whatever the
// coordinates' signs and sizes are.  The sums run over a window of the segment:
// all of it up to 4 bits, 128 2^(8-b) coordinates from 5 bits up, where one
// window of a long segment would leave hi too few bits; windows are added up in
// FP32.  <u, q> = 2 <c - 2^(b-1), hi> + sum hi + (2 <c, lo> - (2^b - 1) sum lo) / 4096.
// Largest error over |u| |q| (512 vectors by 24 queries, 960 long at 8 bits, against
// 64 bits; in brackets of sums of the products by FP32 lanes, and of queries
// with one scale each whose <c, hi> were summed over the whole segment from 0):
// Gaussian coordinates 1.8e-8 (2.0e-8, 3.0e-8), all of one sign 2.2e-8 (2.1e-8,
// 4.1e-6), one of 1,000 among Gaussians 2.0e-8 (2.3e-8, 1.4e-7).
#include <cuda_fp16.h>

#include <algorithm>
#include <cfloat>

#include "saq_internal.h"

namespace saq {

namespace {

struct SegDesc {
    int off, len, bits, words, fidx;  // bits: those that the estimate reads
    int step, window;                 // its first K step and window
    long long code_off;
};
constexpr int kMaxSeg = 64;
struct SegTable {
    SegDesc s[kMaxSeg];
};

// ------------------------------------------------------------ the queries
// out[q * dk + j] = <M_j, q_r - c> for the rows M_j of a dk x d matrix, and with
// qn2 also |q_r - c|^2.  A warp computes CPW columns for QB queries: its lanes
// split the d coordinates (the rows of M are read once, coalesced, and each
// value meets QB centred queries in shared memory), so that a single query
// spreads over dk warps (d = 960: 8.5 us; on the 128 x 128 tiles of the row
// projection, eight blocks, 207 us).  Only the coordinates there are get staged
// (with 1,024 whatever d is: 16,000 queries at d = 128 79 -> 47 us, 8,000 at 1536
// 1,609 -> 1,264, 8,000 at 960 622 -> 611).
// The row projection's tiles, whose sums run over all coordinates in one lane,
// are as fast at 16,000 queries of 128 coordinates (44 us) and faster beyond
// (64,000: 111 against 214).
constexpr int kRotK = 1024;  // coordinates of the queries staged at a time
template <int QB, int CPW, bool V4>
__global__ void __launch_bounds__(256)
k_query_rot(const float *__restrict__ Q, int64_t nq, int d, const float *__restrict__ mean,
            const float *__restrict__ M, int dk, float *__restrict__ out,
            float *__restrict__ qn2) {
    static_assert(QB * CPW == 32 || QB * CPW == 1, "one result per lane, or one per warp");
    __shared__ __align__(16) float qs[QB][kRotK];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q0 = (int64_t)blockIdx.y * QB;
    const int j0 = ((int)blockIdx.x * 8 + warp) * CPW;
    float acc[CPW * QB];
#pragma unroll
    for (int i = 0; i < CPW * QB; ++i) acc[i] = 0.f;
    float n2 = 0.f;
    const bool norm = qn2 && blockIdx.x == 0 && warp < QB;
    const float *row[CPW];
#pragma unroll
    for (int c = 0; c < CPW; ++c) row[c] = M + (int64_t)min(j0 + c, dk - 1) * d;
    for (int k0 = 0; k0 < d; k0 += kRotK) {
        const int kn = min(kRotK, d - k0);
        if (k0) __syncthreads();
        constexpr int kTeam = 256 / QB;  // threads to a query
        const int b = threadIdx.x / kTeam;
#pragma unroll 8
        for (int k = threadIdx.x % kTeam; k < kn; k += kTeam)
            qs[b][k] = q0 + b < nq ? Q[(q0 + b) * d + k0 + k] - mean[k0 + k] : 0.f;
        __syncthreads();
        if (norm)
            for (int k = lane; k < kn; k += 32) n2 = fmaf(qs[warp][k], qs[warp][k], n2);
        if constexpr (V4) {  // d % 4 == 0: every row of M is 16-byte aligned
            for (int k = 4 * lane; k < kn; k += 128) {
                float4 w[CPW];
#pragma unroll
                for (int c = 0; c < CPW; ++c)
                    w[c] = __ldg(reinterpret_cast<const float4 *>(row[c] + k0 + k));
#pragma unroll
                for (int b = 0; b < QB; ++b) {
                    const float4 y = *reinterpret_cast<const float4 *>(&qs[b][k]);
#pragma unroll
                    for (int c = 0; c < CPW; ++c) {
                        float &r = acc[c * QB + b];
                        r = fmaf(w[c].x, y.x, r);
                        r = fmaf(w[c].y, y.y, r);
                        r = fmaf(w[c].z, y.z, r);
                        r = fmaf(w[c].w, y.w, r);
                    }
                }
            }
        } else {
            for (int k = lane; k < kn; k += 32) {
                float w[CPW];
#pragma unroll
                for (int c = 0; c < CPW; ++c) w[c] = __ldg(row[c] + k0 + k);
#pragma unroll
                for (int b = 0; b < QB; ++b)
#pragma unroll
                    for (int c = 0; c < CPW; ++c) acc[c * QB + b] = fmaf(w[c], qs[b][k], acc[c * QB + b]);
            }
        }
    }
    if (norm) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, off);
        if (lane == 0 && q0 + warp < nq) qn2[q0 + warp] = n2;
    }
    if constexpr (QB * CPW == 1) {
        float s = acc[0];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0 && j0 < dk) out[q0 * dk + j0] = s;
    } else {
        // 32 sums over 32 lanes: each exchange halves the values a lane holds,
        // and lane i ends with sum i (column i / QB, query i % QB)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const bool up = lane & off;
#pragma unroll
            for (int i = 0; i < off; ++i) {
                const float give = up ? acc[i] : acc[i + off], keep = up ? acc[i + off] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        }
        const int j = j0 + lane / QB;
        const int64_t q = q0 + lane % QB;
        if (j < dk && q < nq) out[q * dk + j] = acc[0];
    }
}

// sig[q * nk + s] = sigma_Seg(q) = |B_s (q_r - c)| from the rotated values
// pc[q * dk + i] (rows sigma_i v_i^T); one warp per (query, kept segment)
__global__ void k_query_sigma(const float *__restrict__ pc, int64_t nq, int dk, int nk,
                              const __grid_constant__ SegTable t, float *__restrict__ sig) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= nq * nk) return;
    const int64_t q = w / nk;
    const int s = (int)(w % nk);
    const float *p = pc + q * dk + t.s[s].off;
    float acc = 0.f;
    for (int i = lane; i < t.s[s].len; i += 32) acc = fmaf(p[i], p[i], acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) sig[q * nk + s] = sqrtf(acc);
}

// Widths up to kNarrow bits take a segment as one window.
constexpr int kNarrow = 4;
// Pieces (of 128 coordinates, see step_coord) of a window at `bits` > kNarrow:
// 2^(bits-1) times a window's coordinates is 16,384, which leaves hi a scale of
// ~1,000 per standard deviation of a Gaussian window.
__host__ __device__ constexpr int window_pieces(int bits) { return 1 << (8 - bits); }
// Windows of a segment of `words` 64-bit words.
constexpr int window_count(int bits, int words) {
    return bits <= kNarrow ? 1 : ((words + 1) / 2 + window_pieces(bits) - 1) / window_pieces(bits);
}
// Bits that a segment's estimate reads.
constexpr int used_bits(int prefix_bits, int bits) {
    return prefix_bits > 0 && prefix_bits < bits ? prefix_bits : bits;
}

// The exponent of a (query, segment)'s scale, from the largest window sum l1 of
// |q| and the largest |q|: 2^(b-1) sum |hi| <= 2^24 (rounding adds at most 1/2 to
// each of a window's n coordinates, or 2^-11 of it above 2048) and |hi| <= 2^15.
// 0 for an all-zero query or one that is not finite, whose estimates are not
// finite either.
__device__ __forceinline__ int scale_exponent(float l1, float mx, int bits, int n) {
    constexpr float kSlack = 1.f - 0x1p-10f;
    if (!(l1 <= FLT_MAX))  // NaN, an infinity, or finite values whose sum is not
        return l1 == l1 && mx <= FLT_MAX ? -126 : 0;
    if (l1 == 0.f) return 0;
    const float b = fmaxf((float)(1 << (25 - bits)) - 0.5f * (float)n, 1.f) * kSlack;
    const int e = min(ilogbf(b) - ilogbf(l1), 14 - ilogbf(mx));  // within one of the answer
    return max(-126, min(100, e - (scalbnf(l1, e) > b || scalbnf(mx, e) > 32768.f * kSlack)));
}

// The coordinate (of a segment of `words` 64-bit words) that element i (0..3)
// of lane quad position t holds in K step `step` of the segment.  The lanes of
// a quad decode 32 bits of a plane each at a time (8 steps of 16 coordinates):
// lane t bits 32 h .. of word 4 c + t of the chunk of four words c (h = 0, 1:
// the quad reads 32 contiguous bytes over the two), then, of two words left
// over, bits 32 t .. of both, and of a last one 16 bits each (4 steps).
__device__ __forceinline__ int step_coord(int words, int step, int t, int i) {
    const int full = words >> 2, m = step & 7, c = step >> 4;
    const int k = m >> 1, r = 2 * (m & 1) + (i >> 1), hi = i & 1;
    if (c < full) return (4 * c + t) * 64 + ((step >> 3) & 1) * 32 + 4 * k + r + 16 * hi;
    const int at = 256 * full;
    if ((words & 2) && step - 16 * full < 8) return at + 32 * t + 4 * k + r + 16 * hi;
    return at + ((words & 2) ? 128 : 0) + 16 * t + 4 * k + r + 8 * hi;
}

// A scaled coordinate's parts: the nearest integer (multiple of an FP16 unit in
// the last place above 2048), and 4096 times what it leaves, in FP16.
__device__ __forceinline__ float split_hi(float y) {
    // 1.5 * 2^23 times that unit, whose sum with y rounds it off
    const uint32_t e = max(__float_as_uint(fabsf(y)) >> 23, 137u);
    const float m = __uint_as_float((e + 13u) << 23 | 0x400000u);
    return (y + m) - m;
}
__device__ __forceinline__ float split_lo(float y, float hi) { return (y - hi) * 4096.f; }

// B fragments of four queries (block x: column group pass * NT + nt) and one
// segment (block y): entry ((pass * steps + step) * NT + nt) * 32 + lane holds
// the four FP16 values of column lane / 4 (query 4 (pass * NT + nt) + column / 2,
// hi or lo part) for lane quad position lane % 4.  Also, of each query, the
// accumulators' start in every window, -2^(b-1) sum hi (times 2^-24),
// wstart[((pass * windows + window) * NT + nt) * 4 + query], and per segment
// qseg[((pass * segments + segment) * NT + nt) * 4 + query]: the inverse scale and
// what completes <u, q>, sum hi and -(2^b - 1) sum lo / 4096.
// The first block z of a segment forms the sums and the others share its K steps
// (a block that is alone does both); each needs the scales, for which it reads the
// segment once.  Bound by the latency of those reads and sums: 5.8 us for a
// 960-long segment, 7.5 for 3,072 (17.7 with eight warps a block that read one
// piece at a time; under ncu).
constexpr int kSplitPieces = 512;  // pieces whose sums are held at a time
constexpr int kSplitWarps = 16;
// Four sums over a warp's lanes; lane l gets sum l / 16 + 2 (l / 8 % 2).
__device__ __forceinline__ float warp_sums(const float (&a)[4], int lane) {
    const bool u = lane & 16, v = lane & 8;
    const float b0 = (u ? a[1] : a[0]) + __shfl_xor_sync(0xffffffffu, u ? a[0] : a[1], 16);
    const float b1 = (u ? a[3] : a[2]) + __shfl_xor_sync(0xffffffffu, u ? a[2] : a[3], 16);
    float c = (v ? b1 : b0) + __shfl_xor_sync(0xffffffffu, v ? b0 : b1, 8);
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    return c;
}
__global__ void __launch_bounds__(32 * kSplitWarps)
k_query_split(const float *__restrict__ qrot, int64_t nq, int dk,
              const __grid_constant__ SegTable t, int steps, int NT, int windows,
              uint2 *__restrict__ bfrag, float *__restrict__ wstart, float4 *__restrict__ qseg) {
    __shared__ float piece[2][4][kSplitPieces];
    __shared__ float s_max[kSplitWarps], s_l1[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t group = blockIdx.x, pass = group / NT, q0 = 4 * group;
    const int nt = (int)(group % NT), s = blockIdx.y;
    const int len = t.s[s].len, words = t.s[s].words, bits = t.s[s].bits;
    const float *src = qrot + q0 * dk + t.s[s].off;
    // warp w reads the pieces w / 4, w / 4 + 4, ... of query w % 4, four at a time
    // (P to a window)
    const int pieces = (words + 1) / 2, full = words >> 2;
    const int P = bits <= kNarrow ? pieces : window_pieces(bits), nwin = (pieces + P - 1) / P;
    const int wq = warp & 3;
    const bool wlive = q0 + wq < nq;
    const int which = (lane >> 4) | ((lane >> 3) & 1) << 1;  // warp_sums' of the lane
    auto fetch = [&](int p0, float (&x)[4][4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int pi = p0 + 4 * k;
                const int c = pi < 2 * full ? (4 * (pi >> 1) + j) * 64 + (pi & 1) * 32 + lane
                                            : 256 * full + (pi - 2 * full) * 128 + 32 * j + lane;
                x[k][j] = wlive && c < len ? __ldg(src + (int64_t)wq * dk + c) : 0.f;
            }
    };
    auto warp_sum = [](float a) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        return a;
    };
    // ---- the scales
    {
        float mx = 0.f, l1 = 0.f;
        for (int p0 = 0; p0 < pieces; p0 += kSplitPieces) {
            const int pn = min(kSplitPieces, pieces - p0);
            for (int i = warp >> 2; i < pn; i += 16) {
                float x[4][4], a[4];
                fetch(p0 + i, x);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[k] = (fabsf(x[k][0]) + fabsf(x[k][1])) + (fabsf(x[k][2]) + fabsf(x[k][3]));
#pragma unroll
                    for (int j = 0; j < 4; ++j) mx = fmaxf(mx, fabsf(x[k][j]));
                }
                const float c = warp_sums(a, lane);
                if ((lane & 7) == 0 && i + 4 * which < pn) piece[0][wq][i + 4 * which] = c;
            }
            __syncthreads();
            if (warp < 4) {
                if (nwin == 1) {
                    for (int i = lane; i < pn; i += 32) l1 += piece[0][wq][i];
                } else {  // P divides kSplitPieces
                    for (int w = lane; w * P < pn; w += 32) {
                        float a = 0.f;
                        for (int i = w * P; i < min(pn, w * P + P); ++i) a += piece[0][wq][i];
                        l1 = a > l1 || a != a ? a : l1;  // a NaN stays
                    }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float o = __shfl_xor_sync(0xffffffffu, l1, off);
            l1 = nwin == 1 ? l1 + o : o > l1 || o != o ? o : l1;
        }
        if (lane == 0) s_max[warp] = mx;
        if (lane == 0 && warp < 4) s_l1[warp] = l1;
        __syncthreads();
    }
    auto exponent = [&](int b) {
        const float mx = fmaxf(fmaxf(s_max[b], s_max[b + 4]), fmaxf(s_max[b + 8], s_max[b + 12]));
        return scale_exponent(s_l1[b], mx, bits, min(len, 128 * P));
    };
    // ---- the sums
    if (blockIdx.z == 0) {
        const float scale = scalbnf(1.f, exponent(wq));
        const float start = -(float)(1 << (bits - 1)) * 0x1p-24f;
        float hi = 0.f, lo = 0.f;
        float *ws = wstart + (pass * windows + t.s[s].window) * NT * 4 + nt * 4 + wq;
        for (int p0 = 0; p0 < pieces; p0 += kSplitPieces) {
            const int pn = min(kSplitPieces, pieces - p0);
            for (int i = warp >> 2; i < pn; i += 16) {
                float x[4][4], a[4], b[4];
                fetch(p0 + i, x);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    a[k] = b[k] = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float y = x[k][j] * scale, r = split_hi(y);
                        a[k] += r;
                        b[k] += __half2float(__float2half_rn(split_lo(y, r)));
                    }
                }
                const float ca = warp_sums(a, lane), cb = warp_sums(b, lane);
                if ((lane & 7) == 0 && i + 4 * which < pn) {
                    piece[0][wq][i + 4 * which] = ca;
                    piece[1][wq][i + 4 * which] = cb;
                }
            }
            __syncthreads();
            if (warp < 4)
                for (int w = lane; w * P < pn || (nwin == 1 && w < pn); w += 32) {
                    // (one window: a piece each)
                    const int i0 = nwin == 1 ? w : w * P, i1 = nwin == 1 ? w + 1 : min(pn, w * P + P);
                    float a = 0.f;  // integers below 2^24, exact in any order
                    for (int i = i0; i < i1; ++i) {
                        a += piece[0][wq][i];
                        lo += piece[1][wq][i];
                    }
                    hi += a;
                    if (nwin > 1) ws[(int64_t)(p0 / P + w) * NT * 4] = start * a;
                }
            __syncthreads();
        }
        if (warp < 4) {
            hi = warp_sum(hi);
            lo = warp_sum(lo);
            if (lane == 0) {
                if (nwin == 1) ws[0] = start * hi;
                qseg[((pass * gridDim.y + s) * NT + nt) * 4 + wq] =
                    make_float4(scalbnf(1.f, -exponent(wq)), hi,
                                -(float)((1 << bits) - 1) * 0x1p-12f * lo, 0.f);
            }
        }
    }
    // ---- the columns, a K step to a warp
    const int sharing = max(1, (int)gridDim.z - 1), slice = gridDim.z > 1 ? (int)blockIdx.z - 1 : 0;
    if (slice < 0) return;
    const int b = lane >> 3;
    const bool lo = (lane >> 2) & 1, live = q0 + b < nq;
    const float scale = scalbnf(1.f, exponent(b));
    const float *p = src + (int64_t)b * dk;
    uint2 *out = bfrag + ((pass * steps + t.s[s].step) * NT + nt) * 32 + lane;
#pragma unroll 2
    for (int step = slice * kSplitWarps + warp; step < 4 * words; step += kSplitWarps * sharing) {
        float x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = step_coord(words, step, lane & 3, i);
            const float y = live && c < len ? __ldg(p + c) * scale : 0.f;
            const float r = split_hi(y);
            x[i] = lo ? split_lo(y, r) : r;
        }
        const __half2 h0 = __floats2half2_rn(x[0], x[1]), h1 = __floats2half2_rn(x[2], x[3]);
        out[(int64_t)step * NT * 32] =
            make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
    }
}

// ------------------------------------------------------------ the vectors
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t select_bits(uint32_t m, uint32_t a, uint32_t b) {
    return (a & m) | (b & ~m);
}

// 32 coordinates of one vector from their plane words: planes are transposed
// by 4 x 4 bit blocks into words whose nibble j is the code (or four bits of
// it) of bit 4 j + r, in 16 operations for 32 codes.
__device__ __forceinline__ void transpose4(uint32_t (&w)[4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint32_t a = w[q], b = w[q + 2];
        w[q] = select_bits(0x33333333u, a, b << 2);
        w[q + 2] = select_bits(0x33333333u, a >> 2, b);
    }
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
        const uint32_t a = w[q], b = w[q + 1];
        w[q] = select_bits(0x55555555u, a, b << 1);
        w[q + 1] = select_bits(0x55555555u, a >> 1, b);
    }
}
// NP planes (4 or 8), least significant first; planes past the code's width
// are zero.  Two widths only: eight instantiations in one switch took 190
// registers (each alone under 80).
template <int NP> struct Codes {
    uint32_t even[4], odd[4];  // bytes j: the codes of bits 8 j + r and 8 j + 4 + r
    __device__ __forceinline__ void split(const uint32_t (&p)[NP]) {
        uint32_t l[4] = {p[0], p[1], p[2], p[3]};
        transpose4(l);
        if constexpr (NP == 4) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                even[r] = l[r] & 0x0F0F0F0Fu;
                odd[r] = (l[r] >> 4) & 0x0F0F0F0Fu;
            }
        } else {
            uint32_t h[4] = {p[4], p[5], p[6], p[7]};
            transpose4(h);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                even[r] = select_bits(0x0F0F0F0Fu, l[r], h[r] << 4);
                odd[r] = select_bits(0x0F0F0F0Fu, l[r] >> 4, h[r]);
            }
        }
    }
    // the codes of bits 4 k + r (low half) and 4 k + r + 16
    __device__ __forceinline__ uint32_t pair(int k, int r) const {
        return __byte_perm((k & 1) ? odd[r] : even[r], 0u, (k & 2) ? 0x4341 : 0x4240);
    }
    __device__ __forceinline__ uint32_t sum2(uint32_t s) const {  // s + sum c^2
#pragma unroll
        for (int r = 0; r < 4; ++r) s = __dp4a(odd[r], odd[r], __dp4a(even[r], even[r], s));
        return s;
    }
};

struct EstArgs {
    const uint8_t *codes;
    int64_t code_stride;
    const float *factors;
    int nf;
    int64_t n;
    int nk;
    const uint2 *bfrag;
    int steps;
    const float *qn2;
    const float *wstart;  // of a pass, per window and query (see k_query_split)
    const float4 *qseg;   // of a pass, per segment and query
    int windows;          // of all segments
    int64_t nq;
    const float *qsig;  // staged: sigma of (query, segment)
    float m_conf;
    float *out;
};

// The K steps of one decoded 32-bit piece (NS = 8) or 16-bit one (4): A
// fragments from the codes and NT products per step.
template <int NP, int NT, int MT, int NS>
__device__ __forceinline__ void run_steps(const Codes<NP> (&cd)[MT][2], const uint2 *__restrict__ b,
                                          float (&acc)[MT][NT][4]) {
#pragma unroll
    for (int m = 0; m < NS; ++m) {
        const int k = m >> 1, r = 2 * (m & 1);
        uint32_t a[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            a[mt][0] = cd[mt][0].pair(k, r);
            a[mt][1] = cd[mt][1].pair(k, r);
            a[mt][2] = cd[mt][0].pair(k, r + 1);
            a[mt][3] = cd[mt][1].pair(k, r + 1);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const uint2 bv = b[(m * NT + nt) * 32];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                mma16816(acc[mt][nt], a[mt][0], a[mt][1], a[mt][2], a[mt][3], bv.x, bv.y);
        }
    }
}

// Part of a plane word (or a factor) from the staged record (SM) or from
// global memory.
template <bool SM, class T> __device__ __forceinline__ T load_rec(const void *p) {
    if constexpr (SM) return *static_cast<const T *>(p);
    else return __ldg(static_cast<const T *>(p));
}

// A window's accumulators at its start (ws: the lane's query's of the first B
// tile), and what it adds to <u, q> at its end: 2 <c - 2^(b-1), hi> and
// 2 <c, lo> / 4096, from sums that are times 2^-24.
template <bool BS, int NT, int MT>
__device__ __forceinline__ void open_window(const float *__restrict__ ws, float (&acc)[MT][NT][4]) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const float h = load_rec<BS, float>(ws + 4 * nt);
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            acc[mt][nt][0] = acc[mt][nt][2] = h;
            acc[mt][nt][1] = acc[mt][nt][3] = 0.f;
        }
    }
}
template <int NT, int MT>
__device__ __forceinline__ void close_window(const float (&acc)[MT][NT][4], float (&tot)[MT][NT][2]) {
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                tot[mt][nt][h] = fmaf(fmaf(acc[mt][nt][2 * h + 1], 0x1p-12f, acc[mt][nt][2 * h]), 0x1p25f,
                                      tot[mt][nt][h]);
}

// The products of one segment of `bits` bits (its first planes; at most NP)
// for the warp's rows (row pointers at the segment's codes).  tot = <u, q>
// (scaled), S2 += sum c^2 and S1 += sum c over the lane's coordinates.  ws and
// qs: wstart and qseg of the segment at the lane's query of the first B tile (4 NT
// of them a window or segment).
template <int NP, int NT, int MT, bool SM, bool BS>
__device__ __forceinline__ void run_segment(const uint8_t *const (&rp)[MT][2], int bits, int words,
                                            int len, int t, const uint2 *__restrict__ b,
                                            const float *__restrict__ ws,
                                            const float4 *__restrict__ qs,
                                            float (&tot)[MT][NT][2],
                                            uint32_t (&S2)[MT][2], uint32_t (&S1)[MT][2]) {
    float acc[MT][NT][4];
    open_window<BS, NT, MT>(ws, acc);
    // sum hi is small beside <u, q> from 5 bits up
    if constexpr (NP > kNarrow)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float4 c = load_rec<BS, float4>(qs + 4 * nt);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) tot[mt][nt][0] = tot[mt][nt][1] = c.y + c.z;
        }
    // the window ends before piece i (one window up to kNarrow bits, where
    // NP is 4)
    const int P = window_pieces(bits);
    auto window_ends = [&](int i) {
        if constexpr (NP > kNarrow) {
            if (i == 0 || (i & (P - 1)) != 0) return;  // uniform
            close_window<NT, MT>(acc, tot);
            ws += 4 * NT;
            open_window<BS, NT, MT>(ws, acc);
        }
    };
    const bool partial = (len & 63) != 0;  // bits past the end are to read as zero
    // sum of the codes of one lane's plane words
    auto code_sum = [](const uint32_t (&w)[NP]) {
        uint32_t x = 0u;
#pragma unroll
        for (int p = NP - 1; p >= 0; --p) x = 2u * x + (uint32_t)__popc(w[p]);
        return x;
    };
    const int full = words >> 2, pieces = 2 * full + ((words >> 1) & 1);
    const uint32_t stride = (uint32_t)words * 8u;  // bytes of a plane
    // byte offset in a plane of the lane's 32 bits of piece i
    auto piece_at = [&](int i) -> uint32_t {
        return i < 2 * full ? (uint32_t)((((i >> 1) * 4 + t) << 3) + ((i & 1) << 2))
                            : (uint32_t)(32 * full + 4 * t);
    };
    const uint32_t last = (uint32_t)(bits - 1) * stride;  // the least significant plane
    uint32_t nx[MT][2][NP];
    auto fetch = [&](int i) {
        uint32_t at = piece_at(i) + last;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            // an offset the compiler cannot split: it would keep a 64-bit
            // pointer per row and plane in registers otherwise
            asm volatile("" : "+r"(at));
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    nx[mt][h][p] = p < bits ? load_rec<SM, uint32_t>(rp[mt][h] + at) : 0u;
            at -= stride;
        }
    };
    // a staged record is read when it is needed, as the registers that hold the
    // next piece cost warps or spills (100 queries x 100K at 8 b/dim read ahead
    // 717 us, so 675; 1 x 1M at 4 b/dim 278 and 271)
    constexpr bool kAhead = !SM;
    if (kAhead && pieces > 0) fetch(0);
#pragma unroll 1
    for (int i = 0; i < pieces; ++i) {
        if constexpr (!kAhead) fetch(i);
        if (partial) {
            const int left = len - (int)piece_at(i) * 8;
            const uint32_t keep = left >= 32 ? ~0u : left <= 0 ? 0u : (1u << left) - 1u;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int p = 0; p < NP; ++p) nx[mt][h][p] &= keep;
        }
        Codes<NP> cd[MT][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                S1[mt][h] += code_sum(nx[mt][h]);
                cd[mt][h].split(nx[mt][h]);
                S2[mt][h] = cd[mt][h].sum2(S2[mt][h]);
            }
        if (kAhead && i + 1 < pieces) fetch(i + 1);
        window_ends(i);
        run_steps<NP, NT, MT, 8>(cd, b, acc);
        b += 8 * NT * 32;
    }
    if (words & 1) {
        const uint32_t at = (uint32_t)(words - 1) * 8u + 2u * (uint32_t)t;
        const int left = len - (int)at * 8;
        const uint32_t keep = left >= 16 ? 0xFFFFu : left <= 0 ? 0u : (1u << left) - 1u;
        Codes<NP> cd[MT][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t w[NP];
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const uint32_t x =
                        p < bits ? load_rec<SM, uint16_t>(rp[mt][h] + (at + last - p * stride)) & keep : 0u;
                    w[p] = __byte_perm(x, 0u, 0x2120);  // byte 0 at bits 0, byte 1 at bits 16
                }
                S1[mt][h] += code_sum(w);
                cd[mt][h].split(w);
                S2[mt][h] = cd[mt][h].sum2(S2[mt][h]);
            }
        window_ends(pieces);
        run_steps<NP, NT, MT, 4>(cd, b, acc);
    }
    if constexpr (NP > kNarrow) {
        close_window<NT, MT>(acc, tot);
    } else {
        // an exact <u, hi> (at one bit it is small beside its parts), then lo's
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float4 c = load_rec<BS, float4>(qs + 4 * nt);
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    tot[mt][nt][h] = fmaf(acc[mt][nt][2 * h], 0x1p25f, c.y) +
                                     fmaf(acc[mt][nt][2 * h + 1], 0x1p13f, c.z);
        }
    }
}

// Asynchronous copies of 16, 8 or 4 bytes into shared memory.
template <int BYTES> __device__ __forceinline__ void copy_async(void *dst, const void *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES)
                     : "memory");
}

// A warp's 16 code records (rows at `stride` bytes in shared memory) and
// their factors, rows [r0, r0 + rows).
__device__ __forceinline__ void stage_tile(const EstArgs &A, int64_t r0, int rows, uint8_t *dst,
                                           int stride, float *fdst, int lane) {
    const uint8_t *src = A.codes + r0 * A.code_stride;
    const bool wide = (A.code_stride & 15) == 0;
    const int unit = wide ? 16 : 8, per = (int)A.code_stride / unit;
    int r = 0, c = lane;
    for (;;) {
        while (c >= per && r < rows) {
            c -= per;
            ++r;
        }
        if (r >= rows) break;
        if (wide) copy_async<16>(dst + r * stride + c * 16, src + (int64_t)r * A.code_stride + c * 16);
        else copy_async<8>(dst + r * stride + c * 8, src + (int64_t)r * A.code_stride + c * 8);
        c += 32;
    }
    const float *f = A.factors + r0 * A.nf;
    for (int e = lane; e < rows * A.nf; e += 32) copy_async<4>(fdst + e, f + e);
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Shared memory of a pass's wstart and qseg.
__host__ __device__ constexpr size_t table_bytes(int windows, int segments, int NT) {
    return (size_t)(windows + 4 * segments) * 4 * NT * sizeof(float);
}

// Warps of a block of the staged form: as many as their registers allow.
__host__ __device__ constexpr int staged_warps(int NT) { return NT <= 4 ? 24 : 12; }

// A warp takes tiles of 16 MT vectors; the block's NT B columns (4 NT queries
// of pass blockIdx.y) stay in shared memory (BS) for all of its tiles.
// SM: the tile's code records and factors are copied to the warp's own buffer
// in shared memory first (asynchronously, as soon as the previous tile is
// done), so that the loads of the decode take 30 cycles instead of an L2 or
// HBM round trip at the start of every segment; the other warps of the SM
// cover the copy.
// Bound by the instructions of the decode: 1 query x 1M records of 480 B 4,350 ->
// 271 us, 100 x 100K 22,600 -> 227 us, against a warp per (query, vector) that
// decoded a bit per plane and lane.
// Measured on the way: decode to FP16 integers by two more FP16 operations
// per pair 405 us, |u|^2 from two more products per step (their diagonals)
// 360 us, records read from global memory by every lane 390 us.
template <int NT, int MT, bool BS, bool STAGED, bool SM>
__global__ void __launch_bounds__(SM ? 32 * staged_warps(NT) : 256, 1)
k_estimate_mma(const EstArgs A, const __grid_constant__ SegTable tab, int sstride) {
    static_assert(!SM || MT == 1, "a staged tile holds 16 records");
    extern __shared__ __align__(16) uint2 bsm[];
    __shared__ float s_qn2[4 * NT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int64_t q0 = (int64_t)blockIdx.y * 4 * NT;
    const uint2 *bg = A.bfrag + (int64_t)blockIdx.y * A.steps * NT * 32;
    const int64_t tiles = (A.n + 16 * MT - 1) / (16 * MT), tstep = (int64_t)gridDim.x * warps;
    int64_t tile = (int64_t)blockIdx.x * warps + warp;
    // the pass's wstart and qseg, beside B where that is shared
    const float *wstart = A.wstart + (int64_t)blockIdx.y * A.windows * (4 * NT);
    const float4 *qseg = A.qseg + (int64_t)blockIdx.y * A.nk * (4 * NT);
    float4 *tabs = reinterpret_cast<float4 *>(bsm + (BS ? A.steps * NT * 32 : 0));
    // the warp's buffer: 16 records, then their factors
    uint8_t *buf = reinterpret_cast<uint8_t *>(tabs) + (BS ? table_bytes(A.windows, A.nk, NT) : 0) +
                   (SM ? warp * (16 * sstride + ((64 * A.nf + 15) & ~15)) : 0);
    float *fbuf = reinterpret_cast<float *>(buf + 16 * sstride);
    if (SM && tile < tiles)
        stage_tile(A, tile * 16, (int)min((int64_t)16, A.n - tile * 16), buf, sstride, fbuf, lane);
    if constexpr (BS)
        for (int e = threadIdx.x; e < A.steps * NT * 16; e += blockDim.x)
            reinterpret_cast<uint4 *>(bsm)[e] = __ldg(reinterpret_cast<const uint4 *>(bg) + e);
    if constexpr (BS) {
        const int nw = A.windows * (4 * NT), ns = A.nk * (4 * NT);
        float *ws = reinterpret_cast<float *>(tabs + ns);
        for (int e = threadIdx.x; e < ns; e += blockDim.x) tabs[e] = __ldg(qseg + e);
        for (int e = threadIdx.x; e < nw; e += blockDim.x) ws[e] = __ldg(wstart + e);
        qseg = tabs;
        wstart = ws;
    }
    for (int e = threadIdx.x; e < 4 * NT; e += blockDim.x) {
        const int64_t q = q0 + e;
        s_qn2[e] = q < A.nq ? A.qn2[q] : 0.f;
    }
    __syncthreads();
    const uint2 *b0 = (BS ? bsm : bg) + lane;
    for (; tile < tiles; tile += tstep) {
        int64_t v[MT][2];
        const float *fac[MT][2];
        const uint8_t *rec[MT][2];
        if constexpr (SM) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
        }
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                v[mt][h] = tile * (16 * MT) + mt * 16 + h * 8 + g;
                if constexpr (SM) {  // rows past n: whatever the buffer holds
                    fac[mt][h] = fbuf + (h * 8 + g) * A.nf;
                    rec[mt][h] = buf + (h * 8 + g) * sstride;
                } else {
                    const int64_t r = min(v[mt][h], A.n - 1);  // rows past n repeat the last one
                    fac[mt][h] = A.factors + r * A.nf;
                    rec[mt][h] = A.codes + r * A.code_stride;
                }
            }
        float est[MT][NT][2];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) est[mt][nt][0] = est[mt][nt][1] = 0.f;
        auto store = [&](int stage) {
            // value after `stage` segments (or the distance itself)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (v[mt][h] >= A.n) continue;
                    const float f0 = load_rec<SM, float>(fac[mt][h]);
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt) {
                        const int64_t q = q0 + 4 * nt + t;
                        if (q >= A.nq) continue;
                        const float base = f0 + s_qn2[4 * nt + t];
                        const float e = est[mt][nt][h];
                        if constexpr (STAGED) {
                            float rest = 0.f;  // m * sum_{s >= stage} sigma_s
                            for (int s = stage; s < A.nk; ++s) rest += __ldg(A.qsig + q * A.nk + s);
                            rest *= A.m_conf;
                            A.out[(q * A.n + v[mt][h]) * (A.nk + 1) + stage] = base - 2.f * (e + rest);
                        } else {
                            A.out[q * A.n + v[mt][h]] = base - 2.f * e;
                        }
                    }
                }
        };
        if constexpr (STAGED) store(0);
        for (int s = 0; s < A.nk; ++s) {
            const SegDesc &sg = tab.s[s];
            const int bits = sg.bits;
            const uint8_t *rp[MT][2];
            float tot[MT][NT][2];
            uint32_t S2[MT][2], S1[MT][2];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                rp[mt][0] = rec[mt][0] + sg.code_off;
                rp[mt][1] = rec[mt][1] + sg.code_off;
                S2[mt][0] = S2[mt][1] = 0u;
                S1[mt][0] = S1[mt][1] = 0u;
            }
            // the two factors of one of the lane quad's rows in each of its lanes
            const float *fv = fac[0][0];
#pragma unroll
            for (int i = 1; i < 2 * MT; ++i)
                if (t % (2 * MT) == i) fv = fac[i >> 1][i & 1];
            float nrm, cosine;
            auto factors = [&] {
                nrm = load_rec<SM, float>(fv + sg.fidx);
                cosine = load_rec<SM, float>(fv + sg.fidx + 1);
            };
            // (before the products, unless the registers run short)
            if constexpr (NT > 1) factors();
            const uint2 *b = b0 + sg.step * NT * 32;
            const float *ws = wstart + sg.window * (4 * NT) + t;
            const float4 *qs = qseg + s * (4 * NT) + t;
            if (bits <= kNarrow)  // uniform
                run_segment<4, NT, MT, SM, BS>(rp, bits, sg.words, sg.len, t, b, ws, qs, tot, S2, S1);
            else
                run_segment<8, NT, MT, SM, BS>(rp, bits, sg.words, sg.len, t, b, ws, qs, tot, S2, S1);
            if constexpr (NT == 1) factors();
            // |u|^2 = 4 (sum c^2 - cmax sum c) + len cmax^2, the sums spread
            // over the quad; lane t forms the scale of row t % (2 MT)
            const int cmax = (1 << bits) - 1;
            long long c2 = 0;
#pragma unroll
            for (int i = 0; i < 2 * MT; ++i) {
                const uint32_t s2 = S2[i >> 1][i & 1], s1 = S1[i >> 1][i & 1];
                long long x;
                if (sg.len > 65536) {  // uniform
                    x = (long long)s2 - (long long)cmax * s1;
                    x += __shfl_xor_sync(0xffffffffu, x, 1);
                    x += __shfl_xor_sync(0xffffffffu, x, 2);
                } else {
                    uint32_t lo = s2 - (uint32_t)cmax * s1;
                    lo += __shfl_xor_sync(0xffffffffu, lo, 1);
                    lo += __shfl_xor_sync(0xffffffffu, lo, 2);
                    x = lo;
                }
                if (t % (2 * MT) == i) c2 = x;
            }
            // (modulo 2^32 |u|^2 is exact up to 66,051 coordinates of 8 bits)
            const float S = sg.len > 65536
                                ? (float)(4ll * c2 + (long long)sg.len * (cmax * cmax))
                                : (float)(4u * (uint32_t)c2 + (uint32_t)sg.len * (uint32_t)(cmax * cmax));
            const float vs = nrm > 0.f ? nrm / (sqrtf(S) * cosine) : 0.f;
            float vsr[MT][2];
#pragma unroll
            for (int i = 0; i < 2 * MT; ++i)
                vsr[i >> 1][i & 1] = __shfl_sync(0xffffffffu, vs, (g << 2) | i);
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const float inv = load_rec<BS, float>(qs + 4 * nt);
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        est[mt][nt][h] = fmaf(tot[mt][nt][h] * inv, vsr[mt][h], est[mt][nt][h]);
            }
            if constexpr (STAGED) store(s + 1);
        }
        if constexpr (!STAGED) store(0);
        if constexpr (SM) {
            __syncwarp();  // every lane is done with the buffer
            const int64_t next = tile + tstep;
            if (next < tiles)
                stage_tile(A, next * 16, (int)min((int64_t)16, A.n - next * 16), buf, sstride, fbuf,
                           lane);
        }
    }
}

SegTable seg_table(const saq_model *m, int prefix_bits) {
    SegTable t{};
    int step = 0, window = 0;
    for (size_t i = 0; i < m->kept.size(); ++i) {
        const KeptSeg &k = m->kept[i];
        const int bits = used_bits(prefix_bits, k.bits);
        t.s[i] = SegDesc{k.off, k.len, bits, k.words, k.fidx, step, window, (long long)k.code_off};
        step += 4 * k.words;
        window += window_count(bits, k.words);
    }
    return t;
}

// K steps of 16 coordinates over all kept segments.
int total_steps(const saq_model *m) {
    int steps = 0;
    for (const KeptSeg &k : m->kept) steps += 4 * k.words;
    return steps;
}

// Windows over all kept segments.
int total_windows(const saq_model *m, int prefix_bits) {
    int n = 0;
    for (const KeptSeg &k : m->kept) n += window_count(used_bits(prefix_bits, k.bits), k.words);
    return n;
}

constexpr size_t kEstSmemMax = 224 * 1024;  // dynamic shared memory of a block

// Row stride of the staged records: 32 or 96 bytes past a multiple of 128, so
// that the eight rows a quad column reads fall into four bank groups.
int staged_stride(const saq_model *m) {
    const int s = ((int)m->code_bytes + 31) / 32 * 32;
    return s % 64 == 32 ? s : s + 32;
}
// Bytes of a warp's buffer (16 records and their factors).
size_t staged_bytes(const saq_model *m) {
    return (size_t)16 * staged_stride(m) + (((size_t)64 * m->nf + 15) & ~(size_t)15);
}

struct EstPlan {
    int NT = 1, steps = 0;
    int64_t passes = 1;
    bool bs = true;  // B in shared memory (else read through the caches)
    int warps = 0;   // staged form: warps per block (0: the form without staging)
};
// Bytes of a block's B columns and their tables.
size_t column_bytes(const saq_model *m, int NT) {
    return (size_t)total_steps(m) * NT * 256 + table_bytes(total_windows(m, 0), (int)m->kept.size(), NT);
}
// 4 NT queries per pass: the fewest passes whose B columns fit in shared
// memory, then the smallest form that still does them in that many.  Records
// are staged when the buffers of at least eight warps fit beside B.
EstPlan est_plan(const saq_model *m, int64_t nq) {
    static const int forms[] = {1, 4, 8};
    EstPlan p;
    p.steps = total_steps(m);
    const int64_t nts = (nq + 3) / 4;
    const size_t wb = staged_bytes(m);
    const auto choose = [&](size_t beside) {
        int most = 0;
        for (int f : forms)
            if (column_bytes(m, f) + beside <= kEstSmemMax) most = f;
        if (!most) return false;
        const int64_t need = (nts + (nts + most - 1) / most - 1) / ((nts + most - 1) / most);
        for (int f : forms)
            if (f >= need) {
                p.NT = f;
                break;
            }
        p.passes = (nts + p.NT - 1) / p.NT;
        return true;
    };
    if (choose(8 * wb)) {
        const int fit = (int)((kEstSmemMax - column_bytes(m, p.NT)) / wb);
        p.warps = std::min(staged_warps(p.NT), fit);
    } else if (!choose(0)) {
        p.bs = false;
        p.NT = 1;
        p.passes = nts;
    }
    return p;
}

template <int NT, int MT, bool BS, bool STAGED, bool SM>
saq_status launch_form(const EstArgs &a, const SegTable &t, const EstPlan &p, int sstride,
                       size_t cb, size_t wb, cudaStream_t s) {
    const auto kernel = k_estimate_mma<NT, MT, BS, STAGED, SM>;
    const int warps = SM ? p.warps : 8;
    const size_t smem = (BS ? cb : 0) + (SM ? warps * wb : 0);
    int dev = 0, sms = 0, per_sm = 0;
    SAQ_CUDA_CHECK(cudaGetDevice(&dev));
    SAQ_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SAQ_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kEstSmemMax));
    SAQ_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, warps * 32, smem));
    const int64_t tiles = (a.n + 16 * MT - 1) / (16 * MT);
    for (int64_t p0 = 0; p0 < p.passes; p0 += 65535) {
        const int64_t np = std::min<int64_t>(65535, p.passes - p0);
        // the passes share the SMs; a block keeps its B columns over its tiles.
        // No more blocks than are resident at once: seven passes of 22 on 152
        // SMs left two for a wave of their own (100 queries x 100K at 8 b/dim
        // 675 -> 375 us)
        const int64_t each = std::max<int64_t>(1, (int64_t)sms * std::max(1, per_sm) / np);
        // few tiles: as many blocks as there are SMs to take them
        int w = warps;
        if (SM) w = (int)std::max<int64_t>(4, std::min<int64_t>(w, (tiles + each - 1) / each));
        w = std::min(w, warps);
        EstArgs b = a;
        b.bfrag += p0 * a.steps * NT * 32;
        b.qn2 += p0 * 4 * NT;
        b.wstart += p0 * a.windows * 4 * NT;
        b.qseg += p0 * a.nk * 4 * NT;
        if (STAGED) b.qsig += p0 * 4 * NT * a.nk;
        b.nq -= p0 * 4 * NT;
        b.out += p0 * 4 * NT * a.n * (STAGED ? a.nk + 1 : 1);
        {
            LaunchTimer lt_(kKindOther, s);
            kernel<<<dim3((unsigned)std::min((tiles + w - 1) / w, each), (unsigned)np), w * 32, smem,
                     s>>>(b, t, sstride);
        }
        note_launches();
    }
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

template <bool STAGED>
saq_status launch_forms(const saq_model *m, const EstArgs &a, const SegTable &t, const EstPlan &p,
                        cudaStream_t s) {
    const int ss = staged_stride(m);
    const size_t cb = column_bytes(m, p.NT), wb = staged_bytes(m);
    if (!p.bs) return launch_form<1, 1, false, STAGED, false>(a, t, p, ss, cb, wb, s);
    if (p.warps > 0) {
        switch (p.NT) {
            case 1: return launch_form<1, 1, true, STAGED, true>(a, t, p, ss, cb, wb, s);
            case 4: return launch_form<4, 1, true, STAGED, true>(a, t, p, ss, cb, wb, s);
            default: return launch_form<8, 1, true, STAGED, true>(a, t, p, ss, cb, wb, s);
        }
    }
    switch (p.NT) {
        case 1: return launch_form<1, 1, true, STAGED, false>(a, t, p, ss, cb, wb, s);
        case 4: return launch_form<4, 1, true, STAGED, false>(a, t, p, ss, cb, wb, s);
        default: return launch_form<8, 2, true, STAGED, false>(a, t, p, ss, cb, wb, s);
    }
}

// out = (Q - c) M^T (nq x dk) for a dk x d matrix.
saq_status launch_query_rot(const saq_model *m, const float *Q, int64_t nq, const float *M,
                            float *out, float *qn2, cudaStream_t s) {
    // a few queries: one column per warp, so that the rows of M spread over
    // the chip; more: eight queries share each row read
    const bool one = nq <= 2;
    const int qb = one ? 1 : 8, cpw = one ? 1 : 4;
    const unsigned gx = (unsigned)((m->dk + 8 * cpw - 1) / (8 * cpw));
    const bool v4 = m->d % 4 == 0;
    for (int64_t q0 = 0; q0 < nq; q0 += (int64_t)65535 * qb) {
        const int64_t n = std::min<int64_t>(nq - q0, (int64_t)65535 * qb);
        const dim3 grid(gx, (unsigned)((n + qb - 1) / qb));
        const float *Qp = Q + q0 * m->d;
        float *op = out + q0 * m->dk;
        float *np = qn2 ? qn2 + q0 : nullptr;
        LaunchTimer lt_(kKindProject, s);
        if (one && v4) k_query_rot<1, 1, true><<<grid, 256, 0, s>>>(Qp, n, m->d, m->d_mean, M, m->dk, op, np);
        else if (one) k_query_rot<1, 1, false><<<grid, 256, 0, s>>>(Qp, n, m->d, m->d_mean, M, m->dk, op, np);
        else if (v4) k_query_rot<8, 4, true><<<grid, 256, 0, s>>>(Qp, n, m->d, m->d_mean, M, m->dk, op, np);
        else k_query_rot<8, 4, false><<<grid, 256, 0, s>>>(Qp, n, m->d, m->d_mean, M, m->dk, op, np);
        note_launches();
    }
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch: rotated queries, |q - c|^2, wstart and qseg, B fragments and, for the staged bounds, the basis values
// and sigma of (query, segment).
struct EstScratch {
    float *qrot, *qn2, *wstart, *pc, *qsig;
    float4 *qseg;
    uint2 *bfrag;
    size_t bytes;
};
EstScratch est_scratch(const saq_model *m, int64_t nq, const EstPlan &p, bool staged, void *base) {
    EstScratch r{};
    size_t at = 0;
    auto take = [&](size_t bytes) {
        uint8_t *q = static_cast<uint8_t *>(base) + at;
        at += align256(bytes);
        return q;
    };
    const size_t dk = (size_t)std::max(1, m->dk), q = (size_t)nq;
    r.qrot = (float *)take(4 * q * dk);
    r.qn2 = (float *)take(4 * q);
    // (a prefix has no more windows)
    const size_t queries = (size_t)p.passes * p.NT * 4;
    r.wstart = (float *)take(4 * queries * (size_t)total_windows(m, 0));
    r.qseg = (float4 *)take(16 * queries * m->kept.size());
    r.bfrag = (uint2 *)take((size_t)p.passes * p.steps * p.NT * 256);
    if (staged) {
        r.pc = (float *)take(4 * q * dk);
        r.qsig = (float *)take(4 * q * std::max<size_t>(1, m->kept.size()));
    }
    r.bytes = at;
    return r;
}

}  // namespace

size_t estimate_scratch_bytes(const saq_model *m, int64_t nq, bool staged) {
    return est_scratch(m, nq, est_plan(m, nq), staged, nullptr).bytes;
}

saq_status launch_estimate(const saq_model *m, const uint8_t *codes, const float *factors,
                           int64_t n, const float *Q, int64_t nq, int prefix_bits, bool staged,
                           float m_conf, void *scratch, float *out, cudaStream_t s) {
    const int nk = (int)m->kept.size();
    if (nk > kMaxSeg) return set_error(SAQ_ERR_UNSUPPORTED, "more than %d kept segments", kMaxSeg);
    const SegTable t = seg_table(m, prefix_bits);
    const EstPlan p = est_plan(m, nq);
    const EstScratch w = est_scratch(m, nq, p, staged, scratch);
    const int windows = total_windows(m, prefix_bits);
    if (nk == 0) {
        saq_status st = launch_rownorm2(m, Q, nq, w.qn2, 1, s);
        if (st != SAQ_OK) return st;
    } else {
        saq_status st = launch_query_rot(m, Q, nq, m->d_W, w.qrot, w.qn2, s);
        if (st != SAQ_OK) return st;
        // a few queries: blocks that share a segment's steps, a step per warp at
        // most, up to two blocks to an SM
        int dev = 0, sms = 0, steps = 0;
        SAQ_CUDA_CHECK(cudaGetDevice(&dev));
        SAQ_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        for (const KeptSeg &k : m->kept) steps = std::max(steps, 4 * k.words);
        const int64_t blocks = p.passes * p.NT * nk;
        const int64_t share = std::max<int64_t>(
            1, std::min<int64_t>(1 + (steps + kSplitWarps - 1) / kSplitWarps, 2 * sms / blocks));
        {
            LaunchTimer lt_(kKindOther, s);
            k_query_split<<<dim3((unsigned)(p.passes * p.NT), (unsigned)nk, (unsigned)share),
                            32 * kSplitWarps, 0, s>>>(
                w.qrot, nq, m->dk, t, p.steps, p.NT, windows, w.bfrag, w.wstart, w.qseg);
        }
        note_launches();
        if (staged) {
            st = launch_query_rot(m, Q, nq, m->d_B, w.pc, nullptr, s);
            if (st != SAQ_OK) return st;
            {
                LaunchTimer lt_(kKindOther, s);
                k_query_sigma<<<(unsigned)((nq * nk + 7) / 8), 256, 0, s>>>(w.pc, nq, m->dk, nk, t,
                                                                             w.qsig);
            }
            note_launches();
        }
    }
    EstArgs a;
    a.codes = codes;
    a.code_stride = (int64_t)m->code_bytes;
    a.factors = factors;
    a.nf = m->nf;
    a.n = n;
    a.nk = nk;
    a.bfrag = w.bfrag;
    a.steps = p.steps;
    a.qn2 = w.qn2;
    a.wstart = w.wstart;
    a.qseg = w.qseg;
    a.windows = windows;
    a.nq = nq;
    a.qsig = w.qsig;
    a.m_conf = m_conf;
    a.out = out;
    return staged ? launch_forms<true>(m, a, t, p, s) : launch_forms<false>(m, a, t, p, s);
}

}  // namespace saq
