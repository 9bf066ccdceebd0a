// k_caq1.cu -- quantize, adjust and pack one kept segment with one LANE per
// vector-segment (Sec. 3.1 Eq. find_nearest_code, Eq. adj-obj, Algorithm 1;
// Sec. 4.2 "quantize each segment separately").
//
// The 32 lanes of a warp run Algorithm 1 on 32 different vectors in lockstep
// over the coordinates of the segment: step j takes coordinate j of all 32
// vectors (a 128-byte line of the projected rows, stored interleaved by groups
// of 32 rows: O_i[(g * d_kept + col) * 32 + lane]) and their current codes from
// the warp's code store (packed 8 per batch in shared memory, k_caq1_sm, or in a
// global scratch, k_caq1, when they do not fit there), decides the lane's move
// against that lane's own state and applies it.  Each lane therefore executes
// the paper's sequential scan exactly, and an accepted move costs a predicated
// update instead of a serialising pass.
//
// Decision in closed form, without a division: with I = <u, o> > 0,
// S = |u|^2 and u = 2c - (2^B - 1), moving u_i by 2s (s = +-1) raises
// I^2 / S iff (I + 2 s o_i)^2 S > I^2 (S + 4 s u_i + 4), i.e. iff
//     s T I + o_i^2 S > I^2,   T = o_i S - u_i I.
// Only s = sign(T) can pass (the other side is smaller by 2|T|I), which is
// the convex-cone fact that at most one of +-Delta raises the cosine; the
// paper's -Delta trial after an accepted +Delta returns to the old point and
// is rejected.  The range check of c + s reads s*u < 2^B - 1.  A lane whose
// round made no move stops (its state no longer changes).  v_max comes from
// the projection (or a separate pass).  I and S are tracked in FP32 for the
// decisions; S is recounted exactly from the final codes while they are packed
// into bit-planes, during the last round (or, for a warp whose lanes all stop
// earlier, in a pass of its own).
//
// The kernel is bound by the instructions it issues (79% of the issue slots,
// ncu; its DRAM traffic runs at 4.2 TB/s).  A step took ~26 instructions, and at
// 32 warps per SM each round read the rows from HBM anew.  Now a step is 16 (the
// update predicated instead of branched around, codes turned into u two at a
// time, moves summed as floats), rows come by asynchronous copies of 2 KB per
// warp, which need no registers, and 20 warps per SM keep the issue slots filled
// while a part of the rows they return to stays in L2.  1,000,000 rows at d =
// 960, 4 b/dim 5.11 -> 4.03 ms; 100,000 at d = 1536, 2 b/dim 716 -> 510 us;
// 65,537 at d = 3072, 1 b/dim 471 -> 321 us; a 3,072-long segment at 8 bits of
// 20,011 rows, which waits for its own chain of steps, 1,745 -> 729 us.
#include <algorithm>
#include <atomic>

#include "caq_launch.h"

namespace saq {

namespace {

constexpr int kU = 8;  // coordinates of a batch
// the most shared memory eight warps' codes take
constexpr size_t kCaqSmemMax = 72 * 1024;
constexpr int kWarps = 4;  // of a block
// Fewer warps than this per SM are spread over the SMs in blocks of two: 20,011
// rows of a 3,072-long segment (4.1 warps per SM) 901 -> 849 us, 16,000 rows at
// d = 960 (13) 126.5 -> 124.4.
constexpr int kSpreadWarps = 16;

// (a0, a1) * b + c, one instruction
__device__ __forceinline__ void fma2(float a0, float a1, float b, float c, float &d0, float &d1) {
    asm("{\n.reg .b64 a, b, c, d;\n"
        "mov.b64 a, {%2, %3};\nmov.b64 b, {%4, %4};\nmov.b64 c, {%5, %5};\n"
        "fma.rn.f32x2 d, a, b, c;\nmov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b), "f"(c));
}
__device__ __forceinline__ void add2(float a0, float a1, float b, float &d0, float &d1) {
    asm("{\n.reg .b64 a, b, d;\n"
        "mov.b64 a, {%2, %3};\nmov.b64 b, {%4, %4};\n"
        "add.rn.f32x2 d, a, b;\nmov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b));
}
__device__ __forceinline__ void add2_rz(float a0, float a1, float b, float &d0, float &d1) {
    asm("{\n.reg .b64 a, b, d;\n"
        "mov.b64 a, {%2, %3};\nmov.b64 b, {%4, %4};\n"
        "add.rz.f32x2 d, a, b;\nmov.b64 {%0, %1}, d;\n}"
        : "=f"(d0), "=f"(d1)
        : "f"(a0), "f"(a1), "f"(b));
}

// A batch of kU = 8 codes as it is stored: BITS (1, 2, 4 or 8) bits per code in
// kWords registers, code k in the bits from (k * BITS) % 32 of word k * BITS /
// 32.  `expand` spreads it into words y whose fields the steps read:
//   BITS = 8: the words themselves (code k in byte k & 3 of word k >> 2);
//   BITS = 4: byte k >> 1 of word k & 1;  BITS = 2: byte k >> 2 of word k & 3.
// `u_of` gives u = 2c - cmax of the codes as floats: a byte permute puts c into
// bits 8-15 of the float 2^23 (value 2^23 + 256 c), and an FMA with ucst =
// -(2^16 + cmax), two codes at a time, makes it 2c - cmax, exactly.  At one bit
// u is +-1: the code is its sign.
template <int BITS> struct Fields {
    static constexpr int kWords = BITS == 8 ? 2 : 1;
    static constexpr int kY = BITS == 8 || BITS == 4 ? 2 : BITS == 2 ? 4 : 1;
    static __device__ __forceinline__ void expand(const uint32_t (&w)[kWords], uint32_t (&y)[kY]) {
        if constexpr (BITS == 8) {
            y[0] = w[0];
            y[1] = w[1];
        } else if constexpr (BITS == 4) {
            y[0] = w[0] & 0x0F0F0F0Fu;
            y[1] = (w[0] >> 4) & 0x0F0F0F0Fu;
        } else if constexpr (BITS == 2) {
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = (w[0] >> (2 * j)) & 0x0303u;
        } else {
            y[0] = w[0];
        }
    }
    static __device__ __forceinline__ void u_of(const uint32_t (&w)[kWords], float ucst,
                                                float (&u)[kU]) {
        uint32_t y[kY];
        expand(w, y);
#pragma unroll
        for (int k = 0; k < kU; k += 2) {
            if constexpr (BITS == 1) {
                u[k] = __uint_as_float(((y[0] << (31 - k)) & 0x80000000u) ^ 0xBF800000u);
                u[k + 1] = __uint_as_float(((y[0] << (30 - k)) & 0x80000000u) ^ 0xBF800000u);
            } else {
                float f[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int j = k + i;
                    const int word = BITS == 8 ? j >> 2 : BITS == 4 ? j & 1 : j & 3;
                    const int byte = BITS == 8 ? j & 3 : BITS == 4 ? j >> 1 : j >> 2;
                    f[i] = __uint_as_float(
                        __byte_perm(y[word], 0x4B000000u, 0x7404u | (uint32_t)byte << 4));
                }
                fma2(f[0], f[1], 0.0078125f, ucst, u[k], u[k + 1]);
            }
        }
    }
    // Accepted moves of the batch, summed as floats from 1.5 * 2^23 (whose low
    // bits then are the sum): 16 bits of codes per float, code k with unit
    // 1 << move_bit(k).  `apply` adds them to the words.
    static constexpr int kMoves = BITS == 8 ? 4 : BITS == 4 ? 2 : 1;
    static __device__ __forceinline__ int move_word(int k) { return k * BITS / 16; }
    static __device__ __forceinline__ int move_bit(int k) { return k * BITS % 16; }
    static __device__ __forceinline__ void apply(const float (&mv)[kMoves],
                                                 uint32_t (&w)[kWords]) {
#pragma unroll
        for (int i = 0; i < kWords; ++i) {
            w[i] += __float_as_uint(mv[BITS >= 4 ? 2 * i : 0]) - 0x4B400000u;
            if (BITS >= 4) w[i] += __float_as_uint(mv[BITS >= 4 ? 2 * i + 1 : 0]) << 16;
        }
    }
    // The words of eight codes given as floats 2^23 + c (t) and c (cf): a few
    // codes of one float by FMAs (exact: below 2^24), halves joined by bytes.
    static __device__ __forceinline__ void pack(const float (&t)[kU], const float (&cf)[kU],
                                                uint32_t (&w)[kWords]) {
        constexpr float m = (float)(1 << BITS);
        if constexpr (BITS == 8) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
                w[i] = __byte_perm(__float_as_uint(fmaf(cf[4 * i + 1], m, t[4 * i])),
                                   __float_as_uint(fmaf(cf[4 * i + 3], m, t[4 * i + 2])), 0x5410u);
        } else if constexpr (BITS == 4) {
            float h[2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
                h[i] = fmaf(cf[4 * i + 3], m * m * m,
                            fmaf(cf[4 * i + 2], m * m, fmaf(cf[4 * i + 1], m, t[4 * i])));
            w[0] = __byte_perm(__float_as_uint(h[0]), __float_as_uint(h[1]), 0x5410u);
        } else {
            float h = t[0], s = 1.f;
#pragma unroll
            for (int k = 1; k < kU; ++k) h = fmaf(cf[k], s *= m, h);
            w[0] = __float_as_uint(h) & 0xFFFFu;
        }
    }
    // Bit b of the eight codes as byte b of the result (byte b & 3 of word
    // b >> 2), code k in bit k: delta swaps of the words' bit addresses.
    static __device__ __forceinline__ uint32_t swap(uint32_t x, int sh, uint32_t mask) {
        const uint32_t t = (x ^ (x >> sh)) & mask;
        return x ^ t ^ (t << sh);
    }
    static __device__ __forceinline__ void planes(const uint32_t (&w)[kWords],
                                                  uint32_t (&t)[kWords]) {
        if constexpr (BITS == 8) {
            const uint32_t lo = swap(swap(w[0], 7, 0x00AA00AAu), 14, 0x0000CCCCu);
            const uint32_t hi = swap(swap(w[1], 7, 0x00AA00AAu), 14, 0x0000CCCCu);
            t[0] = (lo & 0x0F0F0F0Fu) | ((hi << 4) & 0xF0F0F0F0u);
            t[1] = ((lo >> 4) & 0x0F0F0F0Fu) | (hi & 0xF0F0F0F0u);
        } else if constexpr (BITS == 4) {
            t[0] = swap(swap(swap(swap(w[0], 14, 0x0000CCCCu), 7, 0x00AA00AAu), 2, 0x0C0C0C0Cu), 1,
                        0x22222222u);
        } else if constexpr (BITS == 2) {
            t[0] = swap(swap(swap(w[0], 7, 0x00AAu), 3, 0x0A0Au), 1, 0x2222u);
        } else {
            t[0] = w[0];
        }
    }
};

// The projected rows of a warp's 32 vector-segments, copied into shared memory
// ahead of their steps: D slots of kSlotCols coordinates (two batches, 2 KB on
// end).  The passes over the segment (initial codes, rounds) form one stream of
// slots that wraps around, so the copies run on across rounds.  With CODES a
// slot also takes its whole batches' codes from the global scratch.
constexpr int kSlotCols = 2 * kU;
template <int D, bool CODES> struct Ring {
    static constexpr int kRows = kSlotCols * 128, kSlot = kRows + (CODES ? kSlotCols * 32 : 0);
    static constexpr int kBytes = D * kSlot;
    uint8_t *sm;         // the warp's slots, 16-byte aligned
    const float *rows;   // the segment's first coordinate of the warp's rows
    const uint8_t *codes;
    int len, lane;
    int next;  // first coordinate of the slot to copy next
    int slot;  // byte offset of the slot in use

    template <int OFF> static __device__ __forceinline__ void copy16(uint32_t dst, const void *src) {
        asm volatile("cp.async.cg.shared.global [%0 + %2], [%1 + %2], 16;" ::"r"(dst), "l"(src),
                     "n"(OFF)
                     : "memory");
    }
    __device__ __forceinline__ void issue(int at) {
        const int n = len - next;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(sm) + at + lane * 16;
        const uint8_t *src =
            reinterpret_cast<const uint8_t *>(rows + ((int64_t)next << 5)) + lane * 16;
        const uint8_t *csrc = CODES ? codes + ((int64_t)next << 5) + lane * 16 : nullptr;
        if (n >= kSlotCols) {
            copy16<0>(d, src);
            copy16<512>(d, src);
            copy16<1024>(d, src);
            copy16<1536>(d, src);
            if (CODES) copy16<0>(d + kRows, csrc);
        } else {
            if (lane < 8 * n) copy16<0>(d, src);
            if (lane + 32 < 8 * n) copy16<512>(d, src);
            if (lane + 64 < 8 * n) copy16<1024>(d, src);
            if (lane + 96 < 8 * n) copy16<1536>(d, src);
            if (CODES && n >= kU && lane < 16) copy16<0>(d + kRows, csrc);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        next = n > kSlotCols ? next + kSlotCols : 0;
    }
    __device__ __forceinline__ void start() {
        next = slot = 0;
#pragma unroll 1
        for (int i = 0; i < D; ++i) issue(i * kSlot);
    }
    // the next slot is complete
    __device__ __forceinline__ void wait() const {
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
        __syncwarp();
    }
    // the rows of batch h of the slot (those past the segment's end are not to
    // be used), and its codes
    __device__ __forceinline__ void take(int h, float (&x)[kU]) const {
        const float *p = reinterpret_cast<const float *>(sm + slot + h * (kU * 128)) + lane;
#pragma unroll
        for (int k = 0; k < kU; ++k) x[k] = p[k * 32];
    }
    __device__ __forceinline__ void take_codes(int h, uint32_t (&w)[2]) const {
        const uint32_t *p =
            reinterpret_cast<const uint32_t *>(sm + slot + kRows + h * (kU * 32)) + lane;
        w[0] = p[0];
        w[1] = p[32];
    }
    // the slot is taken: gives it to the copy D slots on
    __device__ __forceinline__ void pass() {
        __syncwarp();
        issue(slot);
        slot = slot + kSlot < kBytes ? slot + kSlot : 0;
    }
    // before the slots are used for anything else
    __device__ __forceinline__ void finish() const {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
    }
};

// Where a lane keeps its vector-segment's codes during the adjustment, in
// batches of kU = 8 coordinates that start at a multiple of 8.  load and store
// move the words of Fields<kBits> of the batch at j0, which has n codes (fields
// past n read 0).
// GlobalCodes: eight bits per code in the byte scratch, a batch as two words
// per lane (the 32 lanes' words of one index are consecutive); the last, partial
// batch of a segment as one byte per code, in the rows' layout, so that a
// segment takes one byte per coordinate and row.
struct GlobalCodes {
    uint8_t *base;  // of the warp's segment
    int lane;
    static constexpr int kBits = 8, kMinB = 1, kMaxB = 8;
    static constexpr bool kWriteChanged = true;  // store a batch only if a code moved
    static constexpr bool kRingCodes = true;
    // slots in flight: a warp often has a scheduler to itself here
    static constexpr int kDepth = 4;
    using R = Ring<kDepth, true>;
    __device__ __forceinline__ void load(int j0, uint32_t (&w)[2], int n) const {
        uint8_t *p = base + ((int64_t)j0 << 5);
        if (n >= kU) {
            w[0] = reinterpret_cast<uint32_t *>(p)[lane];
            w[1] = reinterpret_cast<uint32_t *>(p)[32 + lane];
        } else {
            w[0] = w[1] = 0u;
#pragma unroll
            for (int k = 0; k < kU; ++k)
                if (k < n) w[k >> 2] |= (uint32_t)p[(k << 5) + lane] << (8 * (k & 3));
        }
    }
    __device__ __forceinline__ void store(int j0, const uint32_t (&w)[2], int n) const {
        uint8_t *p = base + ((int64_t)j0 << 5);
        if (n >= kU) {
            reinterpret_cast<uint32_t *>(p)[lane] = w[0];
            reinterpret_cast<uint32_t *>(p)[32 + lane] = w[1];
        } else {
#pragma unroll
            for (int k = 0; k < kU; ++k)
                if (k < n) p[(k << 5) + lane] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
        }
    }
};
// SmemCodes<BITS>: packed in shared memory, BITS bits per code: 1 (B = 1),
// 2 (B = 2), 4 (B = 3, 4) or 8 (B = 5 .. 8).  A batch of 8 codes takes BITS
// bytes of the lane's byte stream, whose byte b is byte b % 4 of the lane's
// word b / 4, and word w of the lane sits at cw[w * 32] (the 32 lanes' words
// of one index are consecutive: no bank conflict).  A batch is stored back
// after its steps as a byte, a half-word or one or two words, so that no other
// batch's codes are rewritten.
template <int BITS> struct SmemCodes {
    uint32_t *cw;
    static constexpr int kBits = BITS;
    static constexpr int kMinB = BITS == 1 ? 1 : BITS == 2 ? 2 : BITS == 4 ? 3 : 5, kMaxB = BITS;
    static constexpr bool kWriteChanged = false;
    static constexpr bool kRingCodes = false;
    static constexpr int kDepth = 2;
    using R = Ring<kDepth, false>;
    static constexpr int kWords = Fields<BITS>::kWords;
    // the batch of coordinates j0 .. j0 + 7: its first word (BITS >= 4) or
    // its byte (BITS < 4)
    __device__ __forceinline__ uint32_t *word_of(int j0) const {
        return cw + (((j0 >> 3) * kWords) << 5);
    }
    __device__ __forceinline__ uint8_t *byte_of(int j0) const {
        const int bo = (j0 >> 3) * BITS;
        return reinterpret_cast<uint8_t *>(cw + ((bo >> 2) << 5)) + (bo & 3);
    }
    __device__ __forceinline__ void load(int j0, uint32_t (&w)[kWords], int) const {
        if constexpr (BITS >= 4) {
#pragma unroll
            for (int i = 0; i < kWords; ++i) w[i] = word_of(j0)[i << 5];
        } else if constexpr (BITS == 2) {
            w[0] = *reinterpret_cast<const uint16_t *>(byte_of(j0));
        } else {
            w[0] = *byte_of(j0);
        }
    }
    __device__ __forceinline__ void store(int j0, const uint32_t (&w)[kWords], int) const {
        if constexpr (BITS >= 4) {
#pragma unroll
            for (int i = 0; i < kWords; ++i) word_of(j0)[i << 5] = w[i];
        } else if constexpr (BITS == 2) {
            *reinterpret_cast<uint16_t *>(byte_of(j0)) = (uint16_t)w[0];
        } else {
            *byte_of(j0) = (uint8_t)w[0];
        }
    }
};

// The bit-planes of one lane's segment (most significant first, 64-bit words)
// and |u|^2 of its codes, exactly, from its batches in order.  Planes are
// gathered and stored by 64 bits, or by 32 from five bits up, where twice as
// many registers would spill.
template <int B, int BITS> struct Planes {
    using F = Fields<BITS>;
    static constexpr bool kWide = B <= 4;
    static constexpr int kCols = kWide ? 64 : 32;  // coordinates of a store
    uint32_t lo[kWide ? B : 1] = {}, hi[B] = {};
    uint32_t c2 = 0, c1 = 0;  // sums of c^2 and c (BITS >= 4), of (c in {0, cmax}) (B = 2)
    // the n codes of the batch at j0 (fields past n are 0)
    __device__ __forceinline__ void add(const uint32_t (&w)[F::kWords], int j0, int n, int len,
                                        bool valid, uint64_t *cout, int words) {
        uint32_t t[F::kWords];
        F::planes(w, t);
        // a batch's byte enters at the top of the plane's word, which moves down
#pragma unroll
        for (int p = 0; p < B; ++p) {
            const int b = B - 1 - p;
            if (kWide) lo[kWide ? p : 0] = __byte_perm(lo[kWide ? p : 0], hi[p], 0x4321u);
            hi[p] = __byte_perm(hi[p], t[b >> 2], 0x0321u | (uint32_t)(4 + (b & 3)) << 12);
        }
        if constexpr (BITS >= 4) {
            uint32_t y[F::kY];
            F::expand(w, y);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                c2 = __dp4a(y[i], y[i], c2);
                c1 = __dp4a(y[i], 0x01010101u, c1);
            }
        } else if constexpr (BITS == 2) {
            c2 += (uint32_t)__popc(~(t[0] ^ (t[0] >> 8)) & ((1u << n) - 1u));
        }
        const bool last = j0 + n >= len;
        if (((j0 + kU) & (kCols - 1)) == 0 || last) {
            const int gap = kCols - kU - (j0 & (kCols - 1));  // bits the last word does not reach
            if (valid) {
                if (kWide) {
#pragma unroll
                    for (int p = 0; p < B; ++p)
                        cout[p * words + (j0 >> 6)] =
                            ((uint64_t)hi[p] << 32 | lo[kWide ? p : 0]) >> gap;
                } else {
                    uint32_t *c32 = reinterpret_cast<uint32_t *>(cout) + (j0 >> 5);
#pragma unroll
                    for (int p = 0; p < B; ++p) {
                        c32[2 * p * words] = hi[p] >> gap;
                        // a plane's last 64-bit word that ends in its first half
                        if (last && (j0 & 32) == 0) c32[2 * p * words + 1] = 0u;
                    }
                }
            }
        }
    }
    // sum of (2c - cmax)^2 over the segment
    __device__ __forceinline__ int u2(int len) const {
        constexpr uint32_t cmax = (1u << B) - 1u;
        if constexpr (BITS >= 4) return (int)(4u * c2 - 4u * cmax * c1 + (uint32_t)len * cmax * cmax);
        else if constexpr (BITS == 2) return len + 8 * (int)c2;
        else return len;
    }
};
template <int B, class CS>
__device__ __forceinline__ int pack_segment(const CS &cs, int len, bool valid,
                                            uint64_t *cout, int words) {
    using F = Fields<CS::kBits>;
    Planes<B, CS::kBits> P;
    for (int j0 = 0; j0 < len; j0 += kU) {
        uint32_t w[F::kWords];
        cs.load(j0, w, len - j0);
        P.add(w, j0, min(kU, len - j0), len, valid, cout, words);
    }
    return P.u2(len);
}

// The adjustment state of one lane's vector-segment.  A lane that is done
// (no move in its last round, or nothing to adjust) holds I2 = +inf, which
// no gain exceeds.
struct LaneState {
    float I, S, I2;
};

// One coordinate of Algorithm 1 for one lane, whose code has u = 2c - cmax: an
// accepted move updates the state and adds +-unit to moves.  s = sign(T) (+ for
// T = +0); s*u < cmax is the range check of c + s.  The update is predicated:
// of a warp's 32 lanes some lane moves in most steps, and a branch around the
// update cost its divergence (94 cycles a step in a warp alone on an SM) and
// more instructions than it skipped.
__device__ __forceinline__ void caq_step(LaneState &L, float x, float u, float cmaxf, float unit,
                                         float &moves) {
    const float xS = x * L.S;
    const float T = fmaf(-u, L.I, xS);
    float su, s2;  // s u and 2 s
    asm("lop3.b32 %0, %1, %2, 0x80000000, 0x78;" : "=f"(su) : "f"(u), "f"(T));  // u ^ (T & sign)
    asm("lop3.b32 %0, %1, %2, 0x80000000, 0xD8;" : "=f"(s2) : "f"(2.f), "f"(T));  // 2, T's sign
    const float gain = fmaf(fabsf(T), L.I, x * xS);
    asm("{\n"
        ".reg .pred p;\n"
        "setp.lt.f32 p, %4, %5;\n"
        "setp.gt.and.f32 p, %6, %2, p;\n"
        "@p fma.rn.f32 %0, %7, %8, %0;\n"
        "@p fma.rn.f32 %1, %4, 0f40800000, %10;\n"
        "@p mul.rn.f32 %2, %0, %0;\n"
        "@p fma.rn.f32 %3, %7, %9, %3;\n"
        "}\n"
        : "+f"(L.I), "+f"(L.S), "+f"(L.I2), "+f"(moves)
        : "f"(su), "f"(cmaxf), "f"(gain), "f"(s2), "f"(x), "f"(0.5f * unit),
          "f"(__fadd_rn(L.S, 4.f)));
}

// The steps of one batch (whole: all kU coordinates, else the first n): w
// becomes the batch's codes after them; nonzero if a code moved.
template <int BITS, bool WHOLE>
__device__ __forceinline__ uint32_t batch_steps(LaneState &L, const float (&x)[kU],
                                                uint32_t (&w)[Fields<BITS>::kWords], int n,
                                                float cmaxf, float ucst) {
    using F = Fields<BITS>;
    float u[kU], mv[F::kMoves];
    F::u_of(w, ucst, u);
#pragma unroll
    for (int i = 0; i < F::kMoves; ++i) mv[i] = 12582912.f;
#pragma unroll
    for (int k = 0; k < kU; ++k)
        if (WHOLE || k < n)
            caq_step(L, x[k], u[k], cmaxf, (float)(1 << F::move_bit(k)), mv[F::move_word(k)]);
    uint32_t any = 0u, old[F::kWords];
#pragma unroll
    for (int i = 0; i < F::kWords; ++i) old[i] = w[i];
    F::apply(mv, w);
#pragma unroll
    for (int i = 0; i < F::kWords; ++i) any |= w[i] ^ old[i];
    return any;
}

// The codes of the batch at j0 (n codes), from the ring where it brings them:
// a batch's codes are copied after they were stored if the segment has more
// slots than the ring.
template <class CS>
__device__ __forceinline__ void load_codes(const CS &cs, const typename CS::R &ring, int j0, int n,
                                           int len, uint32_t (&w)[Fields<CS::kBits>::kWords]) {
    if constexpr (CS::kRingCodes) {
        if (n >= kU && len > kSlotCols * CS::kDepth) {
            ring.take_codes((j0 / kU) & 1, w);
            return;
        }
    }
    cs.load(j0, w, n);
}

// One round of Algorithm 1 over the lane's segment, a slot of the ring at a time:
// both batches are read before the first one's steps, so that the second's reads
// and the next copy run beside them (a batch at a time: 4.28 ms per 1,000,000
// rows at d = 960, 850 us for the 3,072-long segment of 20,011 rows; so: 4.03 and
// 729).  With PACK_B = B > 0 the
// round is the last one: a coordinate's code is final once its own step is
// done, so the bit-planes (most significant first, 64-bit words) and the exact
// |u|^2, which the function returns, are built as the round goes.
template <int PACK_B, class CS>
__device__ __forceinline__ int run_round(LaneState &L, typename CS::R &ring, const CS &cs, int len,
                                         int cmax, bool &moved, bool valid, uint64_t *cout,
                                         int words) {
    using F = Fields<CS::kBits>;
    const float cmaxf = (float)cmax, ucst = -(65536.f + cmaxf);
    const int lenU = len & ~(kSlotCols - 1);  // coordinates in whole slots
    Planes<PACK_B ? PACK_B : 1, CS::kBits> P;
    uint32_t any = 0u;
    for (int j0 = 0; j0 < lenU; j0 += kSlotCols) {
        float x[2][kU];
        uint32_t w[2][F::kWords];
        ring.wait();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            ring.take(h, x[h]);
            load_codes(cs, ring, j0 + h * kU, kU, len, w[h]);
        }
        ring.pass();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + h * kU;
            const uint32_t ch = batch_steps<CS::kBits, true>(L, x[h], w[h], kU, cmaxf, ucst);
            any |= ch;
            if (PACK_B > 0) P.add(w[h], j, kU, len, valid, cout, words);
            else if (!CS::kWriteChanged || ch) cs.store(j, w[h], kU);
        }
    }
    if (lenU < len) {  // the last, partial slot
        ring.wait();
#pragma unroll 1
        for (int j = lenU; j < len; j += kU) {
            const int n = min(kU, len - j);
            float x[kU];
            uint32_t w[F::kWords];
            ring.take((j / kU) & 1, x);
            load_codes(cs, ring, j, n, len, w);
            any |= batch_steps<CS::kBits, false>(L, x, w, n, cmaxf, ucst);
            if (PACK_B > 0) P.add(w, j, n, len, valid, cout, words);
            else cs.store(j, w, n);
        }
        ring.pass();
    }
    moved = any != 0u;
    return PACK_B > 0 ? P.u2(len) : 0;
}

// The last round (which packs as it goes) and the separate packing pass for
// B bits, instantiated only for the bit widths the code store holds.
template <int B, class CS>
__device__ __forceinline__ int last_round(LaneState &L, typename CS::R &ring, const CS &cs, int len,
                                          int cmax, bool &moved, bool valid, uint64_t *cout,
                                          int words) {
    if constexpr (B >= CS::kMinB && B <= CS::kMaxB)
        return run_round<B, CS>(L, ring, cs, len, cmax, moved, valid, cout, words);
    else
        return 0;
}
template <int B, class CS>
__device__ __forceinline__ int pack_only(const CS &cs, int len, bool valid, uint64_t *cout,
                                         int words) {
    if constexpr (B >= CS::kMinB && B <= CS::kMaxB)
        return pack_segment<B, CS>(cs, len, valid, cout, words);
    else
        return 0;
}

// Algorithm 1 on one lane's vector-segment with its codes in store cs:
// initial codes, the rounds, the packing and the two factors.
template <class CS>
__device__ __forceinline__ void caq_segment(const CS &cs, typename CS::R ring, int len, int B,
                                            int words, bool valid, float vmax, int rounds,
                                            uint64_t *cout, float *fo) {
    using F = Fields<CS::kBits>;
    const int cmax = (1 << B) - 1;
    const bool live = valid && vmax > 0.f;
    // initial codes, Eq. find_nearest_code: c = floor((o + v_max) / Delta),
    // Delta = 2 v_max / 2^B; with I = <u, o>, S = |u|^2 and |o|^2 (in FP32:
    // clamped first, then floor as the sum with 2^23 rounded toward zero, whose
    // low bits are the code; |u|^2 is summed in FP32 for the decisions and
    // recounted exactly while packing).  A vector-segment whose v_max is 0 gets
    // codes 0 (its Delta is taken as infinite).  Every lane of the last group of
    // 32 rows reads rows the buffer holds.
    const float inv_delta = live ? (float)(1 << (B - 1)) / vmax : 0.f;
    const float off_c = vmax * inv_delta;  // (o + v_max) / Delta = o / Delta + off_c
    const float cmaxf = (float)cmax;
    float I = 0.f, n2 = 0.f, S = 0.f;
    auto codes_of = [&](float x0, float x1, float &t0, float &t1, float &c0, float &c1) {
        fma2(x0, x1, inv_delta, off_c, t0, t1);
        add2_rz(fminf(fmaxf(t0, 0.f), cmaxf), fminf(fmaxf(t1, 0.f), cmaxf), 8388608.f, t0, t1);
        add2(t0, t1, -8388608.f, c0, c1);
    };
    auto sums = [&](float x, float u) {
        I = fmaf(u, x, I);
        n2 = fmaf(x, x, n2);
        S = fmaf(u, u, S);
    };
    auto init = [&](const float *x, float *t, float *cf) {  // two coordinates
        float u0, u1;
        codes_of(x[0], x[1], t[0], t[1], cf[0], cf[1]);
        fma2(cf[0], cf[1], 2.f, -cmaxf, u0, u1);
        sums(x[0], u0);
        sums(x[1], u1);
    };
    ring.start();
    const int lenU = len & ~(kSlotCols - 1);  // coordinates in whole slots
    for (int j0 = 0; j0 < lenU; j0 += kSlotCols) {
        float x[2][kU];
        ring.wait();
        ring.take(0, x[0]);
        ring.take(1, x[1]);
        ring.pass();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float t[kU], cf[kU];
#pragma unroll
            for (int k = 0; k < kU; k += 2) init(&x[h][k], &t[k], &cf[k]);
            uint32_t w[F::kWords];
            F::pack(t, cf, w);
            cs.store(j0 + h * kU, w, kU);
        }
    }
    if (lenU < len) {
        ring.wait();
#pragma unroll 1
        for (int j = lenU; j < len; j += kU) {
            float x[kU], t[kU], cf[kU];
            ring.take((j / kU) & 1, x);
#pragma unroll
            for (int k = 0; k < kU; ++k) {
                codes_of(x[k], x[k], t[k], t[k], cf[k], cf[k]);
                if (j + k < len) {
                    sums(x[k], fmaf(2.f, cf[k], -cmaxf));
                } else {
                    t[k] = 8388608.f;
                    cf[k] = 0.f;
                }
            }
            uint32_t w[F::kWords];
            F::pack(t, cf, w);
            cs.store(j, w, min(kU, len - j));
        }
        ring.pass();
    }
    LaneState L{I, S, live ? I * I : __int_as_float(0x7f800000)};
    int Si = -1;  // |u|^2 of the final codes, exactly, once they are packed
    for (int r = 0; r < rounds; ++r) {
        if (!__any_sync(0xffffffffu, L.I2 != __int_as_float(0x7f800000))) break;
        bool moved = false;
        if (r == rounds - 1) {  // the last round packs as it goes
            switch (B) {  // uniform per warp
                case 1: Si = last_round<1, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 2: Si = last_round<2, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 3: Si = last_round<3, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 4: Si = last_round<4, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 5: Si = last_round<5, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 6: Si = last_round<6, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                case 7: Si = last_round<7, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
                default: Si = last_round<8, CS>(L, ring, cs, len, cmax, moved, valid, cout, words); break;
            }
            break;
        }
        run_round<0, CS>(L, ring, cs, len, cmax, moved, valid, cout, words);
        if (!moved) L.I2 = __int_as_float(0x7f800000);
    }
    ring.finish();
    I = L.I;
    // every lane done before the last round (or no rounds): pack from the codes
    if (Si < 0) {
        switch (B) {  // uniform per warp
            case 1: Si = pack_only<1, CS>(cs, len, valid, cout, words); break;
            case 2: Si = pack_only<2, CS>(cs, len, valid, cout, words); break;
            case 3: Si = pack_only<3, CS>(cs, len, valid, cout, words); break;
            case 4: Si = pack_only<4, CS>(cs, len, valid, cout, words); break;
            case 5: Si = pack_only<5, CS>(cs, len, valid, cout, words); break;
            case 6: Si = pack_only<6, CS>(cs, len, valid, cout, words); break;
            case 7: Si = pack_only<7, CS>(cs, len, valid, cout, words); break;
            default: Si = pack_only<8, CS>(cs, len, valid, cout, words); break;
        }
    }
    if (valid) {
        if (live) {
            const float nrm = sqrtf(n2);
            fo[0] = nrm;
            fo[1] = I / (sqrtf((float)Si) * nrm);
        } else {
            // all-zero segment (the paper is silent): codes 0, |o| = 0, cos = 1
            fo[0] = 0.f;
            fo[1] = 1.f;
        }
    }
}

// The work of warp w of one model's launch: one warp per (kept segment,
// group of 32 rows).  SMEM_CODES: the codes live in the warp's region of
// the block's shared memory (words_per_lane 32-bit words per lane), else in
// the byte scratch cs.
template <bool SMEM_CODES>
__device__ __forceinline__ void caq1_warp(int64_t w, const float *__restrict__ Oi, int64_t n,
                                          int dk, int nseg, const SegTable &t, int rounds,
                                          uint8_t *__restrict__ cs,
                                          const float *__restrict__ vmax_arr,
                                          uint8_t *__restrict__ codes, int64_t code_stride,
                                          float *__restrict__ factors, int nf,
                                          uint8_t *smem, int words_per_lane) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t groups = (n + 31) / 32;
    const int si = t.order[w / groups];
    const Seg sg = t.s[si];
    const int64_t g = w % groups;
    const int off = sg.off, len = sg.len, B = sg.bits, words = sg.words, fidx = sg.fidx;
    const long long code_off = sg.code_off;
    const int64_t v = g * 32 + lane;
    const bool valid = v < n;
    const float *rows = Oi + ((g * dk + off) << 5);
    // v_max of the lane's vector-segment, recorded by the projection
    const float vmax = valid ? __ldg(vmax_arr + ((g * nseg + si) << 5) + lane) : 0.f;
    uint64_t *cout = reinterpret_cast<uint64_t *>(codes + v * code_stride + code_off);
    float *fo = factors + v * nf + fidx;
    // the block's shared memory: a ring per warp, then the warps' codes
    if constexpr (SMEM_CODES) {
        using R = SmemCodes<8>::R;
        const R ring{smem + warp * R::kBytes, rows, nullptr, len, lane, 0, 0};
        uint32_t *cw = reinterpret_cast<uint32_t *>(smem + (blockDim.x >> 5) * R::kBytes) +
                       warp * (words_per_lane << 5) + lane;
        if (B == 1)  // uniform per warp
            caq_segment(SmemCodes<1>{cw}, ring, len, B, words, valid, vmax, rounds, cout, fo);
        else if (B == 2)
            caq_segment(SmemCodes<2>{cw}, ring, len, B, words, valid, vmax, rounds, cout, fo);
        else if (B <= 4)
            caq_segment(SmemCodes<4>{cw}, ring, len, B, words, valid, vmax, rounds, cout, fo);
        else
            caq_segment(SmemCodes<8>{cw}, ring, len, B, words, valid, vmax, rounds, cout, fo);
    } else {
        using R = GlobalCodes::R;
        uint8_t *cb = cs + ((g * dk + off) << 5);
        const R ring{smem + warp * R::kBytes, rows, cb, len, lane, 0, 0};
        caq_segment(GlobalCodes{cb, lane}, ring, len, B, words, valid, vmax, rounds, cout, fo);
    }
}

// All kept segments of a chunk in one launch.  Blocks of four warps, five of
// them per SM at the d = 960 plan (44 KB each; 80 registers a thread, nothing
// spilled): 4.28 ms per 1,000,000 rows, with blocks of eight (two per SM) 4.54,
// of two 4.36, when the rows were taken a batch at a time (now 4.03).
__global__ void __launch_bounds__(kWarps * 32, 5)
k_caq1(const float *__restrict__ Oi, int64_t n, int dk, int nseg, const SegTable t, int rounds,
       uint8_t *__restrict__ cs, const float *__restrict__ vmax_arr,
       uint8_t *__restrict__ codes, int64_t code_stride, float *__restrict__ factors, int nf) {
    extern __shared__ __align__(16) uint8_t smem_caq[];
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (n + 31) / 32 * nseg) return;  // uniform per warp
    caq1_warp<false>(w, Oi, n, dk, nseg, t, rounds, cs, vmax_arr, codes, code_stride, factors, nf,
                     smem_caq, 0);
}

// The same with every warp's codes in shared memory (words_per_lane 32-bit
// words per lane).
__global__ void __launch_bounds__(kWarps * 32, 5)
k_caq1_sm(const float *__restrict__ Oi, int64_t n, int dk, int nseg, const SegTable t, int rounds,
          const float *__restrict__ vmax_arr, uint8_t *__restrict__ codes, int64_t code_stride,
          float *__restrict__ factors, int nf, int words_per_lane) {
    extern __shared__ __align__(16) uint8_t smem_caq[];
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (n + 31) / 32 * nseg) return;  // uniform per warp
    caq1_warp<true>(w, Oi, n, dk, nseg, t, rounds, nullptr, vmax_arr, codes, code_stride, factors,
                    nf, smem_caq, words_per_lane);
}

// The rows of up to kMaxGroups models (a batch of several collections) in
// one launch: global warp w belongs to the group g with warp_start[g] <= w <
// warp_start[g + 1].
// A persistent warp of a grouped launch: it takes work items (global warp
// indices of the batch) from the device counter `queue` until none is left.
template <bool SMEM_CODES>
__device__ __forceinline__ void caq1_grouped_warp(const CaqBatch<kMaxGroups> &batch, int *queue,
                                                  uint8_t *smem, int words_per_lane) {
    const int64_t total = batch.warp_start[batch.ngroups];
    for (;;) {
        int wi = 0;
        if ((threadIdx.x & 31) == 0) wi = atomicAdd(queue, 1);
        const int64_t wg = __shfl_sync(0xffffffffu, wi, 0);
        if (wg >= total) break;  // uniform per warp
        int gi = 0;
        while (gi + 1 < batch.ngroups && wg >= batch.warp_start[gi + 1]) ++gi;
        const CaqGroup &P = batch.g[gi];
        caq1_warp<SMEM_CODES>(wg - batch.warp_start[gi], P.Oi, P.n, P.dk, P.nseg, P.t, P.rounds,
                              P.cs, P.vmax, P.codes, P.code_stride, P.factors, P.nf, smem,
                              words_per_lane);
    }
}
__global__ void __launch_bounds__(kWarps * 32, 5)
k_caq1_grouped(const __grid_constant__ CaqBatch<kMaxGroups> batch, int *queue) {
    extern __shared__ __align__(16) uint8_t smem_caq[];
    caq1_grouped_warp<false>(batch, queue, smem_caq, 0);
}
// The same with the codes in shared memory (words_per_lane: the largest
// over the groups' segments).
__global__ void __launch_bounds__(kWarps * 32, 5)
k_caq1_grouped_sm(const __grid_constant__ CaqBatch<kMaxGroups> batch, int *queue,
                  int words_per_lane) {
    extern __shared__ __align__(16) uint8_t smem_caq[];
    caq1_grouped_warp<true>(batch, queue, smem_caq, words_per_lane);
}

// The instruction ceiling of the adjustment: caq_step on coordinates held in
// registers (no loads or stores), kU per lane, a sign flip per step keeping
// moves happening; one block of 128 threads per 4 warps of occupancy.
__global__ void __launch_bounds__(128) k_step_ceiling(int iters, int cmax, float *out) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    float x[kU];
    uint32_t w[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < kU; ++k) {
        x[k] = (float)((tid * 7 + k * 13) % 31) * 0.03f - 0.45f;
        w[k >> 2] |= (uint32_t)((tid + k) % (cmax + 1)) << (8 * (k & 3));
    }
    LaneState L{10.f, 200.f, 100.f};
    const float cmaxf = (float)cmax, ucst = -(65536.f + cmaxf);
    uint32_t moves = 0u;
#pragma unroll 1
    for (int it = 0; it < iters; ++it) {
        moves |= batch_steps<8, true>(L, x, w, kU, cmaxf, ucst);
#pragma unroll
        for (int k = 0; k < kU; ++k) x[k] = -x[k];
    }
    out[tid] = L.I + L.S + (float)(moves & 1u) + (float)w[0];
}

// v_max of every (row, kept segment) of interleaved rows: one warp per (group
// of 32 rows, kept segment), lane = row.
__global__ void __launch_bounds__(256)
k_seg_vmax(const float *__restrict__ Oi, int64_t n, int dk, const SegCols sc,
           float *__restrict__ vmax) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t groups = (n + 31) / 32;
    if (w >= groups * sc.nk) return;
    const int64_t g = w / sc.nk;
    const int s = (int)(w % sc.nk);
    const int c0 = s == 0 ? 0 : sc.end[s - 1], c1 = sc.end[s];
    const bool valid = g * 32 + lane < n;
    float mx = 0.f;
    for (int c = c0; c < c1; ++c)
        mx = fmaxf(mx, valid ? fabsf(__ldg(Oi + ((g * dk + c) << 5) + lane)) : 0.f);
    vmax[((g * sc.nk + s) << 5) + lane] = mx;
}

// Row-major O (n x dk, ldo) -> interleaved O_i (groups of 32 rows).
__global__ void k_interleave(const float *__restrict__ O, int64_t ldo, int64_t n, int dk,
                             float *__restrict__ Oi) {
    __shared__ float tile[32][33];
    const int64_t g = blockIdx.y;
    const int c0 = blockIdx.x * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    for (int rr = ty; rr < 32; rr += 8) {
        const int64_t row = g * 32 + rr;
        const int col = c0 + tx;
        tile[rr][tx] = (row < n && col < dk) ? O[row * ldo + col] : 0.f;
    }
    __syncthreads();
    for (int cc = ty; cc < 32; cc += 8) {
        const int col = c0 + cc;
        if (col < dk) Oi[((g * dk + col) << 5) + tx] = tile[tx][cc];
    }
}

}  // namespace

saq_status make_group(const CaqJob &j, CaqGroup *g) {
    const saq_model *m = j.m;
    const int nk = (int)m->kept.size();
    if (nk > kMaxSeg) return set_error(SAQ_ERR_UNSUPPORTED, "more than %d kept segments", kMaxSeg);
    SegTable &t = g->t;
    for (int i = 0; i < nk; ++i) {
        const KeptSeg &k = m->kept[(size_t)i];
        if (k.bits < 1 || k.bits > 8)
            return set_error(SAQ_ERR_INVALID, "segment bits %d outside 1..8", k.bits);
        t.s[i] = Seg{k.off, k.len, k.bits, k.words, k.fidx, (long long)k.code_off};
        t.order[i] = i;
    }
    std::stable_sort(t.order, t.order + nk, [&](int a, int b) { return t.s[a].len > t.s[b].len; });
    g->Oi = j.Oi;
    g->n = j.n;
    g->dk = m->dk;
    g->nseg = nk;
    g->rounds = m->rounds;
    g->nf = m->nf;
    g->cs = j.cs;
    g->vmax = j.vmax;
    g->codes = j.codes;
    g->code_stride = (int64_t)m->code_bytes;
    g->factors = j.factors;
    return SAQ_OK;
}

namespace {

// 32-bit words per lane of the shared-memory code store for model m: its
// largest segment's, at 1, 2, 4 or 8 bits per code (B = 1, 2, 3-4, 5-8),
// a batch of 8 codes in that many bytes.
int words_per_lane(const saq_model *m) {
    int wpl = 0;
    for (const KeptSeg &k : m->kept) {
        const int width = k.bits <= 1 ? 1 : k.bits == 2 ? 2 : k.bits <= 4 ? 4 : 8;
        wpl = std::max(wpl, ((k.len + 7) / 8 * width + 3) / 4);
    }
    return wpl;
}

// The codes go to shared memory when eight warps' take at most kCaqSmemMax.
bool codes_in_smem(int wpl) { return (size_t)wpl * 32 * 4 * 8 <= kCaqSmemMax; }

// Shared memory of a block of `warps` warps: the rings and, with wpl words per
// lane, the codes.
size_t caq_smem_bytes(int wpl, int warps) {
    return codes_in_smem(wpl) ? (size_t)warps * (SmemCodes<8>::R::kBytes + (size_t)wpl * 32 * 4)
                              : (size_t)warps * GlobalCodes::R::kBytes;
}
constexpr size_t kCaqSmemLimit =
    std::max(kCaqSmemMax * kWarps / 8 + kWarps * SmemCodes<8>::R::kBytes,
             (size_t)kWarps * GlobalCodes::R::kBytes);

// Sets the kernel's shared-memory attributes once per device (`done`: one
// bit per device ordinal, devices 0..63; a larger ordinal sets them at
// every launch).
template <class K> saq_status prepare_smem_kernel(K *kernel, std::atomic<uint64_t> &done) {
    int dev = 0;
    SAQ_CUDA_CHECK(cudaGetDevice(&dev));
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return SAQ_OK;
    SAQ_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kCaqSmemLimit));
    // all of the unified L1 / shared storage as shared memory
    SAQ_CUDA_CHECK(cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                        100));
    done.fetch_or(bit, std::memory_order_release);
    return SAQ_OK;
}
std::atomic<uint64_t> g_caq1_ready{0}, g_caq1_sm_ready{0}, g_caq1_grouped_ready{0},
    g_caq1_grouped_sm_ready{0};

}  // namespace

saq_status launch_caq1(const saq_model *m, const float *Oi, int64_t n, uint8_t *cs,
                       const float *vmax, uint8_t *codes, float *factors, cudaStream_t s) {
    if (n <= 0 || m->kept.empty()) return SAQ_OK;
    const CaqJob job{m, Oi, n, cs, vmax, codes, factors};
    bool ran = false;
    saq_status scan = launch_caq_scan(&job, 1, s, &ran);
    if (scan != SAQ_OK || ran) return scan;
    CaqGroup g;
    saq_status st = make_group(job, &g);
    if (st != SAQ_OK) return st;
    const int64_t warps = (n + 31) / 32 * g.nseg;
    // codes in shared memory when they fit, else in the global byte scratch
    const int wpl = words_per_lane(m);
    const bool sm_codes = codes_in_smem(wpl);
    int dev = 0, sms = 0;
    SAQ_CUDA_CHECK(cudaGetDevice(&dev));
    SAQ_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // few warps are spread over the SMs by blocks of two
    const int wpb = warps < (int64_t)kSpreadWarps * sms ? 2 : kWarps;
    const int64_t blocks = (warps + wpb - 1) / wpb;
    const size_t smem = caq_smem_bytes(wpl, wpb);
    st = sm_codes ? prepare_smem_kernel(k_caq1_sm, g_caq1_sm_ready)
                  : prepare_smem_kernel(k_caq1, g_caq1_ready);
    if (st != SAQ_OK) return st;
    {
        LaunchTimer lt_(kKindQuantize, s);
        if (sm_codes) {
            k_caq1_sm<<<(unsigned)blocks, 32 * wpb, smem, s>>>(Oi, n, g.dk, g.nseg, g.t, g.rounds, vmax,
                                                          codes, g.code_stride, factors, g.nf, wpl);
        } else {
            k_caq1<<<(unsigned)blocks, 32 * wpb, smem, s>>>(Oi, n, g.dk, g.nseg, g.t, g.rounds, cs, vmax,
                                                    codes, g.code_stride, factors, g.nf);
        }
    }
    note_launches();
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

saq_status launch_caq1_grouped(const CaqJob *jobs, int njobs, int *queue, cudaStream_t s) {
    if (njobs < 1 || njobs > kMaxGroups)
        return set_error(SAQ_ERR_INVALID, "1..%d models per grouped launch", kMaxGroups);
    bool ran = false;
    saq_status scan = launch_caq_scan(jobs, njobs, s, &ran);
    if (scan != SAQ_OK || ran) return scan;
    CaqBatch<kMaxGroups> b;
    b.ngroups = 0;
    b.warp_start[0] = 0;
    int wpl = 0;
    for (int i = 0; i < njobs; ++i) {
        if (jobs[i].n <= 0 || jobs[i].m->kept.empty()) continue;
        wpl = std::max(wpl, words_per_lane(jobs[i].m));
        saq_status st = make_group(jobs[i], &b.g[b.ngroups]);
        if (st != SAQ_OK) return st;
        b.warp_start[b.ngroups + 1] =
            b.warp_start[b.ngroups] + (jobs[i].n + 31) / 32 * (int64_t)b.g[b.ngroups].nseg;
        ++b.ngroups;
    }
    if (b.ngroups == 0) return SAQ_OK;
    if (b.warp_start[b.ngroups] > 0x7FFFFFFF)
        return set_error(SAQ_ERR_UNSUPPORTED, "too many rows in one call");
    const int64_t blocks = (b.warp_start[b.ngroups] + kWarps - 1) / kWarps;
    const size_t smem = caq_smem_bytes(wpl, kWarps);
    const bool sm_codes = codes_in_smem(wpl);
    saq_status st = sm_codes ? prepare_smem_kernel(k_caq1_grouped_sm, g_caq1_grouped_sm_ready)
                             : prepare_smem_kernel(k_caq1_grouped, g_caq1_grouped_ready);
    if (st != SAQ_OK) return st;
    // persistent: as many blocks as stay resident at once (at most the work)
    int dev = 0, sms = 0, per_sm = 0;
    SAQ_CUDA_CHECK(cudaGetDevice(&dev));
    SAQ_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (sm_codes)
        SAQ_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_caq1_grouped_sm,
                                                                     kWarps * 32, smem));
    else
        SAQ_CUDA_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_caq1_grouped,
                                                                     kWarps * 32, smem));
    const int64_t grid = std::min<int64_t>(blocks, (int64_t)std::max(1, sms * per_sm));
    {
        LaunchTimer lt_(kKindQuantize, s);
        if (sm_codes)
            k_caq1_grouped_sm<<<(unsigned)grid, kWarps * 32, smem, s>>>(b, queue, wpl);
        else
            k_caq1_grouped<<<(unsigned)grid, kWarps * 32, smem, s>>>(b, queue);
    }
    note_launches();
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

saq_status step_ceiling(int warps_per_sm, int bits, double *lane_steps_per_s) {
    int dev = 0, sms = 0;
    SAQ_CUDA_CHECK(cudaGetDevice(&dev));
    SAQ_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int blocks = sms * (warps_per_sm / 4);
    const int iters = 2000;
    float *out = nullptr;
    SAQ_CUDA_CHECK(scratch_alloc((void **)&out, sizeof(float) * (size_t)blocks * 128, 0));
    cudaEvent_t a = nullptr, b = nullptr;
    saq_status st = SAQ_OK;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
        st = set_error(SAQ_ERR_CUDA, "event creation failed");
    } else {
        const int cmax = (1 << bits) - 1;
        k_step_ceiling<<<blocks, 128>>>(iters / 4, cmax, out);  // warm-up
        cudaEventRecord(a, 0);
        k_step_ceiling<<<blocks, 128>>>(iters, cmax, out);
        cudaEventRecord(b, 0);
        note_launches(2);
        float ms = 0.f;
        if (cudaEventSynchronize(b) != cudaSuccess || cudaEventElapsedTime(&ms, a, b) != cudaSuccess ||
            cudaGetLastError() != cudaSuccess || ms <= 0.f)
            st = set_error(SAQ_ERR_CUDA, "step-ceiling measurement failed");
        else
            *lane_steps_per_s = (double)blocks * 128.0 * iters * kU / (ms * 1e-3);
    }
    if (a) cudaEventDestroy(a);
    if (b) cudaEventDestroy(b);
    cudaFreeAsync(out, 0);
    cudaStreamSynchronize(0);
    return st;
}

saq_status launch_seg_vmax(const saq_model *m, const float *Oi, int64_t n, float *vmax,
                           cudaStream_t s) {
    const SegCols sc = seg_cols(m);
    if (n <= 0 || sc.nk == 0) return SAQ_OK;
    const int64_t warps = (n + 31) / 32 * sc.nk;
    {
        LaunchTimer lt_(kKindOther, s);
        k_seg_vmax<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(Oi, n, m->dk, sc, vmax);
    }
    note_launches();
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

saq_status launch_interleave(const float *O, int64_t ldo, int64_t n, int dk, float *Oi,
                             cudaStream_t s) {
    if (n <= 0 || dk <= 0) return SAQ_OK;
    const int64_t groups = (n + 31) / 32;
    dim3 grid((unsigned)((dk + 31) / 32), (unsigned)groups);
    if (groups > 65535) {
        // split along groups to respect the grid's y limit
        for (int64_t g0 = 0; g0 < groups; g0 += 65535) {
            const int64_t gn = std::min<int64_t>(65535, groups - g0);
            dim3 gg((unsigned)((dk + 31) / 32), (unsigned)gn);
            {
                LaunchTimer lt_(kKindOther, s);
                k_interleave<<<gg, dim3(32, 8), 0, s>>>(O + g0 * 32 * ldo, ldo, n - g0 * 32, dk,
                                                        Oi + g0 * 32 * (int64_t)dk);
            }
            note_launches();
        }
    } else {
        {
            LaunchTimer lt_(kKindOther, s);
            k_interleave<<<grid, dim3(32, 8), 0, s>>>(O, ldo, n, dk, Oi);
        }
        note_launches();
    }
    SAQ_CUDA_CHECK(cudaGetLastError());
    return SAQ_OK;
}

}  // namespace saq
