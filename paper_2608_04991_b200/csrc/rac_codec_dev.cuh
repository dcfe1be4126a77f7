// Pieces shared by the RAC codec translation units (sm_100a): kernel parameters, the slab front end (loads,
// Eq. 6 statistics, wire coefficients), packing helpers, and the host-side launch helpers.
#pragma once

#include <math.h>
#include <stdlib.h>

#include <map>
#include <mutex>
#include <tuple>
#include <utility>

#include "rac_common.cuh"

namespace rac {

// ------------------------------------------------------------------------------------------------
// kernel parameters
// ------------------------------------------------------------------------------------------------
struct CodecParams {
    // tensors
    const uint16_t *X;         // encode / calibrate input, bf16[T,d]
    const uint16_t *ref_base;  // bf16[ref_rows,d] or null
    const int32_t *ref_row;    // int32[T] or null
    const uint16_t *gain;      // binary16[d] or null
    const uint16_t *bias;
    const float *step;         // [2,d]
    const float *inv_step;     // [2,d]
    uint8_t *payload;          // encode out / decode in
    uint16_t *X_hat;           // decode out
    float *calib_partial;      // calibrate out: [parts][2][d] sums of e^2, then [parts][2] token counts
    float *tmax;               // encode with outliers: [T][d/32] largest |e| per thread slab (caller workspace)
    uint32_t *status;
    long long T;
    long long ref_rows;
    // geometry
    int d, J, lpg, lpg_shift, topk, rec, code_bytes, stages;
    float inv_group;
    // a subset of the tokens (both null = all T tokens, in order), and a second reference buffer behind ref_base
    const int32_t *tok_list;     // int32[>= *tok_count] token indices in [0, T)
    const int32_t *tok_count;    // device int32[1]
    const uint16_t *intra_base;  // bf16[intra_rows, d]: reference rows ref_rows .. ref_rows + intra_rows - 1, or null
    long long intra_rows;
    // coefficient words shared by the tokens of a segment (Eq. 6 over several fitting positions), outside the record
    const uint32_t *coef_ext;    // u32[n_seg, J] or null (coefficients in the record)
    const int32_t *seg_of;       // int32[T] segment of each token
    float4 *moments;             // segment fit, first pass out: (mean r, mean h, Sxx, Sxy) per (token, group)
    // scale_mode 1 only: quantisation groups, per-group outliers, field offsets in the record
    int Jq, lpq, lpq_shift, kg, scale_off, codes_off, goff_off, gval_off;
    int qgen;   // lanes per quantisation group that is neither a power of two nor the token (lpq == 0 then), else 0
    // only from rac_selftest_bounded_wait: bytes announced on top of what the copies of a stage deliver, so that the
    // (bounded) wait for them cannot complete
    uint32_t test_extra_tx;
};

// parameters every call has in common, with the checks of the arguments they come from (defined in rac_codec.cu)
int fill_common(const Geometry &g, CodecParams *p, long long T, const void *ref_base, long long ref_rows,
                const int32_t *ref_row, const void *gain, const void *bias, uint32_t *status);
// scale_mode 1 (defined in rac_codec_dyn.cu)
int launch_encode_dyn(const Geometry &g, CodecParams &p, long long max_ctas, cudaStream_t stream);
int launch_decode_dyn(const Geometry &g, CodecParams &p, cudaStream_t stream);

constexpr int kMaxStages = 4;
constexpr int kRecBufs = 3;
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer (ties to even) in the low mantissa bits

// control block at the start of dynamic shared memory
struct Ctrl {
    unsigned long long bar[kMaxStages];
    int row[kMaxStages];        // reference row of the token in each stage, -1 = direct
    int seg[kMaxStages];        // segment of the token in each stage (shared coefficients only)
};

__host__ __device__ inline int align_up(int v, int a) { return (v + a - 1) / a * a; }

struct DecSmem {
    int ctrl, stage0, stage_bytes, rec_pad, out0, total;
};
__host__ __device__ inline DecSmem dec_smem_layout(int d, int rec, int stages) {
    DecSmem s;
    s.ctrl = 0;
    s.stage0 = align_up((int)sizeof(Ctrl), 128);
    s.rec_pad = align_up(rec, 128);
    s.stage_bytes = s.rec_pad + 2 * d;
    s.out0 = s.stage0 + stages * s.stage_bytes;
    s.total = s.out0 + kRecBufs * 2 * d;
    return s;
}

// ------------------------------------------------------------------------------------------------
// device helpers
// ------------------------------------------------------------------------------------------------
typedef unsigned long long u64;

__device__ __forceinline__ u64 pack2(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(u64 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 pfma(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 padd(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 psub(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 pmul(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// a 32-bit word of two bf16 -> packed (even channel, odd channel) binary32, exact
__device__ __forceinline__ u64 bf16x2_to_p(uint32_t w) {
    return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
// One binary32 operand and one bf16 half of a packed word, one rounding: the same value as unpacking the half first, without
// the unpacking.  (Per SM quarter a packed binary32 add or multiply-add takes 2 cycles for two values, and so does every
// shift, mask or permute that an unpacking is made of; an add takes 1 for one value.)
__device__ __forceinline__ float add_lo(uint32_t w, float c) {
    float r;
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; add.rn.f32.bf16 %0, l, %2;}" : "=f"(r) : "r"(w), "f"(c));
    return r;
}
__device__ __forceinline__ float add_hi(uint32_t w, float c) {
    float r;
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; add.rn.f32.bf16 %0, h, %2;}" : "=f"(r) : "r"(w), "f"(c));
    return r;
}
__device__ __forceinline__ float sub_lo(uint32_t w, float c) {   // low half - c
    float r;
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; sub.rn.f32.bf16 %0, l, %2;}" : "=f"(r) : "r"(w), "f"(c));
    return r;
}
__device__ __forceinline__ float sub_hi(uint32_t w, float c) {   // high half - c
    float r;
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; sub.rn.f32.bf16 %0, h, %2;}" : "=f"(r) : "r"(w), "f"(c));
    return r;
}
// packed halves of w minus a packed pair
__device__ __forceinline__ u64 sub_pair(uint32_t w, u64 c) {
    float c0, c1;
    unpack2(c, c0, c1);
    return pack2(sub_lo(w, c0), sub_hi(w, c1));
}
// bits of a where m is set, bits of b elsewhere
__device__ __forceinline__ uint32_t bitsel(uint32_t a, uint32_t b, uint32_t m) { return (a & m) | (b & ~m); }

// rotate the four entries right by rot (new[j] = old[(j - rot) & 3])
__device__ __forceinline__ void rot_right4(uint32_t (&w)[4], int rot) {
    if (rot & 1) { uint32_t t = w[3]; w[3] = w[2]; w[2] = w[1]; w[1] = w[0]; w[0] = t; }
    if (rot & 2) { uint32_t t = w[0]; w[0] = w[2]; w[2] = t; t = w[1]; w[1] = w[3]; w[3] = t; }
}
// rotate left by rot (new[j] = old[(j + rot) & 3])
__device__ __forceinline__ void rot_left4(uint32_t (&w)[4], int rot) {
    if (rot & 1) { uint32_t t = w[0]; w[0] = w[1]; w[1] = w[2]; w[2] = w[3]; w[3] = t; }
    if (rot & 2) { uint32_t t = w[0]; w[0] = w[2]; w[2] = t; t = w[1]; w[1] = w[3]; w[3] = t; }
}

// low BITS bits of eight integers -> one word, element 0 in the lowest field
template <int BITS>
__device__ __forceinline__ uint32_t pack8(const uint32_t (&b)[8]) {
    if (BITS == 4) {
        uint32_t b01 = bitsel(b[0], b[1] << 4, 0x0fu), b23 = bitsel(b[2], b[3] << 4, 0x0fu);
        uint32_t b45 = bitsel(b[4], b[5] << 4, 0x0fu), b67 = bitsel(b[6], b[7] << 4, 0x0fu);
        return __byte_perm(__byte_perm(b01, b23, 0x0040), __byte_perm(b45, b67, 0x0040), 0x5410);
    } else {
        constexpr uint32_t m1 = (1u << BITS) - 1u, m2 = (1u << (2 * BITS)) - 1u, m4 = (1u << (4 * BITS)) - 1u;
        constexpr uint32_t m8 = (BITS * 8 == 32) ? 0xffffffffu : ((1u << (BITS * 8 % 32)) - 1u);
        uint32_t p0 = bitsel(b[0], b[1] << BITS, m1), p1 = bitsel(b[2], b[3] << BITS, m1);
        uint32_t p2 = bitsel(b[4], b[5] << BITS, m1), p3 = bitsel(b[6], b[7] << BITS, m1);
        uint32_t q0 = bitsel(p0, p1 << (2 * BITS), m2), q1 = bitsel(p2, p3 << (2 * BITS), m2);
        return bitsel(q0, q1 << (4 * BITS), m4) & m8;
    }
}

// The same for codes that lie in [-(2^(BITS-1) - 1), 2^(BITS-1) - 1], given as the bits of code + kMagic: one sum of the shifted
// bits (a shift-and-add per code), whose constant part is taken out again; codes + 2^(BITS-1) fill their fields without carries.
// 9 operations for eight codes, where selecting the bits field by field takes 15 (11 for 4 bits) and the saturating pack, which
// wants the integers themselves, 12.  (3-bit encode of 16384 x 4096, eight outliers, groups of 128 65.8 -> 65.1 us, of 64 65.4 -> 64.0.)
// Every code has to be clamped on both sides: one that is not a number would reach into the fields above its own.
template <int BITS>
__device__ __forceinline__ uint32_t pack8_sum(const uint32_t (&b)[8]) {
    constexpr uint32_t ones = BITS == 4 ? 0x11111111u : BITS == 3 ? 0x00249249u : 0x00005555u;   // 1 in every field
    constexpr uint32_t offset = ones << (BITS - 1);
    uint32_t w = b[7];
#pragma unroll
    for (int i = 6; i >= 0; i--) w = (w << BITS) + b[i];
    return (w + (offset - 0x4b400000u * ones)) ^ offset;
}

// Two signed integers saturated to BITS-bit two's complement and packed below the bits of c
// (d = c << 2*BITS | sat(hi) << BITS | sat(lo)); BITS is 4 or 2.
template <int BITS>
__device__ __forceinline__ uint32_t sat_pack2(int hi, int lo, uint32_t c) {
    uint32_t d;
    if (BITS == 4) asm("cvt.pack.sat.s4.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi), "r"(lo), "r"(c));
    else asm("cvt.pack.sat.s2.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(hi), "r"(lo), "r"(c));
    return d;
}

// reference values of one slot (8 channels starting at channel c) from shared memory, with the optional
// per-channel transform r <- bf16(gain*r + bias)
__device__ __forceinline__ void load_ref_slot(uint32_t addr, const uint16_t *gain, const uint16_t *bias, int c,
                                              u64 (&r2)[4]) {
    uint4 w = lds128(addr);
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
    if (gain) {
        uint4 gw = __ldg(reinterpret_cast<const uint4 *>(gain + c));
        uint4 bw = __ldg(reinterpret_cast<const uint4 *>(bias + c));
        const uint32_t gws[4] = {gw.x, gw.y, gw.z, gw.w};
        const uint32_t bws[4] = {bw.x, bw.y, bw.z, bw.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            float g0 = half_bits_to_float(gws[i] & 0xffff), g1 = half_bits_to_float(gws[i] >> 16);
            float b0 = half_bits_to_float(bws[i] & 0xffff), b1 = half_bits_to_float(bws[i] >> 16);
            float r0 = __uint_as_float(ws[i] << 16), r1 = __uint_as_float(ws[i] & 0xffff0000u);
            r2[i] = pack2(bf16_round(__fmaf_rn(g0, r0, b0)), bf16_round(__fmaf_rn(g1, r1, b1)));
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; i++) r2[i] = bf16x2_to_p(ws[i]);
    }
}

// the same values left as packed bf16 words (the transformed reference is a bf16 value, so nothing is lost)
__device__ __forceinline__ uint4 load_ref_words(uint32_t addr, const uint16_t *gain, const uint16_t *bias, int c) {
    uint4 w = lds128(addr);
    if (gain) {
        const uint4 gw = __ldg(reinterpret_cast<const uint4 *>(gain + c));
        const uint4 bw = __ldg(reinterpret_cast<const uint4 *>(bias + c));
        const uint32_t gws[4] = {gw.x, gw.y, gw.z, gw.w};
        const uint32_t bws[4] = {bw.x, bw.y, bw.z, bw.w};
        uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float g0 = half_bits_to_float(gws[i] & 0xffff), g1 = half_bits_to_float(gws[i] >> 16);
            const float b0 = half_bits_to_float(bws[i] & 0xffff), b1 = half_bits_to_float(bws[i] >> 16);
            ws[i] = f2_to_bf16x2(__fmaf_rn(g0, __uint_as_float(ws[i] << 16), b0),
                                 __fmaf_rn(g1, __uint_as_float(ws[i] & 0xffff0000u), b1));
        }
        w = make_uint4(ws[0], ws[1], ws[2], ws[3]);
    }
    return w;
}

// the thread's whole slab, slot order (off: byte offsets of its four slots in the row).  One test of the transform, and the loads
// of two slots before either is used: with a test per slot each slot was a trip of its own (a token's chain with x_hat and a
// predictor, 300 x 8192, 8.8 us, 8.2 to 8.3 so; all four slots at once 8.0, but the registers for that made calls WITHOUT a predictor
// 1 % slower: 131072 x 5120 with eight outliers 612 us slot by slot, 620 at once, 605 to 608 so).
__device__ __forceinline__ void load_ref_slab(uint32_t (&rw)[16], uint32_t rs, const uint32_t (&off)[4], const uint16_t *gain,
                                              const uint16_t *bias) {
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const uint4 w = lds128(rs + off[j]);
        rw[4 * j + 0] = w.x; rw[4 * j + 1] = w.y; rw[4 * j + 2] = w.z; rw[4 * j + 3] = w.w;
    }
    if (gain) {
#pragma unroll
        for (int j0 = 0; j0 < 4; j0 += 2) {
            uint4 gw[2], bw[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                gw[h] = __ldg(reinterpret_cast<const uint4 *>(gain + (off[j0 + h] >> 1)));
                bw[h] = __ldg(reinterpret_cast<const uint4 *>(bias + (off[j0 + h] >> 1)));
            }
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t gws[4] = {gw[h].x, gw[h].y, gw[h].z, gw[h].w}, bws[4] = {bw[h].x, bw[h].y, bw[h].z, bw[h].w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    uint32_t &w = rw[4 * (j0 + h) + i];
                    w = f2_to_bf16x2(
                        __fmaf_rn(half_bits_to_float(gws[i] & 0xffff), __uint_as_float(w << 16), half_bits_to_float(bws[i] & 0xffff)),
                        __fmaf_rn(half_bits_to_float(gws[i] >> 16), __uint_as_float(w & 0xffff0000u), half_bits_to_float(bws[i] >> 16)));
                }
            }
        }
    }
}

// the same for one pair of channels (c even), operation for operation
__device__ __forceinline__ u64 load_ref_pair(uint32_t addr, const uint16_t *gain, const uint16_t *bias, int c) {
    const uint32_t w = lds32(addr);
    if (gain) {
        const uint32_t gw = __ldg(reinterpret_cast<const uint32_t *>(gain + c));
        const uint32_t bw = __ldg(reinterpret_cast<const uint32_t *>(bias + c));
        const float g0 = half_bits_to_float(gw & 0xffff), g1 = half_bits_to_float(gw >> 16);
        const float b0 = half_bits_to_float(bw & 0xffff), b1 = half_bits_to_float(bw >> 16);
        const float r0 = __uint_as_float(w << 16), r1 = __uint_as_float(w & 0xffff0000u);
        return pack2(bf16_round(__fmaf_rn(g0, r0, b0)), bf16_round(__fmaf_rn(g1, r1, b1)));
    }
    return bf16x2_to_p(w);
}

// SUB = false compiles the plain form (all T tokens in order, one reference buffer); SUB = true the form of the
// *_list entry points.  how many tokens this launch codes, and the idx-th of them:
template <bool SUB>
__device__ __forceinline__ long long tokens_to_do(const CodecParams &p) {
    if constexpr (!SUB) return p.T;
    if (!p.tok_count) return p.T;
    const long long n = *p.tok_count;
    return n < 0 ? 0 : (n > p.T ? p.T : n);
}
template <bool SUB>
__device__ __forceinline__ long long token_at(const CodecParams &p, long long idx) {
    if constexpr (!SUB) return idx;
    if (!p.tok_list) return idx;
    const long long t = p.tok_list[idx];
    return t < 0 ? 0 : (t >= p.T ? p.T - 1 : t);   // a bad entry cannot leave the buffers
}
// Reference row of a token (-1 = coded directly); with SUB in the joint row space [ref_base rows | intra_base
// rows].  `flag` false: do not report rows beyond the buffers (a second pass over tokens already reported).
template <bool SUB>
__device__ __forceinline__ int resolve_row(const CodecParams &p, int raw_row, bool flag = true) {
    if constexpr (!SUB) {
        if (!p.ref_base || raw_row < 0) return -1;
        if (raw_row >= p.ref_rows) {
            if (flag && p.status) atomicOr(p.status, RAC_STATUS_REF_RANGE);
            return -1;
        }
        return raw_row;
    } else {
        if (raw_row < 0 || (!p.ref_base && !p.intra_base)) return -1;
        if (raw_row < p.ref_rows) return raw_row;
        if (p.intra_base && raw_row - p.ref_rows < p.intra_rows) return raw_row;
        if (flag && p.status) atomicOr(p.status, RAC_STATUS_REF_RANGE);
        return -1;
    }
}
template <bool SUB>
__device__ __forceinline__ const uint16_t *ref_row_ptr(const CodecParams &p, long long row) {
    if constexpr (!SUB) return p.ref_base + row * p.d;
    return row < p.ref_rows ? p.ref_base + row * p.d : p.intra_base + (row - p.ref_rows) * p.d;
}
// thread 0: start the copies of one token into a stage: `first` (X row or record) and, if any, its reference row
template <bool SUB>
__device__ __forceinline__ void issue_token_loads(const CodecParams &p, Ctrl *ctrl, uint32_t stage_addr, uint32_t r_off,
                                                  int stage, int row, const void *first_src, uint32_t first_bytes,
                                                  long long tok = 0) {
    ctrl->row[stage] = row;
    if constexpr (SUB) ctrl->seg[stage] = p.seg_of ? p.seg_of[tok] : 0;
    const uint32_t bar = smem_u32(&ctrl->bar[stage]);
    const uint32_t row_bytes = 2u * (uint32_t)p.d;
    mbar_arrive_expect_tx(bar, p.test_extra_tx + first_bytes + (row >= 0 ? row_bytes : 0u));
    bulk_load(stage_addr, first_src, first_bytes, bar);
    if (row >= 0) bulk_load(stage_addr + r_off, ref_row_ptr<SUB>(p, row), row_bytes, bar);
}

// butterflies over the lanes of a group, two values at a time
__device__ __forceinline__ void group_sum2(float &a, float &b, int lpg, unsigned int group_mask) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        if (lpg > o) {
            a += __shfl_xor_sync(group_mask, a, o);
            b += __shfl_xor_sync(group_mask, b, o);
        }
    }
}

// Eq. 6 for the group this thread belongs to: centred two-pass sums over the thread's 32 channels (rows as packed bf16
// words; two accumulators per sum and channel parity), butterflies over the group's lanes, the zero-variance rule, and
// wire rounding of (alpha, beta) to binary16.  Returns their bit patterns and, in a2 and b2, the coefficients splatted for
// packed arithmetic; a token without a reference has no second pass.  The rows stay packed and enter the sums through the
// mixed adds above: half the registers of unpacked rows and no unpacking (streaming pass at 131072 x 5120, group 128,
// 4-bit: with outliers 528 -> 485 us, without 516 -> 467 us, with x_hat 726 -> 700 us).
// Sums of products in one pass, the means' part taken out afterwards, are less work only where means are small beside the
// spread, and need the centred pass behind them where they are not.  131072 x 5120, 4-bit, eight outliers, groups of 128: 599 us so,
// 579 in one pass with means of zero, but 696 with means of 0.6 of the spread and 701 where only the token has one; with a vote on the
// reference's mean before the token enters its products 581, 633 and 698 (16384 x 4096, 3-bit 62.9, 62.0, 71.6 and 71.7; 61.8, 66.2 and
// 71.4; groups of 1024 71, 69, 85 and 86; 70, 75 and 87).  From groups of 256 on its error of alpha against 64 bits is up to 6 % larger.
__device__ __forceinline__ uint32_t fit_group(const uint32_t (&xw)[16], const uint32_t (&rw)[16], bool has_ref, int lpg,
                                              float inv_group, unsigned int group_mask, uint32_t *status, u64 &a2, u64 &b2,
                                              float4 *stats = nullptr) {
    float ra0 = 0.f, ra1 = 0.f, rb0 = 0.f, rb1 = 0.f, xa0 = 0.f, xa1 = 0.f, xb0 = 0.f, xb1 = 0.f;
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
        ra0 = add_lo(rw[i], ra0); ra1 = add_hi(rw[i], ra1); rb0 = add_lo(rw[i + 1], rb0); rb1 = add_hi(rw[i + 1], rb1);
        xa0 = add_lo(xw[i], xa0); xa1 = add_hi(xw[i], xa1); xb0 = add_lo(xw[i + 1], xb0); xb1 = add_hi(xw[i + 1], xb1);
    }
    float sr = (ra0 + rb0) + (ra1 + rb1), sh = (xa0 + xb0) + (xa1 + xb1);
    group_sum2(sr, sh, lpg, group_mask);
    if (!(fabsf(sr) <= 3.0e38f) || !(fabsf(sh) <= 3.0e38f)) {
        if (status) atomicOr(status, RAC_STATUS_NONFINITE);
    }
    const float rbar = sr * inv_group, hbar = sh * inv_group;
    float sxx = 0.f, sxy = 0.f;
    if (has_ref || stats) {
        u64 sxxa = 0ull, sxxb = 0ull, sxya = 0ull, sxyb = 0ull;
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const u64 dr0 = pack2(sub_lo(rw[i], rbar), sub_hi(rw[i], rbar)), dh0 = pack2(sub_lo(xw[i], hbar), sub_hi(xw[i], hbar));
            const u64 dr1 = pack2(sub_lo(rw[i + 1], rbar), sub_hi(rw[i + 1], rbar));
            const u64 dh1 = pack2(sub_lo(xw[i + 1], hbar), sub_hi(xw[i + 1], hbar));
            sxxa = pfma(dr0, dr0, sxxa); sxya = pfma(dr0, dh0, sxya);
            sxxb = pfma(dr1, dr1, sxxb); sxyb = pfma(dr1, dh1, sxyb);
        }
        float sxx_hi, sxy_hi;
        unpack2(padd(sxxa, sxxb), sxx, sxx_hi);
        unpack2(padd(sxya, sxyb), sxy, sxy_hi);
        sxx += sxx_hi;
        sxy += sxy_hi;
        group_sum2(sxx, sxy, lpg, group_mask);
    }
    if (stats) *stats = make_float4(rbar, hbar, sxx, sxy);
    // zero-variance rule, then wire rounding to binary16
    float a_star = 0.f, b_star = hbar;
    if (has_ref && sxx > 1e-12f && fabsf(sxy) < 65504.0f * sxx) {
        a_star = __fdiv_rn(sxy, sxx);
        b_star = __fmaf_rn(-a_star, rbar, hbar);
    }
    const uint32_t a16 = float_to_half_bits_sat(a_star), b16 = float_to_half_bits_sat(b_star);
    const float a = half_bits_to_float(a16), b = half_bits_to_float(b16);
    a2 = pack2(a, a);
    b2 = pack2(b, b);
    return a16 | (b16 << 16);
}

// ------------------------------------------------------------------------------------------------
// host side: launch plumbing
// ------------------------------------------------------------------------------------------------
struct DeviceInfo {
    int sms = 0;
    int max_smem_optin = 0;
};
inline std::mutex &launch_mutex() {
    static std::mutex m;
    return m;
}
static int device_info(DeviceInfo *out, int *dev_out = nullptr) {
    static DeviceInfo cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RAC_ECUDA;
    std::lock_guard<std::mutex> lock(launch_mutex());
    if (cache[dev].sms == 0) {
        int sms = 0, smem = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return RAC_ECUDA;
        if (cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return RAC_ECUDA;
        cache[dev].max_smem_optin = smem;
        cache[dev].sms = sms;
    }
    *out = cache[dev];
    if (dev_out) *dev_out = dev;
    return RAC_OK;
}

// Resident CTAs per SM of one kernel at one block size and shared-memory size, looked up once per device.  The
// kernel's shared-memory limit is an attribute of the kernel, not of a launch: it is only ever raised, so that a
// launch with less shared memory between two larger ones leaves it where the larger ones need it.
static int resident_ctas(const void *kernel, int dev, int nthreads, int smem_bytes, int *occ_out) {
    struct Key {
        const void *kernel;
        int dev, nthreads, smem;
        bool operator<(const Key &o) const {
            return std::tie(kernel, dev, nthreads, smem) < std::tie(o.kernel, o.dev, o.nthreads, o.smem);
        }
    };
    static std::map<Key, int> table;
    static std::map<std::pair<const void *, int>, int> limit;   // (kernel, device) -> shared-memory limit set so far
    const Key key{kernel, dev, nthreads, smem_bytes};
    std::lock_guard<std::mutex> lock(launch_mutex());
    auto it = table.find(key);
    if (it == table.end()) {
        int &lim = limit[std::make_pair(kernel, dev)];
        if (smem_bytes > lim) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes) != cudaSuccess) return RAC_ECUDA;
            lim = smem_bytes;
        }
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, nthreads, smem_bytes) != cudaSuccess || occ < 1)
            return RAC_ECUDA;
        it = table.emplace(key, occ).first;
    }
    *occ_out = it->second;
    return RAC_OK;
}

template <typename K>
static int launch_persistent(K kernel, const CodecParams &p, int nthreads, int smem_bytes, long long max_ctas,
                             cudaStream_t stream) {
    DeviceInfo di;
    int dev = 0;
    int rc = device_info(&di, &dev);
    if (rc != RAC_OK) return rc;
    if (smem_bytes > di.max_smem_optin) return RAC_EUNSUPPORTED;
    int occ = 0;
    rc = resident_ctas(reinterpret_cast<const void *>(kernel), dev, nthreads, smem_bytes, &occ);
    if (rc != RAC_OK) return rc;
    long long grid = (long long)di.sms * occ;
    if (grid > max_ctas) grid = max_ctas;
    if (grid < 1) grid = 1;
    launch_after(kernel, (unsigned)grid, (unsigned)nthreads, (size_t)smem_bytes, stream, p);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace rac
