// RAC codec kernels for sm_100a: encode (Sec. IV-C, Eq. 6-8 + packing, outlier split) and reconstruct (Eq. 9).
//
// Shape of the streaming kernels: persistent CTAs, one token per CTA iteration, one thread per 32
// consecutive channels.  Rows travel between HBM and shared memory only as 1-D bulk copies (TMA without a
// tensor map): a ring of stages is filled ahead and signalled through mbarriers, finished records and rows
// leave through bulk stores.  Every wait on an mbarrier is bounded; a copy that never lands ends the kernel
// with a status bit instead of a hang.  The arithmetic that decides integers (residual, scaling, rounding)
// is binary32 with one rounding per operation, written with explicit intrinsics / PTX so the compiler
// cannot contract or reorder it.
//
// Shared-memory reads of a thread's 64-byte slab go through a per-lane rotation of the four 16-byte
// pieces (piece (j + lane/2) mod 4 in step j), which makes the 128-bit accesses bank-conflict free
// on a plain linear row.
//
// Kernels: encode_ws_kernel (encode without outliers, or the streaming pass of one with them; optionally also the sender-side
// x_hat), outlier_kernel (second launch of some encodes with outliers: the k largest |e| per token), encode_top_kernel (both in
// one launch, where that is the better form), decode_kernel and decode_ws_kernel
// (receiver and sender reconstruction, with and without per-token outliers), split_waves_kernel (tokens that
// reference the same prompt go second).  The kernels of the per-group-scale quantiser (Eq. 8 as printed) live in
// rac_codec_dyn.cu; this file holds the C ABI of both.  Step tables, segment fit and reconstruction error: rac_calib.cu.
#include <cstring>

#include "rac_codec_dev.cuh"

namespace rac {

// ------------------------------------------------------------------------------------------------
// geometry / validation (host)
// ------------------------------------------------------------------------------------------------
static bool is_pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }

int make_geometry(const rac_codec_cfg *cfg, Geometry *g) {
    if (!cfg) return RAC_EINVAL;
    if (cfg->d <= 0 || cfg->group <= 0 || cfg->topk < 0 || cfg->bits <= 0) return RAC_EINVAL;
    if (cfg->qgroup < 0 || cfg->topk_group < 0) return RAC_EINVAL;
    if ((cfg->coef_fmt != 0 && cfg->coef_fmt != 1) || cfg->flags != 0) return RAC_EUNSUPPORTED;
    if (cfg->scale_mode != 0 && cfg->scale_mode != 1) return RAC_EUNSUPPORTED;
    if (cfg->d % cfg->group) return RAC_EINVAL;
    if (cfg->d % 32 || cfg->d > 8192) return RAC_EUNSUPPORTED;
    if (!is_pow2(cfg->group) || cfg->group < 32 || cfg->group > 1024) return RAC_EUNSUPPORTED;
    if (cfg->topk > 16 || cfg->topk > cfg->d) return RAC_EUNSUPPORTED;
    int qgroup = cfg->qgroup ? cfg->qgroup : cfg->group;
    int lpq = 0, qgen = 0;
    if (cfg->scale_mode == 0) {
        // the static table: one grouping, per-token outliers, 2..4 bits
        if (qgroup != cfg->group || cfg->topk_group != 0) return RAC_EUNSUPPORTED;
        if (cfg->bits < 2 || cfg->bits > 4) return RAC_EUNSUPPORTED;
        lpq = cfg->group / 32;
    } else {
        // Eq. 8 takes the scale from the dense values, i.e. after the outliers are known.  The per-token
        // selection runs as a second launch, after the codes exist, so this mode offers the paper's own
        // per-group outliers (picked inside the streaming pass) and not the per-token ones.
        if (cfg->topk != 0) return RAC_EUNSUPPORTED;
        if (cfg->bits != 2 && cfg->bits != 3 && cfg->bits != 4 && cfg->bits != 8) return RAC_EUNSUPPORTED;
        if (cfg->d % qgroup) return RAC_EINVAL;
        if (is_pow2(qgroup) && qgroup >= 32 && qgroup <= 1024) lpq = qgroup / 32;
        else if (qgroup == cfg->d) lpq = 0;   // one scale per token, exchanged through shared memory
        else if (qgroup % 32 == 0) { lpq = 0; qgen = qgroup / 32; }   // any other whole number of lanes: the same exchange
        else return RAC_EUNSUPPORTED;
        if (cfg->topk_group > 8) return RAC_EUNSUPPORTED;
        if (cfg->topk_group > 0 && lpq == 0) return RAC_EUNSUPPORTED;   // a group must lie within one warp
    }
    g->d = cfg->d;
    g->group = cfg->group;
    g->bits = cfg->bits;
    g->topk = cfg->topk;
    g->J = cfg->d / cfg->group;
    g->lpg = cfg->group / 32;
    g->nthreads = ((cfg->d / 32) + 31) / 32 * 32;
    g->code_bytes = cfg->d * cfg->bits / 8;
    g->scale_mode = cfg->scale_mode;
    g->qgroup = qgroup;
    g->Jq = cfg->d / qgroup;
    g->lpq = lpq;
    g->qgen = qgen;
    g->topk_group = cfg->topk_group;
    g->coef_fmt = cfg->coef_fmt;
    g->scale_off = cfg->coef_fmt == 1 ? 0 : 4 * g->J;
    g->codes_off = g->scale_off + (cfg->scale_mode == 1 ? (2 * g->Jq + 3) / 4 * 4 : 0);
    const int ng = g->Jq * g->topk_group;
    g->goff_off = g->codes_off + g->code_bytes + 4 * cfg->topk;
    g->gval_off = g->goff_off + (ng * (qgroup > 256 ? 2 : 1) + 1) / 2 * 2;   // one-byte offsets up to 256 channels, two beyond
    const int raw = g->gval_off + 2 * ng;
    g->rec = (raw + 15) / 16 * 16;
    return RAC_OK;
}

// ------------------------------------------------------------------------------------------------
// encode
// ------------------------------------------------------------------------------------------------
// Without outliers one launch of the streaming pass; with outliers one launch of encode_top_kernel (below) or two launches (the
// rule is one_launch's).  (1) The streaming pass (this kernel): statistics, coefficients, residual, codes; every
// warp of the CTA works on its 1024 channels of the token and ends with ONE arrival on the stage's `done`
// mbarrier -- there is no CTA barrier in the loop.  Handing the finished record to the copy engine and
// refilling the stage is the duty of warp (i mod warps) for token i; the other warps are already in the
// next token and only ever wait for data (`full`).  With outliers, every thread also writes the largest
// |e| of its 32 channels to the caller's workspace.  (2) outlier_kernel picks the k largest |e| per token
// from those maxima with one warp per token -- thousands of tokens in flight, so the serial selection
// (threshold, candidates, ranking) costs latency nobody waits for -- and patches the records in place.
struct WsCtrl {
    unsigned long long full[kMaxStages];
    unsigned long long done[kMaxStages];
    int row[kMaxStages];
    int seg[kMaxStages];   // segment of the token in each stage (shared coefficients only)
    int abort;
};

struct WsSmem {
    int stage0, stage_bytes, rec_off, tm_off, tm_bytes, total;
};
__host__ __device__ inline WsSmem ws_smem_layout(int d, int rec, int stages, bool topk) {
    WsSmem s;
    s.stage0 = align_up((int)sizeof(WsCtrl), 128);
    s.rec_off = 4 * d;  // after X row + R row: two record slots, used alternately (by the stage's parity)
    s.tm_off = s.rec_off + 2 * rec;  // two slots of per-slab maxima (outliers only), same alternation
    s.tm_bytes = topk ? align_up((d / 32) * 4, 16) : 0;
    s.stage_bytes = align_up(s.tm_off + 2 * s.tm_bytes, 128);
    s.total = s.stage0 + stages * s.stage_bytes;
    return s;
}

// Both step tables in shared memory, laid out by thread: the 16-byte pieces that a thread reads in one step of its work (for half h
// of slot j piece 2j + h of a row of inverse steps; a slot's binary16 steps are one piece) stand side by side for all threads of a
// token, so that a warp's access is 512 consecutive bytes.  Read in place a warp's access touches 32 cache lines (9 wavefronts of
// the L1 data pipe against 4), and with x_hat the four rows of a width of 5120 are more than the L1 beside the stages.
// There is room for 24 pieces per thread.  TABLES = 1: both rows of inverse steps and both rows of steps as binary16, which holds
// calibrated tables.  TABLES = 2, for a caller's own steps that it does not hold: both rows of steps as binary32 and the first row of
// inverse steps; directly coded tokens read the second in place.  (Gathered rows, 28 % of them direct, binary16 / binary32 / without
// these tables, us: 12000 x 3072 48.4 / 49.0 / 51.5, x 4096 61.1 / 63.2 / 65.4, x 5120 80.9 / 87.5 / 88.0, 16000 x 6144 123.0 / 132.3 / 139.0;
// groups of 256 at 24000 x 5120 165 / 184 / 173.  One body for both, with a test per slot, took 2 to 5 % longer than two.)
struct SlabTables {
    uint32_t inv = 0, step = 0;            // this thread's first pieces
    uint32_t pitch = 0;                    // bytes from one piece of a thread to its next
};
__device__ __forceinline__ float4 lds128f(uint32_t addr) {
    const uint4 w = lds128(addr);
    return make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
}

// One thread's 32 channels of one token, rows and record in shared memory: Eq. 6, Eq. 7, Eq. 8 with the static table, packing,
// the sender-side reconstruction (over the X row), and the largest |e| of the slab.
// STEPREG: every token has a reference, and the thread holds its steps (row 0 of the table, slot order) in st0.
// SATPACK: 4- and 2-bit codes beside x_hat through the saturating pack, as without x_hat, instead of the sum of shifted bits: that
// is more operations in a shorter chain.  One CTA per token of up to 160 threads: gathered 2960 x 5120 24.7 us by the sum, 23.4 so,
// x 4608 22.4 and 21.9, 64 x 4096 6.28 and 6.22; of more threads 300 x 6144 7.5 and 7.8; teams 16384 x 3072 63.7 and 64.8; the streaming pass
// the same by either.
template <int BITS, bool TOPK, bool XHAT, int LPG, bool STEPREG, int TABLES = 0, bool SATPACK = false>
__device__ __forceinline__ void encode_slab(const CodecParams &p, int tid, int lane, int rot, int d, int Jc, bool shared, int coff,
                                            const uint32_t (&off)[4], unsigned int group_mask, uint32_t xs, uint32_t rs,
                                            bool has_ref, int seg, unsigned char *rec, float *tm, const u64 (&st0)[STEPREG ? 16 : 1],
                                            const SlabTables tab = SlabTables()) {
    constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
    const u64 magic2 = pack2(kMagic, kMagic);
    // ---- (1) the slab: 4 slots of 8 channels, slot j holds piece (j + rot) & 3
    uint32_t xw[16], rw[16];   // packed bf16, slot order
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const uint4 w = lds128(xs + off[j]);
        xw[4 * j + 0] = w.x; xw[4 * j + 1] = w.y; xw[4 * j + 2] = w.z; xw[4 * j + 3] = w.w;
    }
    if (has_ref) {
        load_ref_slab(rw, rs, off, p.gain, p.bias);
    } else {
#pragma unroll
        for (int i = 0; i < 16; i++) rw[i] = 0u;
    }
    // ---- (2) Eq. 6 and wire rounding
    u64 a2, b2;
    constexpr int kShift = LPG == 4 ? 2 : 1;
    const int lpg = LPG ? LPG : p.lpg, lpg_shift = LPG ? kShift : p.lpg_shift;
    if (shared) {
        const uint32_t cw = p.coef_ext[(long long)seg * Jc + (tid >> lpg_shift)];
        const float a = half_bits_to_float(cw & 0xffffu), b = half_bits_to_float(cw >> 16);
        a2 = pack2(a, a);
        b2 = pack2(b, b);
    } else {
        const uint32_t coef_word = fit_group(xw, rw, has_ref, lpg, p.inv_group, group_mask, p.status, a2, b2);
        if ((lane & (lpg - 1)) == 0) reinterpret_cast<uint32_t *>(rec)[tid >> lpg_shift] = coef_word;
    }

    // ---- (3) Eq. 7 residual, Eq. 8 quantisation with the static table, packing
    const float *inv_tab = p.inv_step + (has_ref ? 0 : d);
    const float *step_tab = p.step + (has_ref ? 0 : d);
    uint32_t words[4];
    float tmax = 0.f;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const int c = (int)(off[j] >> 1);
        float4 iv0, iv1;
        if (TABLES == 1 || (TABLES == 2 && has_ref)) {
            const uint32_t a = tab.inv + (has_ref ? 0u : 8u * tab.pitch) + 2 * j * tab.pitch;
            iv0 = lds128f(a);
            iv1 = lds128f(a + tab.pitch);
        } else {
            iv0 = __ldg(reinterpret_cast<const float4 *>(inv_tab + c));
            iv1 = __ldg(reinterpret_cast<const float4 *>(inv_tab + c + 4));
        }
        const u64 inv2[4] = {pack2(iv0.x, iv0.y), pack2(iv0.z, iv0.w), pack2(iv1.x, iv1.y), pack2(iv1.z, iv1.w)};
        u64 st2[4] = {0ull, 0ull, 0ull, 0ull};
        if (XHAT) {
            if (STEPREG) {
#pragma unroll
                for (int i = 0; i < 4; i++) st2[i] = st0[STEPREG ? 4 * j + i : 0];
            } else if (TABLES == 1) {
                const uint4 w = lds128(tab.step + (has_ref ? 0u : 4u * tab.pitch) + j * tab.pitch);
                const uint32_t hw[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&hw[i]));
                    st2[i] = pack2(f.x, f.y);
                }
            } else {
                float4 s0, s1;
                if (TABLES == 2) {
                    const uint32_t a = tab.step + (has_ref ? 0u : 8u * tab.pitch) + 2 * j * tab.pitch;
                    s0 = lds128f(a);
                    s1 = lds128f(a + tab.pitch);
                } else {
                    s0 = __ldg(reinterpret_cast<const float4 *>(step_tab + c));
                    s1 = __ldg(reinterpret_cast<const float4 *>(step_tab + c + 4));
                }
                st2[0] = pack2(s0.x, s0.y); st2[1] = pack2(s0.z, s0.w); st2[2] = pack2(s1.x, s1.y); st2[3] = pack2(s1.z, s1.w);
            }
        }
        float ev[8];
        uint32_t xh[4];
        uint32_t w = 0;
        if (BITS == 3 || (XHAT && !SATPACK)) {
            // clamped on both sides: 3-bit codes have no saturating pack, and with x_hat the float is used again
            uint32_t bits8[8];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const u64 rt = pfma(a2, bf16x2_to_p(rw[4 * j + i]), b2);
                const u64 e = sub_pair(xw[4 * j + i], rt);
                float v0, v1, t0, t1;
                unpack2(pmul(e, inv2[i]), v0, v1);
                t0 = fminf(fmaxf(v0, -qmax), qmax);
                t1 = fminf(fmaxf(v1, -qmax), qmax);
                const u64 tt = padd(pack2(t0, t1), magic2);
                unpack2(tt, t0, t1);
                bits8[2 * i] = __float_as_uint(t0);
                bits8[2 * i + 1] = __float_as_uint(t1);
                unpack2(e, ev[2 * i], ev[2 * i + 1]);
                if (XHAT) {
                    // Eq. 9 with the code just chosen: x_hat = bf16(fma(q, step, alpha*r + beta)); a binary16-valued
                    // step makes q*step exact, so the fused form and (alpha*r + beta) + q*step are the same bits
                    float x0, x1;
                    unpack2(pfma(psub(tt, magic2), st2[i], rt), x0, x1);
                    xh[i] = f2_to_bf16x2(x0, x1);
                }
            }
            w = pack8_sum<BITS>(bits8);
        } else {
            // 4- and 2-bit codes: clamp from below in binary32, round by the magic add, take the integer
            // out of the mantissa and let the saturating pack clamp from above (its range is
            // [-2^(BITS-1), 2^(BITS-1)-1], whose upper end is Qmax)
#pragma unroll
            for (int i = 3; i >= 0; i--) {
                const u64 rt = pfma(a2, bf16x2_to_p(rw[4 * j + i]), b2);
                const u64 e = sub_pair(xw[4 * j + i], rt);
                float v0, v1, t0, t1;
                unpack2(pmul(e, inv2[i]), v0, v1);
                v0 = fmaxf(v0, -qmax);
                v1 = fmaxf(v1, -qmax);
                if (XHAT) { v0 = fminf(v0, qmax); v1 = fminf(v1, qmax); }  // the float is used again below
                const u64 tt = padd(pack2(v0, v1), magic2);
                unpack2(tt, t0, t1);
                w = sat_pack2<BITS>((int)__float_as_uint(t1) - 0x4b400000, (int)__float_as_uint(t0) - 0x4b400000, w);
                unpack2(e, ev[2 * i], ev[2 * i + 1]);
                if (XHAT) {
                    float x0, x1;
                    unpack2(pfma(psub(tt, magic2), st2[i], rt), x0, x1);
                    xh[i] = f2_to_bf16x2(x0, x1);
                }
            }
        }
        words[j] = w;
        // sender-side reconstruction: the thread's own slab of the X row now carries x_hat
        if (XHAT) sts128(xs + off[j], make_uint4(xh[0], xh[1], xh[2], xh[3]));
        if (TOPK) {
            const float m0 = fmaxf(fmaxf(fabsf(ev[0]), fabsf(ev[1])), fmaxf(fabsf(ev[2]), fabsf(ev[3])));
            const float m1 = fmaxf(fmaxf(fabsf(ev[4]), fabsf(ev[5])), fmaxf(fabsf(ev[6]), fabsf(ev[7])));
            tmax = fmaxf(tmax, fmaxf(m0, m1));
        }
    }
    rot_right4(words, rot);  // words[q] is now the code word of piece q
    uint32_t *cw = reinterpret_cast<uint32_t *>(rec + coff) + tid * BITS;
    if (BITS == 4) {
        cw[0] = words[0]; cw[1] = words[1]; cw[2] = words[2]; cw[3] = words[3];
    } else if (BITS == 3) {
        cw[0] = words[0] | (words[1] << 24);
        cw[1] = (words[1] >> 8) | (words[2] << 16);
        cw[2] = (words[2] >> 16) | (words[3] << 8);
    } else {
        cw[0] = words[0] | (words[1] << 16);
        cw[1] = words[2] | (words[3] << 16);
    }
    // (4) the largest |e| of this thread's 32 channels, for the outlier pass
    if (TOPK) tm[tid] = tmax;
}

// SUB: the token-list / second-reference-buffer form (see rac_codec_dev.cuh).
// LPG: lanes per alignment group as a compile-time constant (4 = groups of 128 channels, 2 = groups of 64), or 0 to
// read it from the parameters; the constant removes the uniform branches of the shuffle reductions.
// D: the hidden width as a compile-time constant (4096 and 5120 are compiled in), or 0 to read it from the parameters;
// the constant folds the address arithmetic of the rows and stages (without outliers, 131072 x 5120 485 -> 458 us, x 4096 394 ->
// 383 us; with x_hat, gathered rows and a predictor, with eight outliers, 100000 x 5120 815 -> 786 us in both launches).
// REF: every token has a reference row (identity rows: no row list, a reference buffer): the per-token test and the
// second row of the tables go away (without outliers, 131072 x 5120 474 -> 458 us; with x_hat see launch_stream_lpg).
template <int BITS, bool TOPK, bool XHAT, int MINB, bool SUB, int LPG = 0, int D = 0, bool REF = false>
__global__ void __launch_bounds__(MINB == 4 ? 160 : 256, MINB) encode_ws_kernel(const CodecParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = D ? (D / 32 + 31) / 32 : nt >> 5;
    const int rot = (lane >> 1) & 3;
    const int d = D ? D : p.d;
    const bool valid = tid * 32 < d;
    constexpr int S = 2;   // stages of the ring (the host sets p.stages to the same)
    // with the width and the group compiled in, the record geometry is a constant too (those variants are launched for
    // no outliers or eight per token only)
    constexpr bool kGeo = D != 0 && LPG != 0;
    const int Jc = kGeo ? D / (32 * (LPG ? LPG : 1)) : p.J;
    const int codeb = kGeo ? D * BITS / 8 : p.code_bytes;
    const int recb = kGeo ? (4 * (D / (32 * (LPG ? LPG : 1))) + D * BITS / 8 + (TOPK ? 32 : 0) + 15) / 16 * 16 : p.rec;
    const WsSmem L = ws_smem_layout(d, recb, S, TOPK);
    WsCtrl *ctrl = reinterpret_cast<WsCtrl *>(smem);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t row_bytes = 2u * (uint32_t)d;

    if (p.T <= gridDim.x) grid_launch_dependents();
    if (tid == 0) {
        for (int s = 0; s < S; s++) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->done[s]), nwarps);
        }
        ctrl->abort = 0;
        mbar_init_fence();
    }
    // shared coefficients (one pair per segment and group, Eq. 6 over several positions) come from outside the
    // records: no coefficient words in front of the codes
    bool shared = false;
    if constexpr (SUB) shared = p.coef_ext != nullptr;
    const int coff = shared ? 0 : 4 * Jc;
    {
        // padding words of the records are written once and never touched again
        const int raw = coff + codeb + 4 * p.topk;
        for (int s = 0; s < 2 * S; s++)
            for (int o = raw + 4 * tid; o < recb; o += 4 * nt)
                *reinterpret_cast<uint32_t *>(smem + L.stage0 + (s >> 1) * L.stage_bytes + L.rec_off + (s & 1) * recb + o) = 0u;
    }
    __syncthreads();
    grid_dependency_wait();
    const int first = blockIdx.x, stride = gridDim.x;
    const long long n_tok = tokens_to_do<SUB>(p);
    const int n_my = (n_tok > first) ? (int)((n_tok - first + stride - 1) / stride) : 0;
    auto raw_row_of = [&](int k) -> int {  // raw ref_row entry of this CTA's k-th token
        long long t = token_at<SUB>(p, first + (long long)k * stride);
        return p.ref_row ? p.ref_row[t] : (int)t;
    };
    // one lane: start the copies of this CTA's k-th token into stage s
    auto issue = [&](int k, int s, int raw_row) {
        const long long t = token_at<SUB>(p, first + (long long)k * stride);
        const int row = resolve_row<SUB>(p, raw_row);
        ctrl->row[s] = row;
        if constexpr (SUB) ctrl->seg[s] = p.seg_of ? p.seg_of[t] : 0;
        const uint32_t bar = smem_u32(&ctrl->full[s]);
        const uint32_t base = sbase + L.stage0 + s * L.stage_bytes;
        mbar_arrive_expect_tx(bar, p.test_extra_tx + row_bytes + (row >= 0 ? row_bytes : 0u));
        bulk_load(base, p.X + t * d, row_bytes, bar);
        if (row >= 0) bulk_load(base + row_bytes, ref_row_ptr<SUB>(p, row), row_bytes, bar);
    };
    if (tid == 0)
        for (int k = 0; k < S && k < n_my; k++) issue(k, k, raw_row_of(k));

    uint32_t off[4];
#pragma unroll
    for (int j = 0; j < 4; j++) off[j] = (uint32_t)(tid * 64 + ((j + rot) & 3) * 16);
    const unsigned int group_mask = __ballot_sync(0xffffffffu, valid);

    // x_hat where every token has a reference: the thread's steps stay in registers (it always owns the same channels), which
    // leaves L1 to the other table (65536 x 5120 without outliers 346 -> 330 us, 9000 x 8192 130 -> 103 us).  Where a call can
    // contain direct tokens the same with a branch per token was slower (long uplink 905 -> 980 us).
    constexpr bool kStepReg = XHAT && REF;
    u64 st0[kStepReg ? 16 : 1] = {};
    if (kStepReg) {
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
            if (valid) {
                s0 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1)));
                s1 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1) + 4));
            }
            st0[kStepReg ? 4 * j + 0 : 0] = pack2(s0.x, s0.y);
            st0[kStepReg ? 4 * j + 1 : 0] = pack2(s0.z, s0.w);
            st0[kStepReg ? 4 * j + 2 : 0] = pack2(s1.x, s1.y);
            st0[kStepReg ? 4 * j + 3 : 0] = pack2(s1.z, s1.w);
        }
    }

    int stage = 0, duty = 0;  // duty: the warp whose turn the tail of this token is
    uint32_t parity = 0;
    bool timed_out = false;
    for (int it = 0; it < n_my; it++) {
        if (*reinterpret_cast<volatile int *>(&ctrl->abort)) break;
        unsigned char *stg = smem + L.stage0 + stage * L.stage_bytes;
        const uint32_t xs = sbase + L.stage0 + stage * L.stage_bytes;
        const uint32_t rs = xs + row_bytes;
        unsigned char *rec = stg + L.rec_off + parity * recb;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->full[stage]), parity))) { timed_out = true; break; }
        const bool has_ref = REF ? true : ctrl->row[stage] >= 0;

        if (valid)
            encode_slab<BITS, TOPK, XHAT, LPG, kStepReg>(p, tid, lane, rot, d, Jc, shared, coff, off, group_mask, xs, rs, has_ref,
                                               SUB ? ctrl->seg[stage] : 0, rec,
                                               reinterpret_cast<float *>(stg + L.tm_off + parity * L.tm_bytes), st0);
        // this warp's share of the token is in shared memory: one arrival per warp
        fence_async_smem();  // the record (and x_hat) bytes written above will be read by the copy engine
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&ctrl->done[stage])) : "memory");

        if (warp == duty) {
            // ---- this warp's turn: hand the record over and refill the stage; the others have moved on
            const int k_next = it + S;
            int raw_next = 0;
            if (lane == 0 && k_next < n_my) raw_next = raw_row_of(k_next);  // in flight while the tail runs
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->done[stage]), parity))) { timed_out = true; break; }
            // ---- refill the stage, then hand the record to the copy engine.  The record sits in the slot of the
            // stage's current parity; the stage's next token writes the other slot, and the one after that
            // cannot start before this warp has arrived for the token in between, which it does only after the
            // wait below.  So the refill need not wait for the record to leave.  (With x_hat the X row itself
            // is the source of a store and must have been read before new data may land on it.)
            if (lane == 0) {
                const long long t = token_at<SUB>(p, first + (long long)it * stride);
                if (TOPK)  // the slab maxima travel like the record: one bulk copy from this parity's slot
                    bulk_store(p.tmax + t * (L.tm_bytes >> 2), xs + L.tm_off + parity * L.tm_bytes, (uint32_t)L.tm_bytes);
                if (XHAT) {
                    bulk_store(p.payload + t * recb, smem_u32(rec), (uint32_t)recb);
                    bulk_store(p.X_hat + t * d, xs, row_bytes);
                    bulk_commit();
                    bulk_wait_read<0>();
                    if (k_next < n_my) issue(k_next, stage, raw_next);
                } else {
                    if (k_next < n_my) issue(k_next, stage, raw_next);
                    bulk_store(p.payload + t * recb, smem_u32(rec), (uint32_t)recb);
                    bulk_commit();
                    bulk_wait_read<0>();
                }
            }
            __syncwarp();
        }
        if (++stage == S) { stage = 0; parity ^= 1u; }
        if (++duty == nwarps) duty = 0;
    }
    if (timed_out) {
        ctrl->abort = 1;
        if (p.status) atomicOr(p.status, RAC_STATUS_TIMEOUT);
    }
    __syncthreads();
    if (lane == 0) bulk_wait_all();  // every lane that stored records waits for its own copies
    if (tid == 0 && *reinterpret_cast<volatile int *>(&ctrl->abort)) {
        // give copies that may still be in flight a bounded chance to land before the CTA retires
        for (int s = 0; s < S; s++) {
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 0);
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 1);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// encode, second launch: outlier split (the k largest |e| per token, ties to the lower channel)
// ------------------------------------------------------------------------------------------------
// One warp per token.  Input: the per-thread maxima the streaming pass left in the workspace (one value per
// 32-channel slab); lane l holds the NV consecutive slabs NV*l .. NV*l+NV-1, so lane order is channel order.
// (a) Threshold tau: every lane offers its two largest maxima (two different slabs); k-1 rounds of a warp-wide
// maximum over the heads, the lowest lane that holds it moving on to its second value, then one more maximum.
// The k values seen are maxima of k different slabs, so at least k elements reach tau, and an element that
// reaches it can only sit in a slab whose maximum does.  tau is the exact k-th largest slab maximum unless one
// lane holds three of the k largest, and then only lower: a few more slabs are looked at, the result is the same.
// (b) The slabs that reach tau -- k of them unless maxima tie -- are listed in slab order and their residuals
// recomputed from X, the reference row and the wire coefficients in the record, four lanes per slab, eight
// channels per lane, with the same binary32 operations as the streaming pass (so the same bits).  Elements at or
// above tau are candidates, collected in channel order, one per lane.  (c) While there are more than k, the
// smallest goes (smallest magnitude; among equals the highest channel): the survivors are the k largest with
// ties to the lower channel, still in channel order.  More than 32 candidates (many equal magnitudes, e.g. an
// all-zero residual): a pass over the whole token instead.  (d) The winners go into the record's
// outlier fields in channel order, their dense codes are cleared (E^d = E - O), and with the sender-side
// reconstruction those channels of x_hat are replaced.
constexpr int kOutCap = 32;        // candidates per token: one per lane

// eight values by a run-time index, as a select tree (no local-memory array)
__device__ __forceinline__ float pick8(const float (&v)[8], int i) {
    const float a0 = (i & 1) ? v[1] : v[0], a1 = (i & 1) ? v[3] : v[2], a2 = (i & 1) ? v[5] : v[4], a3 = (i & 1) ? v[7] : v[6];
    const float b0 = (i & 2) ? a1 : a0, b1 = (i & 2) ? a3 : a2;
    return (i & 4) ? b1 : b0;
}

// Whole-token path (rare): the k largest |e| of all d channels, ties to the lower channel, by one warp.  One pass over the rows
// in channel order, 256 channels at a time, eight per lane; lanes 0..k-1 hold the k best so far, lane r returns its channel,
// residual and aligned reference (in no order).  What comes later has the higher channel, so it replaces the smallest held one
// only with a larger magnitude, and of equal ones held the highest channel goes: at most k replacements per 256 channels.
// Bound by the trips for the rows, the next of which is under way while one is looked at.  k rounds of a maximum over the whole
// token, one channel per lane and trip, took 150 us per token at d = 4096, k = 8; this takes 5.  (16384 such tokens, all residuals
// zero: 1.61 ms when the warps of a second launch did it, 4.40 ms when the selectors of encode_top_kernel did, 0.17 ms so.)
struct Winner {
    int c;
    float e, rt;
};
__device__ __noinline__ Winner select_whole_token(int d, int k, int coef_shift, const uint16_t *xrow, const uint16_t *rrow,
                                                  const uint16_t *gain, const uint16_t *bias, const uint32_t *coef, int lane) {
    int held = lane < k ? -1 : 0x7fffffff;     // magnitude (bits) this lane holds, -1: none yet
    int hc = 0x10000 + lane;                   // its channel
    float he = 0.f, hrt = 0.f;
    uint4 xn = make_uint4(0u, 0u, 0u, 0u), rn = xn;
    auto load = [&](int c) {
        if (c < d) {
            xn = __ldcg(reinterpret_cast<const uint4 *>(xrow + c));
            if (rrow) rn = __ldcg(reinterpret_cast<const uint4 *>(rrow + c));
        }
    };
    load(8 * lane);
    for (int base = 0; base < d; base += 256) {
        const int c0 = base + 8 * lane;
        const bool act = c0 < d;
        const uint32_t xw[4] = {xn.x, xn.y, xn.z, xn.w};
        uint32_t rw[4] = {rn.x, rn.y, rn.z, rn.w};      // zero without a reference
        load(c0 + 256);
        const uint32_t cf = act ? coef[c0 >> coef_shift] : 0u;
        if (rrow && gain && act) {
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int c = c0 + 2 * i;
                rw[i] = f2_to_bf16x2(__fmaf_rn(half_bits_to_float(gain[c]), __uint_as_float(rw[i] << 16), half_bits_to_float(bias[c])),
                                     __fmaf_rn(half_bits_to_float(gain[c + 1]), __uint_as_float(rw[i] & 0xffff0000u),
                                               half_bits_to_float(bias[c + 1])));
            }
        }
        const float ca = half_bits_to_float(cf & 0xffff), cb = half_bits_to_float(cf >> 16);
        const u64 a2 = pack2(ca, ca), b2 = pack2(cb, cb);
        float e[8], rt[8];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const u64 rt2 = pfma(a2, bf16x2_to_p(rw[i]), b2);
            unpack2(rt2, rt[2 * i], rt[2 * i + 1]);
            unpack2(psub(bf16x2_to_p(xw[i]), rt2), e[2 * i], e[2 * i + 1]);
        }
        uint32_t left = act ? 0xffu : 0u;      // elements not taken yet
        while (true) {
            int best = -1, at = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const int mag = (int)(__float_as_uint(e[i]) & 0x7fffffffu);
                if (((left >> i) & 1u) && mag > best) { best = mag; at = i; }
            }
            const int top = __reduce_max_sync(0xffffffffu, best);
            const int low = __reduce_min_sync(0xffffffffu, held);
            if (top <= low) break;
            const int from = __ffs(__ballot_sync(0xffffffffu, best == top)) - 1;      // the lowest channel of them
            const int worst = __reduce_max_sync(0xffffffffu, held == low ? hc : -1);  // the highest channel of the smallest held
            const int tc = __shfl_sync(0xffffffffu, c0 + at, from);
            const float te = __shfl_sync(0xffffffffu, pick8(e, at), from), trt = __shfl_sync(0xffffffffu, pick8(rt, at), from);
            if (lane == from) left &= ~(1u << at);
            if (held == low && hc == worst) { held = top; hc = tc; he = te; hrt = trt; }
        }
    }
    return Winner{hc, he, hrt};
}

// NV: slab maxima per lane (d <= 32*32*NV).  KT: the number of outliers when it is 8 (unrolled), else 0 = p.topk.
// bits: code width (only the clearing of the codes depends on it).  A warp works on kOutPair tokens at a time, phase
// by phase, so that their trips to memory (scattered 32-byte reads of X, the reference row and the record, which
// bound this pass) overlap.
constexpr int kOutPair = 2;

// W: warps per CTA.  7 = four CTAs of 72 registers per SM (56 tokens in flight), 8 = three CTAs of 80 registers (48 tokens); see
// launch_encode.
template <int NV, int KT, bool SUB, int W>
__global__ void __launch_bounds__(W * 32, W == 7 ? 4 : 3) outlier_kernel(const CodecParams p, const int bits) {
    constexpr int U = kOutPair;
    __shared__ float s_e[W][U][kOutCap];
    __shared__ float s_rt[W][U][kOutCap];
    __shared__ unsigned short s_c[W][U][kOutCap];
    __shared__ unsigned char s_hot[W][U][32 * NV];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int d = p.d, nth = d >> 5;
    const int k = KT ? KT : p.topk;
    const uint32_t cmask = (1u << bits) - 1u;
    const long long tstride = (long long)gridDim.x * W * U;
    const unsigned int lt_mask = (1u << lane) - 1u;
    const int tm_stride = (nth + 3) & ~3;       // rows of slab maxima are padded to 16 bytes
    const bool want_xhat = p.X_hat != nullptr;
    const int my0 = NV * lane;                  // first slab of this lane
    const int my_n = min(NV, max(0, nth - my0));  // how many of its NV slabs exist
    const int coef_shift = 5 + p.lpg_shift;
    bool shared = false;   // coefficient words per segment, outside the records
    if constexpr (SUB) shared = p.coef_ext != nullptr;
    const int coff = shared ? 0 : 4 * p.J;
    // everything this kernel reads was written by the streaming pass launched just before it
    if (p.T <= gridDim.x * W * U) grid_launch_dependents();
    grid_dependency_wait();
    const long long n_tok = tokens_to_do<SUB>(p);

    for (long long ti0 = ((long long)blockIdx.x * W + warp) * U; ti0 < n_tok; ti0 += tstride) {
        long long t[U];
        const uint16_t *xrow[U], *rrow[U];
        const uint32_t *coefp[U];
        unsigned char *rec[U];
        unsigned int tau[U];
        int nh[U], n[U];
        bool live[U];
        // ---- (a) slab maxima, threshold, and the slabs that reach it, in slab order
#pragma unroll
        for (int u = 0; u < U; u++) {
            live[u] = ti0 + u < n_tok;
            t[u] = live[u] ? token_at<SUB>(p, ti0 + u) : 0;
            unsigned int tv[NV];
            {
                const float *tm = p.tmax + t[u] * tm_stride + my0;
                const int lim = live[u] ? my_n : 0;
                if (NV % 4 == 0) {
#pragma unroll
                    for (int j = 0; j < NV / 4; j++) {
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        if (4 * j < lim) v = __ldg(reinterpret_cast<const uint4 *>(tm) + j);   // rows are padded to 16 bytes
                        tv[4 * j + 0] = 4 * j + 0 < lim ? v.x : 0u;
                        tv[4 * j + 1] = 4 * j + 1 < lim ? v.y : 0u;
                        tv[4 * j + 2] = 4 * j + 2 < lim ? v.z : 0u;
                        tv[4 * j + 3] = 4 * j + 3 < lim ? v.w : 0u;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < NV; i++) tv[i] = i < lim ? __float_as_uint(__ldg(tm + i)) : 0u;
                }
            }
            // reference row of the token, by the same rules as the streaming pass (which already reported bad rows)
            const int row = live[u] ? resolve_row<SUB>(p, p.ref_row ? p.ref_row[t[u]] : (int)t[u], false) : -1;
            xrow[u] = p.X + t[u] * d;
            rrow[u] = row >= 0 ? ref_row_ptr<SUB>(p, row) : nullptr;
            rec[u] = p.payload + t[u] * p.rec;
            coefp[u] = reinterpret_cast<const uint32_t *>(rec[u]);
            if constexpr (SUB)
                if (shared) coefp[u] = p.coef_ext + (long long)(live[u] ? p.seg_of[t[u]] : 0) * p.J;
            // threshold.  Bit patterns of non-negative floats order like integers.
            unsigned int m1 = tv[0], m2 = 0u;
#pragma unroll
            for (int i = 1; i < NV; i++) {
                m2 = max(m2, min(m1, tv[i]));
                m1 = max(m1, tv[i]);
            }
#pragma unroll
            for (int r = 1; r < k; r++) {
                const unsigned int top = __reduce_max_sync(0xffffffffu, m1);
                const unsigned int bal = __ballot_sync(0xffffffffu, m1 == top);
                const bool pop = m1 == top && (bal & lt_mask) == 0u;
                m1 = pop ? m2 : m1;
                m2 = pop ? 0u : m2;
            }
            tau[u] = __reduce_max_sync(0xffffffffu, m1);
            // tau == 0: fewer than k slabs hold anything but zeros, every element is a candidate: whole-token path
            nh[u] = 0;
            n[u] = live[u] ? kOutCap + 1 : 0;
            if (tau[u] != 0u) {
                unsigned int hm = 0u;
#pragma unroll
                for (int i = 0; i < NV; i++) hm |= (tv[i] >= tau[u]) ? (1u << i) : 0u;
                int incl = __popc(hm);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, incl, o);
                    incl += lane >= o ? up : 0;
                }
                nh[u] = __shfl_sync(0xffffffffu, incl, 31);
                int at = incl - __popc(hm);
                while (hm) {
                    s_hot[warp][u][at++] = (unsigned char)(my0 + __ffs(hm) - 1);
                    hm &= hm - 1u;
                }
                n[u] = 0;
            }
        }
        __syncwarp();
        // ---- (b) candidates: eight slabs per round, four lanes per slab, eight channels per lane.  The first
        // round of every token is loaded before any of them is used.
        auto load_round = [&](int u, int base, int &c0, bool &act, uint4 &xw, uint4 &rw, uint32_t &cf) {
            const int hi = base + (lane >> 2);
            act = hi < nh[u];
            c0 = act ? (int)s_hot[warp][u][hi] * 32 + (lane & 3) * 8 : 0;
            xw = make_uint4(0u, 0u, 0u, 0u);
            rw = xw;
            cf = 0u;
            if (act) {
                xw = __ldg(reinterpret_cast<const uint4 *>(xrow[u] + c0));
                if (rrow[u]) rw = __ldg(reinterpret_cast<const uint4 *>(rrow[u] + c0));
                cf = coefp[u][c0 >> coef_shift];
            }
        };
        auto use_round = [&](int u, int c0, bool act, const uint4 &xw, const uint4 &rw, uint32_t cf) {
            const uint32_t xs[4] = {xw.x, xw.y, xw.z, xw.w};
            const uint32_t rs[4] = {rw.x, rw.y, rw.z, rw.w};
            const float ca = half_bits_to_float(cf & 0xffff), cb = half_bits_to_float(cf >> 16);
            float e[8], rt[8];
            if (rrow[u] && p.gain) {
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    const uint32_t xb = (i & 1) ? (xs[i >> 1] & 0xffff0000u) : (xs[i >> 1] << 16);
                    const uint32_t rb = (i & 1) ? (rs[i >> 1] & 0xffff0000u) : (rs[i >> 1] << 16);
                    const float r = bf16_round(__fmaf_rn(half_bits_to_float(p.gain[c0 + i]), __uint_as_float(rb),
                                                         half_bits_to_float(p.bias[c0 + i])));
                    rt[i] = __fmaf_rn(ca, r, cb);
                    e[i] = __fsub_rn(__uint_as_float(xb), rt[i]);
                }
            } else {
                // without a reference rw is zero, which is the zero reference of a directly coded token
                const u64 a2 = pack2(ca, ca), b2 = pack2(cb, cb);
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const u64 rt2 = pfma(a2, bf16x2_to_p(rs[i]), b2);
                    unpack2(rt2, rt[2 * i], rt[2 * i + 1]);
                    unpack2(psub(bf16x2_to_p(xs[i]), rt2), e[2 * i], e[2 * i + 1]);
                }
            }
            // which of the lane's eight elements reach the threshold (tau > 0 here; for finite values the
            // comparison of magnitudes is the comparison of their bit patterns)
            const float tauf = __uint_as_float(tau[u]);
            uint32_t m = 0u;
#pragma unroll
            for (int i = 0; i < 8; i++) m |= (fabsf(e[i]) >= tauf) ? (1u << i) : 0u;
            if (!act) m = 0u;
            const int cnt = __popc(m);
            // position of the lane's first candidate (candidates come out in channel order).  Almost always no
            // lane has two, and a ballot does; otherwise a prefix sum over the lanes.
            int pos, total;
            if (!__any_sync(0xffffffffu, cnt > 1)) {
                const unsigned int bal = __ballot_sync(0xffffffffu, cnt != 0);
                pos = n[u] + __popc(bal & lt_mask);
                total = __popc(bal);
            } else {
                int inc2 = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int up = __shfl_up_sync(0xffffffffu, inc2, o);
                    inc2 += lane >= o ? up : 0;
                }
                pos = n[u] + inc2 - cnt;
                total = __shfl_sync(0xffffffffu, inc2, 31);
            }
            while (m) {
                const int i = __ffs(m) - 1;
                m &= m - 1u;
                if (pos < kOutCap) {
                    s_e[warp][u][pos] = pick8(e, i);
                    s_c[warp][u][pos] = (unsigned short)(c0 + i);
                    if (want_xhat) s_rt[warp][u][pos] = pick8(rt, i);
                }
                pos++;
            }
            n[u] += total;
        };
        {
            int c0[U];
            bool act[U];
            uint4 xw[U], rw[U];
            uint32_t cf[U];
#pragma unroll
            for (int u = 0; u < U; u++) load_round(u, 0, c0[u], act[u], xw[u], rw[u], cf[u]);
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (nh[u] > 0) use_round(u, c0[u], act[u], xw[u], rw[u], cf[u]);
                for (int base = 8; base < nh[u] && n[u] <= kOutCap; base += 8) {
                    load_round(u, base, c0[u], act[u], xw[u], rw[u], cf[u]);
                    use_round(u, c0[u], act[u], xw[u], rw[u], cf[u]);
                }
            }
        }
        __syncwarp();
        // ---- (c) one candidate per lane, in channel order; while there are too many the smallest goes
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!live[u]) continue;
            bool won;
            int wc = 0;
            float we = 0.f, wrt = 0.f;
            if (n[u] <= kOutCap) {
                won = lane < n[u];
                if (won) {
                    wc = s_c[warp][u][lane];
                    we = s_e[warp][u][lane];
                    if (want_xhat) wrt = s_rt[warp][u][lane];
                }
                unsigned int mag = won ? (__float_as_uint(we) & 0x7fffffffu) : 0xffffffffu;
                for (int extra = n[u] - k; extra > 0; extra--) {
                    const unsigned int low = __reduce_min_sync(0xffffffffu, mag);
                    const unsigned int bal = __ballot_sync(0xffffffffu, mag == low);
                    if (lane == 31 - __clz(bal)) { mag = 0xffffffffu; won = false; }   // among equals the highest channel
                }
            } else {
                const Winner w = select_whole_token(d, k, coef_shift, xrow[u], rrow[u], p.gain, p.bias, coefp[u], lane);
                wc = w.c;
                we = w.e;
                wrt = w.rt;
                won = lane < k;
            }
            // ---- (d) outlier fields in channel order, dense codes at those channels cleared
            int pos = __popc(__ballot_sync(0xffffffffu, won) & lt_mask);
            if (n[u] > kOutCap) {   // the whole-token path returns its winners in no order
                pos = 0;
                for (int y = 0; y < k; y++) {
                    const int cy = __shfl_sync(0xffffffffu, wc, y);
                    pos += cy < wc ? 1 : 0;
                }
            }
            if (won) {
                unsigned short *oidx = reinterpret_cast<unsigned short *>(rec[u] + coff + p.code_bytes);
                const uint32_t hv = float_to_half_bits_sat(we);
                oidx[pos] = (unsigned short)wc;
                oidx[k + pos] = (unsigned short)hv;
                // the sender-side reconstruction of an outlier channel: (alpha*r + beta) + the binary16 value
                if (want_xhat)
                    p.X_hat[t[u] * d + wc] = __bfloat16_as_ushort(__float2bfloat16_rn(__fadd_rn(wrt, half_bits_to_float(hv))));
                uint32_t *codes32 = reinterpret_cast<uint32_t *>(rec[u] + coff);
                const int bit = wc * bits, wd = bit >> 5, sh = bit & 31;
                atomicAnd(&codes32[wd], ~(cmask << sh));
                if (sh + bits > 32) atomicAnd(&codes32[wd + 1], ~(cmask >> (32 - sh)));
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------------
// encode with outliers in one launch
// ------------------------------------------------------------------------------------------------
// The streaming pass with NSEL further warps per CTA, the selectors.  A selector takes every NSEL-th token: when the streaming
// warps have finished it, it refills the stage at once (two stages), finds the k largest |e| from the slab maxima by the steps
// of outlier_kernel -- the rows of the few slabs that hold them are read again, from L2, where they passed microseconds ago --,
// patches the record in shared memory and sends it off.  Nothing goes through DRAM twice, and there is
// no second launch.  A token's selection is a chain of ~3000 cycles; NSEL of them
// run beside the streaming warps of NSEL later tokens, so records live in four slots (token mod 4), with a barrier each for
// "all streaming warps are done" and "the record has left".
// The row reads bypass L1, which holds the step table.  Shapes by width (streaming warps + selectors, CTAs per SM): measured at
// 131072 x 5120 3 CTAs of 5 + 3 warps 0.537 ms, 3 of 5 + 2 0.570, 4 of 5 + 2 0.589 to 0.649, 4 of 5 + 3 0.611 (two launches
// 0.601); at 16384 x 4096 4 CTAs of 4 + 2 66 us, 4 of 4 + 3 68, 5 of 4 + 2 72 (two launches 81).  Reading the slabs from the
// stage and refilling it afterwards was slower in every shape.  With x_hat the CTAs keep two selectors and the registers that
// three of them per SM leave; see one_launch for where that form is the better one.
//
// Teams: with x_hat a token needs the inverse steps and the steps, in calls with direct tokens two rows of each, and several CTAs
// per SM each with their stages leave them too little L1.  So in calls of many tokens an SM runs ONE CTA of several teams, each
// of which is what is a CTA otherwise (its streaming and selector warps, stages and barriers), and all of them read one copy of the tables in
// shared memory (SlabTables).  131072 x 5120, 28 % direct tokens, in long runs: 828 us against 966 with a CTA per token and 899 in two
// launches; 65536 x 4096 305 against 348 with a CTA per token, x 3072 238 against 269, 16000 x 6144 123 against 139 in two launches; long
// uplink with retrieval 944 -> 856.  The registers spill a little at five streaming and three selector warps (80 of them, 32 bytes); two
// selectors at 96 registers do not and take 852 us, since a token's selection is the longer chain.  (Four teams with fewer registers
// at 4096 channels 437 against 439 us, and spills.)  Teams without x_hat (one row in L1 is no trouble there) 574 against 568.
struct TopCtrl {
    unsigned long long full[2];     // data of the stage has landed
    unsigned long long done[4];     // every streaming warp has finished token (mod 4)
    unsigned long long left[4];     // the record in slot (token mod 4) has been read by the copy engine
    int row[2];
    int abort;
};
constexpr int kHotCap = 64;        // slabs looked at; more (many maxima tie): the whole token
constexpr int kPatchWords = 64;    // outliers of x_hat rows that have left, per selector
template <int NSEL, bool XHAT>
struct TopSel {
    float e[NSEL][kOutCap];
    unsigned short c[NSEL][kOutCap];
    unsigned char hot[NSEL][kHotCap];
    float rt[XHAT ? NSEL : 1][XHAT ? kOutCap : 1];
    uint32_t patch[XHAT ? NSEL : 1][XHAT ? kPatchWords : 1];
};
struct TopSmem {
    int stage0, stage_bytes, rec_off, tm_off, sel0, total;
};
__host__ __device__ inline TopSmem top_smem_layout(int d, int rec, int sel_bytes) {
    TopSmem s;
    s.stage0 = align_up((int)sizeof(TopCtrl), 128);
    s.rec_off = 4 * d;                        // behind X row and R row: two record slots
    s.tm_off = s.rec_off + 2 * rec;           // slab maxima (read before the stage is refilled)
    s.stage_bytes = align_up(s.tm_off + d / 8, 128);
    s.sel0 = s.stage0 + 2 * s.stage_bytes;
    s.total = s.sel0 + sel_bytes;
    return s;
}

// NV: slab maxima per lane (d <= 1024 * NV).  KT: the number of outliers when it is 8, else 0 = p.topk.  LPG, D, REF: as for
// encode_ws_kernel.  TEAMS > 1: tables in shared memory; no gain and bias (they would be read past an L1 that is not there).
template <int BITS, int KT, bool XHAT, int NV, int NSEL, int MAXT, int MINB, int LPG, int D = 0, bool REF = false, int TEAMS = 1>
__global__ void __launch_bounds__(MAXT, MINB) encode_top_kernel(const CodecParams p) {
    extern __shared__ __align__(128) unsigned char smem_all[];
    // everything below is about this thread's team
    const int nt = TEAMS == 1 ? blockDim.x : blockDim.x / TEAMS, team = TEAMS == 1 ? 0 : threadIdx.x / nt;
    const int tid = TEAMS == 1 ? threadIdx.x : threadIdx.x - team * nt;
    const int lane = tid & 31, warp = tid >> 5, nstream = D ? (D / 32 + 31) / 32 : (nt >> 5) - NSEL;
    const int rot = (lane >> 1) & 3;
    const int d = D ? D : p.d;
    constexpr bool kGeo = D != 0 && LPG != 0 && KT == 8;
    const int Jc = kGeo ? D / (32 * (LPG ? LPG : 1)) : p.J;
    const int codeb = kGeo ? D * BITS / 8 : p.code_bytes;
    const int recb = kGeo ? (4 * (D / (32 * (LPG ? LPG : 1))) + D * BITS / 8 + 32 + 15) / 16 * 16 : p.rec;
    const int coff = 4 * Jc;
    const TopSmem L = top_smem_layout(d, recb, (int)sizeof(TopSel<NSEL, XHAT>));
    unsigned char *smem = smem_all + (TEAMS == 1 ? 0 : team * align_up(L.total, 128));
    TopCtrl *ctrl = reinterpret_cast<TopCtrl *>(smem);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t row_bytes = 2u * (uint32_t)d;

    if (TEAMS == 1 && p.T <= gridDim.x) grid_launch_dependents();
    if (tid == 0) {
        for (int s = 0; s < 2; s++) mbar_init(smem_u32(&ctrl->full[s]), 1);
        for (int s = 0; s < 4; s++) {
            mbar_init(smem_u32(&ctrl->done[s]), nstream);
            mbar_init(smem_u32(&ctrl->left[s]), 1);
        }
        ctrl->abort = 0;
        mbar_init_fence();
    }
    {
        // padding words of the records are written once and never touched again
        const int raw = coff + codeb + 4 * p.topk;
        for (int s = 0; s < 4; s++)
            for (int o = raw + 4 * tid; o < recb; o += 4 * nt)
                *reinterpret_cast<uint32_t *>(smem + L.stage0 + (s >> 1) * L.stage_bytes + L.rec_off + (s & 1) * recb + o) = 0u;
    }
    __syncthreads();
    grid_dependency_wait();
    SlabTables tab;
    bool half_steps = true;
    if constexpr (TEAMS > 1) {
        const bool mine = warp < nstream && tid * 32 < d;
        const uint32_t t0 = smem_u32(smem_all) + TEAMS * align_up(L.total, 128);
        tab.pitch = (uint32_t)nstream * 512u;
        tab.inv = t0 + tid * 16u;
        tab.step = tab.inv + 16u * tab.pitch;
        // row r, slot j of both tables by team (4r + j) mod TEAMS
        for (int q = team; mine && q < 8; q += TEAMS) {
            const int r = q >> 2, j = q & 3, c = r * d + tid * 32 + ((j + rot) & 3) * 8;
            const uint4 i0 = __ldg(reinterpret_cast<const uint4 *>(p.inv_step + c)), i1 = __ldg(reinterpret_cast<const uint4 *>(p.inv_step + c + 4));
            sts128(tab.inv + (8 * r + 2 * j) * tab.pitch, i0);
            sts128(tab.inv + (8 * r + 2 * j + 1) * tab.pitch, i1);
            const float4 s0 = __ldg(reinterpret_cast<const float4 *>(p.step + c)), s1 = __ldg(reinterpret_cast<const float4 *>(p.step + c + 4));
            const float v[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
            uint32_t hw[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
                const float2 back = __half22float2(h);
                half_steps = half_steps && back.x == v[2 * i] && back.y == v[2 * i + 1];
                hw[i] = *reinterpret_cast<const uint32_t *>(&h);
            }
            sts128(tab.step + (4 * r + j) * tab.pitch, make_uint4(hw[0], hw[1], hw[2], hw[3]));
        }
        half_steps = __syncthreads_and(half_steps) != 0;
        if (!half_steps) {      // calibrated tables are binary16 values, a caller's own need not be
            tab.step = tab.inv + 8u * tab.pitch;
            for (int q = team; mine && q < 8; q += TEAMS) {
                const int r = q >> 2, j = q & 3, c = r * d + tid * 32 + ((j + rot) & 3) * 8;
                sts128(tab.step + (8 * r + 2 * j) * tab.pitch, __ldg(reinterpret_cast<const uint4 *>(p.step + c)));
                sts128(tab.step + (8 * r + 2 * j + 1) * tab.pitch, __ldg(reinterpret_cast<const uint4 *>(p.step + c + 4)));
            }
            __syncthreads();
        }
    }
    const int first = blockIdx.x + gridDim.x * team, stride = gridDim.x * TEAMS;
    const int n_my = p.T > first ? (int)((p.T - first + stride - 1) / stride) : 0;
    auto token = [&](int k) -> long long { return first + (long long)k * stride; };   // this CTA's k-th token
    auto raw_row_of = [&](int k) -> int { return p.ref_row ? p.ref_row[token(k)] : (int)token(k); };
    // one lane: start the copies of this CTA's k-th token
    auto issue = [&](int k, int raw_row) {
        const int s = k & 1, row = resolve_row<false>(p, raw_row);
        ctrl->row[s] = row;
        const uint32_t bar = smem_u32(&ctrl->full[s]);
        const uint32_t base = sbase + L.stage0 + s * L.stage_bytes;
        mbar_arrive_expect_tx(bar, p.test_extra_tx + row_bytes + (row >= 0 ? row_bytes : 0u));
        bulk_load(base, p.X + token(k) * d, row_bytes, bar);
        if (row >= 0) bulk_load(base + row_bytes, p.ref_base + (long long)row * d, row_bytes, bar);
    };

    bool timed_out = false;
    if (warp < nstream) {
        // ---- streaming warps
        const bool valid = tid * 32 < d;
        uint32_t off[4];
#pragma unroll
        for (int j = 0; j < 4; j++) off[j] = (uint32_t)(tid * 64 + ((j + rot) & 3) * 16);
        const unsigned int group_mask = __ballot_sync(0xffffffffu, valid);
        const u64 no_steps[1] = {0ull};
        for (int it = 0; it < n_my; it++) {
            if (*reinterpret_cast<volatile int *>(&ctrl->abort)) break;
            const int stage = it & 1;
            const uint32_t parity = (it >> 1) & 1;
            unsigned char *stg = smem + L.stage0 + stage * L.stage_bytes;
            const uint32_t xs = sbase + L.stage0 + stage * L.stage_bytes;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->full[stage]), parity))) { timed_out = true; break; }
            const bool has_ref = REF ? true : ctrl->row[stage] >= 0;
            auto slab = [&](auto tables) {
                encode_slab<BITS, true, XHAT, LPG, false, decltype(tables)::value, TEAMS == 1 && NV <= 5>(
                    p, tid, lane, rot, d, Jc, false, coff, off, group_mask, xs, xs + row_bytes, has_ref, 0, stg + L.rec_off + parity * recb,
                    reinterpret_cast<float *>(stg + L.tm_off), no_steps, tab);
            };
            if (valid) {
                if (TEAMS > 1 && !half_steps) slab(std::integral_constant<int, TEAMS == 1 ? 0 : 2>{});
                else slab(std::integral_constant<int, TEAMS == 1 ? 0 : 1>{});
            }
            fence_async_smem();     // the record bytes written above will be read by the copy engine
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&ctrl->done[it & 3])) : "memory");
        }
    } else {
        // ---- selectors
        const int sel = warp - nstream;
        const int nth = d >> 5, k = KT ? KT : p.topk;
        TopSel<NSEL, XHAT> *sc = reinterpret_cast<TopSel<NSEL, XHAT> *>(smem + L.sel0);
        float *s_e = sc->e[sel];
        unsigned short *s_c = sc->c[sel];
        unsigned char *s_hot = sc->hot[sel];
        // x_hat rows leave as bulk stores before their outliers are known.  The outliers wait here until the rows are in place:
        // one wait for the stores of several tokens (a wait per token cost 0.2 ms at 131072 x 5120)
        float *s_rt = sc->rt[XHAT ? sel : 0];
        uint32_t *s_patch = sc->patch[XHAT ? sel : 0];
        int n_patch = 0, it_patch = sel;        // tokens that wait, and the first of them
        auto flush_patches = [&]() {
            if (lane == 0) bulk_wait_all();
            __syncwarp();
            for (int q = lane; q < n_patch * k; q += 32) {
                const uint32_t w = s_patch[q];
                p.X_hat[token(it_patch + (q / k) * NSEL) * d + (w & 0xffffu)] = (uint16_t)(w >> 16);
            }
            __syncwarp();
            it_patch += n_patch * NSEL;
            n_patch = 0;
        };
        const unsigned int lt_mask = (1u << lane) - 1u;
        constexpr uint32_t cmask = (1u << BITS) - 1u;
        const int coef_shift = 5 + (LPG ? (LPG == 4 ? 2 : 1) : p.lpg_shift);
        if (sel == 0 && lane == 0)
            for (int q = 0; q < 2 && q < n_my; q++) issue(q, raw_row_of(q));
        for (int it = sel; it < n_my; it += NSEL) {
            if (*reinterpret_cast<volatile int *>(&ctrl->abort)) break;
            const int s = it & 1, next = it + 2;
            unsigned char *stg = smem + L.stage0 + s * L.stage_bytes;
            unsigned char *rec = stg + L.rec_off + ((it >> 1) & 1) * recb;
            const long long t = token(it);
            int raw_next = 0;
            if (lane == 0 && next < n_my) raw_next = raw_row_of(next);
            if (XHAT && (n_patch + 1) * k > kPatchWords) flush_patches();
            if (lane == 0 && it >= NSEL) {      // this selector's last record
                bulk_wait_read<0>();
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&ctrl->left[(it - NSEL) & 3])) : "memory");
            }
            // (a parity tells neighbouring phases apart only: this barrier's last token, it - 4, is done, since the streaming
            // warps go through the tokens in order and this selector's last one was it - NSEL >= it - 4)
            static_assert(NSEL <= 4, "one phase at a time");
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->done[it & 3]), (it >> 2) & 1))) { timed_out = true; break; }
            const int row = ctrl->row[s];
            unsigned int tv[NV];                // maxima of slabs 32 * i + lane: bit patterns of non-negative floats order like integers
#pragma unroll
            for (int i = 0; i < NV; i++)
                tv[i] = 32 * i + lane < nth ? *reinterpret_cast<volatile unsigned int *>(stg + L.tm_off + (32 * i + lane) * 4) : 0u;
            __syncwarp();
            if (XHAT && lane == 0) {            // the X row carries x_hat now and must have been read before the refill
                bulk_store(p.X_hat + t * d, sbase + L.stage0 + s * L.stage_bytes, row_bytes);
                bulk_commit();
                bulk_wait_read<0>();
            }
            if (next < n_my) {
                // the next token of this stage writes the record slot of token it - 2
                if (it >= 2 && !__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->left[next & 3]), ((next >> 2) - 1) & 1))) {
                    timed_out = true;
                    break;
                }
                if (lane == 0) issue(next, raw_next);
            }
            // ---- threshold and the slabs that reach it, in slab order (see outlier_kernel)
            unsigned int m1 = tv[0], m2 = 0u;
#pragma unroll
            for (int i = 1; i < NV; i++) {
                m2 = max(m2, min(m1, tv[i]));
                m1 = max(m1, tv[i]);
            }
#pragma unroll
            for (int r = 1; r < k; r++) {
                const unsigned int top = __reduce_max_sync(0xffffffffu, m1);
                const unsigned int bal = __ballot_sync(0xffffffffu, m1 == top);
                const bool pop = m1 == top && (bal & lt_mask) == 0u;
                m1 = pop ? m2 : m1;
                m2 = pop ? 0u : m2;
            }
            const unsigned int tau = __reduce_max_sync(0xffffffffu, m1);
            const float tauf = __uint_as_float(tau);
            // tau == 0: fewer than k slabs hold anything but zeros, every element is a candidate: whole-token path
            int nh = 0, n = kOutCap + 1;
            if (tau != 0u) {
#pragma unroll
                for (int i = 0; i < NV; i++) {
                    const bool hit = tv[i] >= tau;
                    const unsigned int bal = __ballot_sync(0xffffffffu, hit);
                    const int at = nh + __popc(bal & lt_mask);
                    if (hit && at < kHotCap) s_hot[at] = (unsigned char)(32 * i + lane);
                    nh += __popc(bal);
                }
                n = nh <= kHotCap ? 0 : kOutCap + 1;
            }
            __syncwarp();
            // ---- candidates: eight slabs per round, four lanes per slab, eight channels per lane
            const uint16_t *xrow = p.X + t * d, *rrow = row >= 0 ? p.ref_base + (long long)row * d : nullptr;
            const uint32_t *coefp = reinterpret_cast<const uint32_t *>(rec);
            for (int base = 0; base < nh && n <= kOutCap; base += 8) {
                const int hi = base + (lane >> 2);
                const bool act = hi < nh;
                const int c0 = act ? (int)s_hot[hi] * 32 + (lane & 3) * 8 : 0;
                uint4 xv = make_uint4(0u, 0u, 0u, 0u), rv = xv;
                uint32_t cf = 0u;
                if (act) {
                    xv = __ldcg(reinterpret_cast<const uint4 *>(xrow + c0));
                    if (rrow) rv = __ldcg(reinterpret_cast<const uint4 *>(rrow + c0));
                    cf = coefp[c0 >> coef_shift];
                }
                const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
                uint32_t rw[4] = {rv.x, rv.y, rv.z, rv.w};      // zero without a reference, as in the streaming warps
                if (rrow && p.gain) {
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const int c = c0 + 2 * i;
                        rw[i] = f2_to_bf16x2(__fmaf_rn(half_bits_to_float(p.gain[c]), __uint_as_float(rw[i] << 16), half_bits_to_float(p.bias[c])),
                                             __fmaf_rn(half_bits_to_float(p.gain[c + 1]), __uint_as_float(rw[i] & 0xffff0000u),
                                                       half_bits_to_float(p.bias[c + 1])));
                    }
                }
                const float ca = half_bits_to_float(cf & 0xffff), cb = half_bits_to_float(cf >> 16);
                const u64 a2 = pack2(ca, ca), b2 = pack2(cb, cb);
                float e[8], rt[8];
                uint32_t m = 0u;
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const u64 rt2 = pfma(a2, bf16x2_to_p(rw[i]), b2);
                    unpack2(rt2, rt[2 * i], rt[2 * i + 1]);
                    unpack2(sub_pair(xw[i], rt2), e[2 * i], e[2 * i + 1]);
                    m |= (fabsf(e[2 * i]) >= tauf ? 1u : 0u) << (2 * i) | (fabsf(e[2 * i + 1]) >= tauf ? 2u : 0u) << (2 * i);
                }
                if (!act) m = 0u;
                const int cnt = __popc(m);
                // position of the lane's first candidate (candidates come out in channel order).  Almost always no lane has two.
                int pos, total;
                if (!__any_sync(0xffffffffu, cnt > 1)) {
                    const unsigned int bal = __ballot_sync(0xffffffffu, cnt != 0);
                    pos = n + __popc(bal & lt_mask);
                    total = __popc(bal);
                } else {
                    int incl = cnt;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int up = __shfl_up_sync(0xffffffffu, incl, o);
                        incl += lane >= o ? up : 0;
                    }
                    pos = n + incl - cnt;
                    total = __shfl_sync(0xffffffffu, incl, 31);
                }
                while (m) {
                    const int i = __ffs(m) - 1;
                    m &= m - 1u;
                    if (pos < kOutCap) {
                        s_e[pos] = pick8(e, i);
                        s_c[pos] = (unsigned short)(c0 + i);
                        if (XHAT) s_rt[pos] = pick8(rt, i);
                    }
                    pos++;
                }
                n += total;
            }
            __syncwarp();
            // ---- one candidate per lane, in channel order; while there are too many the smallest goes
            bool won;
            int wc = 0, pos;
            float we = 0.f, wrt = 0.f;
            if (n <= kOutCap) {
                won = lane < n;
                if (won) {
                    wc = s_c[lane];
                    we = s_e[lane];
                    if (XHAT) wrt = s_rt[lane];
                }
                unsigned int mag = won ? (__float_as_uint(we) & 0x7fffffffu) : 0xffffffffu;
                for (int extra = n - k; extra > 0; extra--) {
                    const unsigned int low = __reduce_min_sync(0xffffffffu, mag);
                    const unsigned int bal = __ballot_sync(0xffffffffu, mag == low);
                    if (lane == 31 - __clz(bal)) { mag = 0xffffffffu; won = false; }   // among equals the highest channel
                }
                pos = __popc(__ballot_sync(0xffffffffu, won) & lt_mask);
            } else {
                const Winner w = select_whole_token(d, k, coef_shift, xrow, rrow, p.gain, p.bias, coefp, lane);
                wc = w.c;
                we = w.e;
                wrt = w.rt;
                won = lane < k;
                pos = 0;                         // the whole-token path returns its winners in no order
                for (int y = 0; y < k; y++) {
                    const int cy = __shfl_sync(0xffffffffu, wc, y);
                    pos += cy < wc ? 1 : 0;
                }
            }
            // ---- outlier fields in channel order, dense codes at those channels cleared
            if (won) {
                unsigned short *oidx = reinterpret_cast<unsigned short *>(rec + coff + codeb);
                oidx[pos] = (unsigned short)wc;
                const uint32_t hv = float_to_half_bits_sat(we);
                oidx[k + pos] = (unsigned short)hv;
                // the sender-side reconstruction of an outlier channel: (alpha*r + beta) + the binary16 value
                if (XHAT) {
                    const uint16_t xh = __bfloat16_as_ushort(__float2bfloat16_rn(__fadd_rn(wrt, half_bits_to_float(hv))));
                    s_patch[n_patch * k + pos] = (uint32_t)wc | (uint32_t)xh << 16;
                }
                uint32_t *codes32 = reinterpret_cast<uint32_t *>(rec + coff);
                const int bit = wc * BITS, wd = bit >> 5, sh = bit & 31;
                atomicAnd(&codes32[wd], ~(cmask << sh));
                if (BITS == 3 && sh + BITS > 32) atomicAnd(&codes32[wd + 1], ~(cmask >> (32 - sh)));
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                bulk_store(p.payload + t * recb, smem_u32(rec), (uint32_t)recb);
                bulk_commit();
            }
            n_patch++;
        }
        if (XHAT) flush_patches();
    }
    if (timed_out) {
        ctrl->abort = 1;
        if (p.status) atomicOr(p.status, RAC_STATUS_TIMEOUT);
    }
    __syncthreads();
    if (lane == 0) bulk_wait_all();  // every lane that stored records waits for its own copies
    if (tid == 0 && *reinterpret_cast<volatile int *>(&ctrl->abort)) {
        // give copies that may still be in flight a bounded chance to land before the CTA retires
        for (int s = 0; s < 2; s++) {
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 0);
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 1);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// reconstruct (receiver and sender)
// ------------------------------------------------------------------------------------------------
// Per token: record and reference row arrive in a stage; every thread dequantises its 32 channels
// (code -> binary32 through the 2^23 trick, times the step), adds the aligned reference, rounds to bf16
// into an output row in shared memory, patches the outliers it owns, and the row leaves as one bulk store.
// The step table row of referenced tokens lives in registers for the whole kernel (a thread always owns
// the same channels); direct tokens read row 1 through L1.
template <int BITS, int KT, bool SUB>
__global__ void __launch_bounds__(256) decode_kernel(const CodecParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int rot = (lane >> 1) & 3;
    const int d = p.d;
    const bool valid = tid * 32 < d;
    const DecSmem L = dec_smem_layout(d, p.rec, p.stages);
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(smem);
    const uint32_t sbase = smem_u32(smem);
    const int S = p.stages;
    constexpr uint32_t cmask = (1u << BITS) - 1u;
    constexpr uint32_t H = 1u << (BITS - 1);
    // 1 in every one of the 8 fields of a code word, and H in every field
    constexpr uint32_t ones = (BITS == 4) ? 0x11111111u : (BITS == 3) ? 0x00249249u : 0x00005555u;
    constexpr uint32_t highs = ones << (BITS - 1);
    constexpr float kBase = 8388608.0f + (float)H;  // 2^23 + H
    const uint32_t row_bytes = 2u * (uint32_t)d;

    if (p.T <= gridDim.x) grid_launch_dependents();
    if (tid == 0) {
        for (int s = 0; s < S; s++) mbar_init(smem_u32(&ctrl->bar[s]), 1);
        mbar_init_fence();
    }
    __syncthreads();
    grid_dependency_wait();

    bool shared = false;   // coefficient words per segment, outside the records
    if constexpr (SUB) shared = p.coef_ext != nullptr;
    const int coff = shared ? 0 : 4 * p.J;
    const int first = blockIdx.x, stride = gridDim.x;
    const long long n_tok = tokens_to_do<SUB>(p);
    const int n_my = (n_tok > first) ? (int)((n_tok - first + stride - 1) / stride) : 0;

    int next_raw = 0;
    auto raw_row_of = [&](int k) -> int {
        long long t = token_at<SUB>(p, first + (long long)k * stride);
        return p.ref_row ? p.ref_row[t] : (int)t;
    };
    if (tid == 0) {
        for (int k = 0; k < S - 1 && k < n_my; k++) {
            long long t = token_at<SUB>(p, first + (long long)k * stride);
            issue_token_loads<SUB>(p, ctrl, sbase + L.stage0 + k * L.stage_bytes, L.rec_pad, k, resolve_row<SUB>(p, raw_row_of(k)),
                              p.payload + t * p.rec, (uint32_t)p.rec, t);
        }
        if (S - 1 < n_my) next_raw = raw_row_of(S - 1);
    }

    uint32_t off[4];
#pragma unroll
    for (int j = 0; j < 4; j++) off[j] = (uint32_t)(tid * 64 + ((j + rot) & 3) * 16);
    // step table, row 0, in slot order
    u64 st0[16];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
        if (valid) {
            s0 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1)));
            s1 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1) + 4));
        }
        st0[4 * j + 0] = pack2(s0.x, s0.y);
        st0[4 * j + 1] = pack2(s0.z, s0.w);
        st0[4 * j + 2] = pack2(s1.x, s1.y);
        st0[4 * j + 3] = pack2(s1.z, s1.w);
    }
    const u64 base2 = pack2(kBase, kBase);

    int stage = 0, obuf = 0, issue_stage = S - 1;
    bool aborted = false;
    uint32_t parity = 0;
    for (int it = 0; it < n_my; it++) {
        const long long t = token_at<SUB>(p, first + (long long)it * stride);
        if (tid == 0 && it + S - 1 < n_my) {
            const int k = it + S - 1;
            const long long tk = token_at<SUB>(p, first + (long long)k * stride);
            issue_token_loads<SUB>(p, ctrl, sbase + L.stage0 + issue_stage * L.stage_bytes, L.rec_pad, issue_stage,
                              resolve_row<SUB>(p, next_raw), p.payload + tk * p.rec, (uint32_t)p.rec, tk);
            if (k + 1 < n_my) next_raw = raw_row_of(k + 1);
        }
        const bool timed_out = !mbar_wait_bounded(smem_u32(&ctrl->bar[stage]), parity);
        if (timed_out && p.status) atomicOr(p.status, RAC_STATUS_TIMEOUT);
        const bool has_ref = ctrl->row[stage] >= 0;
        const unsigned char *rec = smem + L.stage0 + stage * L.stage_bytes;
        const uint32_t rs = sbase + L.stage0 + stage * L.stage_bytes + L.rec_pad;
        unsigned char *ob = smem + L.out0 + obuf * (int)row_bytes;
        const uint32_t obs = smem_u32(ob);

        if (valid) {
            uint32_t cf;
            if (shared) cf = p.coef_ext[(long long)ctrl->seg[stage] * p.J + (tid >> p.lpg_shift)];
            else cf = reinterpret_cast<const uint32_t *>(rec)[tid >> p.lpg_shift];
            const float a = half_bits_to_float(cf & 0xffff), b = half_bits_to_float(cf >> 16);
            const u64 a2 = pack2(a, a), b2 = pack2(b, b);
            // code words of the four pieces, in piece order, then rotated into slot order
            const uint32_t *cw = reinterpret_cast<const uint32_t *>(rec + coff) + tid * BITS;
            uint32_t words[4];
            if (BITS == 4) {
                words[0] = cw[0]; words[1] = cw[1]; words[2] = cw[2]; words[3] = cw[3];
            } else if (BITS == 3) {
                uint32_t w0 = cw[0], w1 = cw[1], w2 = cw[2];
                words[0] = w0 & 0xffffffu;
                words[1] = (w0 >> 24) | ((w1 & 0xffffu) << 8);
                words[2] = (w1 >> 16) | ((w2 & 0xffu) << 16);
                words[3] = w2 >> 8;
            } else {
                uint32_t w0 = cw[0], w1 = cw[1];
                words[0] = w0 & 0xffffu; words[1] = w0 >> 16; words[2] = w1 & 0xffffu; words[3] = w1 >> 16;
            }
            uint32_t reserved = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                uint32_t v = words[q] ^ highs;  // field == 0  <=>  code == -2^(BITS-1)
                reserved |= (v - ones) & ~v & highs;
                words[q] = v;                   // fields now hold code + H (offset binary)
            }
            if (reserved && p.status) atomicOr(p.status, RAC_STATUS_RESERVED_CODE);
            rot_left4(words, rot);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int c = (int)(off[j] >> 1);
                u64 r2[4], st2[4];
                if (has_ref) {
                    load_ref_slot(rs + off[j], p.gain, p.bias, c, r2);
#pragma unroll
                    for (int i = 0; i < 4; i++) st2[i] = st0[4 * j + i];
                } else {
                    const float4 s0 = __ldg(reinterpret_cast<const float4 *>(p.step + d + c));
                    const float4 s1 = __ldg(reinterpret_cast<const float4 *>(p.step + d + c + 4));
                    st2[0] = pack2(s0.x, s0.y); st2[1] = pack2(s0.z, s0.w); st2[2] = pack2(s1.x, s1.y); st2[3] = pack2(s1.z, s1.w);
#pragma unroll
                    for (int i = 0; i < 4; i++) r2[i] = 0ull;
                }
                const uint32_t w = words[j];
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    // exact integer -> binary32 without a convert: 2^23 + (code + H), minus (2^23 + H)
                    const float q0 = __uint_as_float(0x4b000000u | ((w >> (BITS * (2 * i))) & cmask));
                    const float q1 = __uint_as_float(0x4b000000u | ((w >> (BITS * (2 * i + 1))) & cmask));
                    float x0, x1;
                    unpack2(pfma(psub(pack2(q0, q1), base2), st2[i], pfma(a2, r2[i], b2)), x0, x1);
                    o[i] = f2_to_bf16x2(x0, x1);
                }
                sts128(obs + off[j], make_uint4(o[0], o[1], o[2], o[3]));
            }
            if (KT > 0) {
                // outliers whose channel this thread owns replace what the dense pass wrote
                const unsigned short *oidx = reinterpret_cast<const unsigned short *>(rec + coff + p.code_bytes);
                const unsigned short *oval = oidx + p.topk;
#pragma unroll
                for (int n = 0; n < KT; n++) {
                    if (n < p.topk) {
                        const int c = oidx[n];
                        if ((c >> 5) == tid) {
                            float r = 0.f;
                            if (has_ref) {
                                r = __uint_as_float((uint32_t)(*reinterpret_cast<const unsigned short *>(rec + L.rec_pad + 2 * c)) << 16);
                                if (p.gain) r = bf16_round(__fmaf_rn(half_bits_to_float(p.gain[c]), r, half_bits_to_float(p.bias[c])));
                            }
                            const float xh = __fadd_rn(__fmaf_rn(a, r, b), half_bits_to_float(oval[n]));
                            reinterpret_cast<unsigned short *>(ob)[c] = __bfloat16_as_ushort(__float2bfloat16_rn(xh));
                        }
                    }
                }
            }
        }
        if (KT > 0 && tid == 0) {
            const unsigned short *oidx = reinterpret_cast<const unsigned short *>(rec + coff + p.code_bytes);
            bool bad = false;
            for (int n = 0; n < p.topk; n++) bad |= oidx[n] >= d;
            if (bad && p.status) atomicOr(p.status, RAC_STATUS_OUTLIER_RANGE);
        }
        fence_async_smem();
        if (__syncthreads_or(timed_out)) { aborted = true; break; }  // one vote: every thread leaves together
        if (tid == 0) {
            bulk_store(p.X_hat + t * d, obs, row_bytes);
            bulk_commit();
            bulk_wait_read<1>();
        }
        if (++stage == S) { stage = 0; parity ^= 1u; }
        if (++issue_stage == S) issue_stage = 0;
        if (++obuf == kRecBufs) obuf = 0;
    }
    if (tid == 0) {
        bulk_wait_all();
        if (aborted) {
            for (int s = 0; s < S; s++) {
                mbar_wait_bounded(smem_u32(&ctrl->bar[s]), 0);
                mbar_wait_bounded(smem_u32(&ctrl->bar[s]), 1);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------
// reconstruct, streaming form: no CTA barrier in the loop
// ------------------------------------------------------------------------------------------------
// Same arithmetic as decode_kernel.  Every warp ends its share of a token with one arrival on the stage's `done`
// mbarrier and moves on, and the warp whose turn it is (token i: warp i mod warps) waits for `done`, sends the
// row off as a bulk store, and refills the stage once the store has read it.
// Records without per-token outliers: the output row is written IN PLACE over the token's reference row in the
// stage (a thread reads its 64-byte slab of r and writes x_hat there), so a stage is record + one row.
// Records with outliers: the output row is a row of its own, so that the reference survives the dense pass; the
// warp whose turn it is prepares the outliers while it waits for the others (lane n takes outlier n: aligned
// reference of that channel + the stored binary16 value) and writes them over the dense results once every warp
// has arrived.  No other thread looks at the outlier fields.  (A first version that let every thread test the
// outlier list for channels it owns cost ~150 warp instructions per 32 channels and lost to the barrier form.)
struct DwSmem {
    int stage0, stage_bytes, rec_pad, total;
};
__host__ __device__ inline DwSmem dw_smem_layout(int d, int rec, int stages, bool out_row) {
    DwSmem s;
    s.stage0 = align_up((int)sizeof(WsCtrl), 128);
    s.rec_pad = align_up(rec, 128);
    s.stage_bytes = s.rec_pad + 2 * d + (out_row ? 2 * d : 0);   // record, reference row (, output row)
    s.total = s.stage0 + stages * s.stage_bytes;
    return s;
}

// KT > 0: records with per-token outliers (the output row is a row of its own behind the reference row).
// ROW1: the call can contain directly coded tokens (a row list, or no reference at all); they take their steps
// from row 1 of the table, which this form keeps in registers as well.
// D: the hidden width as a compile-time constant (5120: -1 % on the reconstruction with directly coded tokens; at 4096
// the constant measured the same at 131072 tokens and 5 % slower at 16384, so that width reads it from the parameters).
template <int BITS, int KT, bool SUB, bool ROW1, int D = 0>
__global__ void __launch_bounds__(256, 2) decode_ws_kernel(const CodecParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = D ? (D / 32 + 31) / 32 : nt >> 5;
    const int rot = (lane >> 1) & 3;
    const int d = D ? D : p.d;
    const bool valid = tid * 32 < d;
    const int S = D ? (D / 32 > 128 ? 3 : 2) : p.stages;   // the host's rule: three stages for CTAs of more than 128 threads
    const DwSmem L = dw_smem_layout(d, p.rec, S, KT > 0);
    WsCtrl *ctrl = reinterpret_cast<WsCtrl *>(smem);
    const uint32_t sbase = smem_u32(smem);
    constexpr uint32_t cmask = (1u << BITS) - 1u;
    constexpr uint32_t H = 1u << (BITS - 1);
    constexpr uint32_t ones = (BITS == 4) ? 0x11111111u : (BITS == 3) ? 0x00249249u : 0x00005555u;
    constexpr uint32_t highs = ones << (BITS - 1);
    constexpr float kBase = 8388608.0f + (float)H;  // 2^23 + H
    const uint32_t row_bytes = 2u * (uint32_t)d;

    if (p.T <= gridDim.x) grid_launch_dependents();
    if (tid == 0) {
        for (int s = 0; s < S; s++) {
            mbar_init(smem_u32(&ctrl->full[s]), 1);
            mbar_init(smem_u32(&ctrl->done[s]), nwarps);
        }
        ctrl->abort = 0;
        mbar_init_fence();
    }
    __syncthreads();
    grid_dependency_wait();
    const int first = blockIdx.x, stride = gridDim.x;
    const long long n_tok = tokens_to_do<SUB>(p);
    const int n_my = (n_tok > first) ? (int)((n_tok - first + stride - 1) / stride) : 0;
    auto raw_row_of = [&](int k) -> int {
        long long t = token_at<SUB>(p, first + (long long)k * stride);
        return p.ref_row ? p.ref_row[t] : (int)t;
    };
    auto issue = [&](int k, int s, int raw_row) {
        const long long t = token_at<SUB>(p, first + (long long)k * stride);
        const int row = resolve_row<SUB>(p, raw_row);
        ctrl->row[s] = row;
        const uint32_t bar = smem_u32(&ctrl->full[s]);
        const uint32_t base = sbase + L.stage0 + s * L.stage_bytes;
        mbar_arrive_expect_tx(bar, p.test_extra_tx + (uint32_t)p.rec + (row >= 0 ? row_bytes : 0u));
        bulk_load(base, p.payload + t * p.rec, (uint32_t)p.rec, bar);
        if (row >= 0) bulk_load(base + L.rec_pad, ref_row_ptr<SUB>(p, row), row_bytes, bar);
    };
    if (tid == 0)
        for (int k = 0; k < S && k < n_my; k++) issue(k, k, raw_row_of(k));

    uint32_t off[4];
#pragma unroll
    for (int j = 0; j < 4; j++) off[j] = (uint32_t)(tid * 64 + ((j + rot) & 3) * 16);
    // step table, row 0, in slot order
    u64 st0[16];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
        if (valid) {
            s0 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1)));
            s1 = __ldg(reinterpret_cast<const float4 *>(p.step + (off[j] >> 1) + 4));
        }
        st0[4 * j + 0] = pack2(s0.x, s0.y);
        st0[4 * j + 1] = pack2(s0.z, s0.w);
        st0[4 * j + 2] = pack2(s1.x, s1.y);
        st0[4 * j + 3] = pack2(s1.z, s1.w);
    }
    // Row 1 (directly coded tokens) as packed binary16 in 16 registers, when binary16 holds every entry of the row
    // exactly -- which is how the calibration writes them.  Otherwise those tokens read the row from memory.
    uint32_t sh1[16];
    bool row1_exact = ROW1;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
        if (ROW1 && valid) {
            s0 = __ldg(reinterpret_cast<const float4 *>(p.step + d + (off[j] >> 1)));
            s1 = __ldg(reinterpret_cast<const float4 *>(p.step + d + (off[j] >> 1) + 4));
        }
        const float v[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
            const float2 back = __half22float2(h);
            row1_exact = row1_exact && back.x == v[2 * i] && back.y == v[2 * i + 1];
            sh1[4 * j + i] = *reinterpret_cast<const uint32_t *>(&h);
        }
    }
    if (ROW1) row1_exact = __syncthreads_and(row1_exact) != 0;
    const u64 base2 = pack2(kBase, kBase);

    int stage = 0, duty = 0;
    uint32_t parity = 0;
    bool timed_out = false;
    for (int it = 0; it < n_my; it++) {
        if (*reinterpret_cast<volatile int *>(&ctrl->abort)) break;
        unsigned char *rec = smem + L.stage0 + stage * L.stage_bytes;
        const uint32_t rs = sbase + L.stage0 + stage * L.stage_bytes + L.rec_pad;
        const uint32_t os = KT > 0 ? rs + row_bytes : rs;     // where x_hat goes: its own row, or over the reference
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->full[stage]), parity))) { timed_out = true; break; }
        const bool has_ref = ctrl->row[stage] >= 0;

        if (valid) {
            const uint32_t cf = reinterpret_cast<const uint32_t *>(rec)[tid >> p.lpg_shift];
            const float a = half_bits_to_float(cf & 0xffff), b = half_bits_to_float(cf >> 16);
            const u64 a2 = pack2(a, a), b2 = pack2(b, b);
            // code words of the four pieces, in piece order, then rotated into slot order
            const uint32_t *cw = reinterpret_cast<const uint32_t *>(rec + 4 * p.J) + tid * BITS;
            uint32_t words[4];
            if (BITS == 4) {
                words[0] = cw[0]; words[1] = cw[1]; words[2] = cw[2]; words[3] = cw[3];
            } else if (BITS == 3) {
                uint32_t w0 = cw[0], w1 = cw[1], w2 = cw[2];
                words[0] = w0 & 0xffffffu;
                words[1] = (w0 >> 24) | ((w1 & 0xffffu) << 8);
                words[2] = (w1 >> 16) | ((w2 & 0xffu) << 16);
                words[3] = w2 >> 8;
            } else {
                uint32_t w0 = cw[0], w1 = cw[1];
                words[0] = w0 & 0xffffu; words[1] = w0 >> 16; words[2] = w1 & 0xffffu; words[3] = w1 >> 16;
            }
            uint32_t reserved = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                uint32_t v = words[q] ^ highs;  // field == 0  <=>  code == -2^(BITS-1)
                reserved |= (v - ones) & ~v & highs;
                words[q] = v;                   // fields now hold code + H (offset binary)
            }
            if (reserved && p.status) atomicOr(p.status, RAC_STATUS_RESERVED_CODE);
            rot_left4(words, rot);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int c = (int)(off[j] >> 1);
                u64 r2[4], st2[4];
                if (has_ref) {
                    load_ref_slot(rs + off[j], p.gain, p.bias, c, r2);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++) r2[i] = 0ull;
                }
                if (has_ref) {
#pragma unroll
                    for (int i = 0; i < 4; i++) st2[i] = st0[4 * j + i];
                } else if (ROW1 && row1_exact) {
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&sh1[4 * j + i]));
                        st2[i] = pack2(f.x, f.y);
                    }
                } else {
                    const float4 s0 = __ldg(reinterpret_cast<const float4 *>(p.step + d + c));
                    const float4 s1 = __ldg(reinterpret_cast<const float4 *>(p.step + d + c + 4));
                    st2[0] = pack2(s0.x, s0.y); st2[1] = pack2(s0.z, s0.w); st2[2] = pack2(s1.x, s1.y); st2[3] = pack2(s1.z, s1.w);
                }
                const uint32_t w = words[j];
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float q0 = __uint_as_float(0x4b000000u | ((w >> (BITS * (2 * i))) & cmask));
                    const float q1 = __uint_as_float(0x4b000000u | ((w >> (BITS * (2 * i + 1))) & cmask));
                    float x0, x1;
                    unpack2(pfma(psub(pack2(q0, q1), base2), st2[i], pfma(a2, r2[i], b2)), x0, x1);
                    o[i] = f2_to_bf16x2(x0, x1);
                }
                sts128(os + off[j], make_uint4(o[0], o[1], o[2], o[3]));
            }
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&ctrl->done[stage])) : "memory");

        if (warp == duty) {
            const int k_next = it + S;
            int raw_next = 0;
            if (lane == 0 && k_next < n_my) raw_next = raw_row_of(k_next);
            // outliers: lane n prepares outlier n (Eq. 9: aligned reference + binary16 value) while the other warps
            // are still busy; record and reference row do not change any more
            int patch_c = -1;
            unsigned short patch_x = 0;
            if (KT > 0) {
                const unsigned short *oidx = reinterpret_cast<const unsigned short *>(rec + 4 * p.J + p.code_bytes);
                const unsigned short *oval = oidx + p.topk;
                const int c = lane < p.topk ? (int)oidx[lane] : -1;
                const bool ok = c >= 0 && c < d;
                if (ok) {
                    const uint32_t cf = reinterpret_cast<const uint32_t *>(rec)[c >> (5 + p.lpg_shift)];
                    float r = 0.f;
                    if (has_ref) {
                        r = __uint_as_float((uint32_t)(*reinterpret_cast<const unsigned short *>(rec + L.rec_pad + 2 * c)) << 16);
                        if (p.gain) r = bf16_round(__fmaf_rn(half_bits_to_float(p.gain[c]), r, half_bits_to_float(p.bias[c])));
                    }
                    const float xh = __fadd_rn(__fmaf_rn(half_bits_to_float(cf & 0xffff), r, half_bits_to_float(cf >> 16)),
                                               half_bits_to_float(oval[lane]));
                    patch_x = __bfloat16_as_ushort(__float2bfloat16_rn(xh));
                }
                // a malformed record may name a channel twice: the later entry wins, as in a serial pass
                const unsigned int same = __match_any_sync(0xffffffffu, ok ? c : -1 - lane);
                if (ok && (31 - __clz(same)) == lane) patch_c = c;
                if (__any_sync(0xffffffffu, c >= d) && lane == 0 && p.status) atomicOr(p.status, RAC_STATUS_OUTLIER_RANGE);
            }
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&ctrl->done[stage]), parity))) { timed_out = true; break; }
            if (KT > 0) {
                if (patch_c >= 0)
                    reinterpret_cast<unsigned short *>(rec + L.rec_pad + row_bytes)[patch_c] = patch_x;
                fence_async_smem();
                __syncwarp();
            }
            if (lane == 0) {
                const long long t = token_at<SUB>(p, first + (long long)it * stride);
                bulk_store(p.X_hat + t * d, os, row_bytes);
                bulk_commit();
                bulk_wait_read<0>();      // the row has been read: the stage may be refilled
                if (k_next < n_my) issue(k_next, stage, raw_next);
            }
            __syncwarp();
        }
        if (++stage == S) { stage = 0; parity ^= 1u; }
        if (++duty == nwarps) duty = 0;
    }
    if (timed_out) {
        ctrl->abort = 1;
        if (p.status) atomicOr(p.status, RAC_STATUS_TIMEOUT);
    }
    __syncthreads();
    if (lane == 0) bulk_wait_all();
    if (tid == 0 && *reinterpret_cast<volatile int *>(&ctrl->abort)) {
        for (int s = 0; s < S; s++) {
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 0);
            mbar_wait_bounded(smem_u32(&ctrl->full[s]), 1);
        }
    }
}

// ------------------------------------------------------------------------------------------------
// host side: launch plumbing
// ------------------------------------------------------------------------------------------------

int fill_common(const Geometry &g, CodecParams *p, long long T, const void *ref_base, long long ref_rows,
                       const int32_t *ref_row, const void *gain, const void *bias, uint32_t *status) {
    if (T < 0 || ref_rows < 0) return RAC_EINVAL;
    if ((gain == nullptr) != (bias == nullptr)) return RAC_EINVAL;
    if (ref_base && !ref_row && ref_rows < T) return RAC_EINVAL;
    if (ref_base && !aligned16(ref_base)) return RAC_EALIGN;
    if (gain && (!aligned16(gain) || !aligned16(bias))) return RAC_EALIGN;
    if (ref_rows > 0x7fffffffLL) return RAC_EUNSUPPORTED;
    p->ref_base = static_cast<const uint16_t *>(ref_base);
    p->ref_rows = ref_base ? ref_rows : 0;
    p->ref_row = ref_row;
    p->gain = static_cast<const uint16_t *>(gain);
    p->bias = static_cast<const uint16_t *>(bias);
    p->status = status;
    p->T = T;
    p->d = g.d;
    p->J = g.J;
    p->lpg = g.lpg;
    p->lpg_shift = 0;
    while ((1 << p->lpg_shift) < g.lpg) p->lpg_shift++;
    p->topk = g.topk;
    p->rec = g.rec;
    p->code_bytes = g.code_bytes;
    p->inv_group = 1.0f / (float)g.group;
    p->Jq = g.Jq;
    p->lpq = g.lpq;
    p->qgen = g.qgen;
    p->lpq_shift = 0;
    while ((1 << p->lpq_shift) < g.lpq) p->lpq_shift++;
    p->kg = g.topk_group;
    p->scale_off = g.scale_off;
    p->codes_off = g.codes_off;
    p->goff_off = g.goff_off;
    p->gval_off = g.gval_off;
    p->test_extra_tx = 0;
    return RAC_OK;
}

// Encode with outliers, all tokens: the one-launch form.  The shape follows from the number of streaming warps; without x_hat
// the widths 4096 and 5120 with groups of 128 or 64 channels have variants with these compiled in, and of those one for calls
// in which every token has its reference row; with x_hat the width is compiled in for groups of 128.  Everything else has groups
// of 128 and of 64 compiled in (groups of 64 read from the parameters / compiled in, 3-bit, four outliers: 195312 x 1536 527 / 501
// us, 146484 x 2048 398 / 378, 585937 x 512 with x_hat 1187 / 1089; 4-bit, eight: 58593 x 5120 with x_hat 419 / 393).
template <int BITS, int KT, bool XHAT, int NV, int NSEL, int MAXT, int MINB, int D>
static int launch_top_shape(const Geometry &g, CodecParams &p, bool allref, cudaStream_t stream) {
    const int nt = g.nthreads + 32 * NSEL, smem = top_smem_layout(g.d, g.rec, (int)sizeof(TopSel<NSEL, XHAT>)).total;
#define RAC_TOP(G, R) launch_persistent(encode_top_kernel<BITS, KT, XHAT, NV, NSEL, MAXT, MINB, G, D, R>, p, nt, smem, p.T, stream)
    if constexpr (D != 0 && !XHAT) {
        if (g.lpg == 4) return allref ? RAC_TOP(4, true) : RAC_TOP(4, false);
        return allref ? RAC_TOP(2, true) : RAC_TOP(2, false);
    } else if constexpr (D != 0) {
        return RAC_TOP(4, false);
    } else {
        if (g.lpg == 2) return RAC_TOP(2, false);
        return g.lpg == 4 ? RAC_TOP(4, false) : RAC_TOP(0, false);
    }
#undef RAC_TOP
}
template <int BITS, int KT>
static int launch_top_bits(const Geometry &g, CodecParams &p, cudaStream_t stream) {
    const bool allref = p.ref_row == nullptr && p.ref_base != nullptr;   // identity rows
    if (p.X_hat) {
        if constexpr (KT == 8) {
            if (g.lpg == 4 && g.d == 5120) return launch_top_shape<BITS, KT, true, 5, 2, 224, 3, 5120>(g, p, false, stream);
            if (g.lpg == 4 && g.d == 4096) return launch_top_shape<BITS, KT, true, 4, 2, 192, 3, 4096>(g, p, false, stream);
        }
        if (g.nthreads <= 64) return launch_top_shape<BITS, KT, true, 2, 2, 128, 5, 0>(g, p, false, stream);
        if (g.nthreads <= 96) return launch_top_shape<BITS, KT, true, 4, 2, 160, 4, 0>(g, p, false, stream);
        if (g.nthreads <= 128) return launch_top_shape<BITS, KT, true, 4, 2, 192, 3, 0>(g, p, false, stream);
        if (g.nthreads <= 160) return launch_top_shape<BITS, KT, true, 5, 2, 224, 3, 0>(g, p, false, stream);
        return launch_top_shape<BITS, KT, true, 8, 2, 320, 2, 0>(g, p, false, stream);
    }
    if constexpr (KT == 8) {
        if (g.lpg == 4 || g.lpg == 2) {
            if (g.d == 5120) return launch_top_shape<BITS, KT, false, 5, 3, 256, 3, 5120>(g, p, allref, stream);
            if (g.d == 4096) return launch_top_shape<BITS, KT, false, 4, 2, 192, 4, 4096>(g, p, allref, stream);
        }
    }
    if (g.nthreads <= 64) return launch_top_shape<BITS, KT, false, 2, 3, 160, 6, 0>(g, p, false, stream);
    if (g.nthreads <= 128) return launch_top_shape<BITS, KT, false, 4, 2, 192, 4, 0>(g, p, false, stream);
    if (g.nthreads <= 160) return launch_top_shape<BITS, KT, false, 5, 3, 256, 3, 0>(g, p, false, stream);
    return launch_top_shape<BITS, KT, false, 8, 3, 352, 2, 0>(g, p, false, stream);
}
// Which calls with outliers take the one-launch form (two launches / one launch, 4-bit, eight outliers).  Without x_hat all of
// them.  With x_hat everything up to 4096 channels: 512 x 4096 11.7 / 7.8 us, 2048 x 4096 22.3 / 17.4, gathered 100000 x 4096
// 590 / 487, 40000 x 1536 128 / 114.  At 5120 channels the selectors' registers and the step tables in L1 are short: 2048 x 5120
// 24.7 / 21.0, identity rows 100000 x 5120 627 / 619, but with direct tokens, which bring a second row of both tables, 8192
// tokens 62.5 / 62.5 and 100000 tokens 647 / 662.  Beyond, 512 x 8192 19.5 / 17.4 but 4096 x 8192 54 / 62.
static bool one_launch(const Geometry &g, const CodecParams &p) {
    if (!p.X_hat || g.nthreads <= 128) return true;
    if (g.nthreads <= 160) return p.ref_row == nullptr || p.T <= 8192;
    return p.T <= 1024;
}
// The one-launch form in teams: with x_hat, from 2080 to 7168 channels, where one CTA's shared memory holds the teams and the tables,
// in calls of so many tokens that the tables' way there and the CTA's longer start are made up for.  NS: most streaming warps of
// a team.  The line by the threads of a token (one_launch's choice / teams, us; rows g: gathered, 28 % direct):
// up to 96, 64 tokens per SM: 8000 x 3072 35.3 / 35.6, 10000 44.6 / 43.0, 10000 x 2112 40.7 / 38.4;
// up to 128, 54: 6000 x 4096 33.9 / 34.1, 8000 46.3 / 44.6, 8000 x 3584 49.1 / 42.1;
// up to 160, identity rows, 160: 8000 x 5120 59.0 / 59.7, 12000 x 4608 83.7 / 84.4, 24000 x 4608 164.8 / 160.5, x 5120 169.6 / 165.3;
// up to 160, rows g, 56, where one_launch goes over to two launches: 8000 x 4608 55.9 / 57.3, 8300 61.3 / 58.6, 12000 83.7 / 80.4; from
// 4896 channels on 40, since the rows of the tables are more than L1 there: 6000 x 4864 43.7 / 45.8, x 5120 46.8 / 45.4, 8000 x 5120
// 62.8 / 57.0;
// beyond, where it is two launches from 1025 tokens on, 20: 2960 x 6144 32.5 / 30.6, g 33.5 / 28.8, 16000 136.6 / 126.9, g 139.0 / 123.0.
// The width as a constant: 131072 x 5120 rows g 840 -> 828, 12000 82.3 -> 80.9, 12000 x 4096 61.7 -> 61.1.
template <int BITS, int KT, int NV, int NS, int NSEL, int TEAMS, int D>
static int launch_teams_shape(const Geometry &g, CodecParams &p, const DeviceInfo &di, cudaStream_t stream) {
    const TopSmem L = top_smem_layout(g.d, g.rec, (int)sizeof(TopSel<NSEL, true>));
    const int table = g.nthreads * 16;                  // bytes of a piece for all threads of a token
    const int smem = TEAMS * align_up(L.total, 128) + 24 * table, nt = TEAMS * (g.nthreads + 32 * NSEL);
    if (smem > di.max_smem_optin) return RAC_EUNSUPPORTED;
    constexpr int kMaxT = TEAMS * 32 * (NS + NSEL);
#define RAC_TEAMS(G, W) launch_persistent(encode_top_kernel<BITS, KT, true, NV, NSEL, kMaxT, 1, G, W, false, TEAMS>, p, nt, smem, p.T, stream)
    if (D != 0 && g.d == D && g.lpg == 4) return RAC_TEAMS(4, D);
    if (g.lpg == 2) return RAC_TEAMS(2, 0);
    return g.lpg == 4 ? RAC_TEAMS(4, 0) : RAC_TEAMS(0, 0);
#undef RAC_TEAMS
}
// RAC_EUNSUPPORTED: not a call for them
static int launch_teams(const Geometry &g, CodecParams &p, cudaStream_t stream) {
    if (!p.X_hat || p.gain || g.nthreads <= 64 || g.nthreads > 224) return RAC_EUNSUPPORTED;
    DeviceInfo di;
    if (int rc = device_info(&di)) return rc;
    const long long per_sm = g.nthreads <= 96    ? 64
                             : g.nthreads <= 128 ? 54
                             : g.nthreads > 160  ? 20
                             : !p.ref_row        ? 160
                             : g.d > 4864        ? 40
                                                 : 56;
    if (p.T < per_sm * di.sms) return RAC_EUNSUPPORTED;
#define RAC_TEAMS(B, K)                                                                             \
    (g.nthreads <= 96    ? launch_teams_shape<B, K, 3, 3, 2, 4, 0>(g, p, di, stream)                 \
     : g.nthreads <= 128 ? launch_teams_shape<B, K, 4, 4, 2, 3, K == 8 ? 4096 : 0>(g, p, di, stream) \
     : g.nthreads <= 160 ? launch_teams_shape<B, K, 5, 5, 3, 3, K == 8 ? 5120 : 0>(g, p, di, stream) \
                         : launch_teams_shape<B, K, 7, 7, 2, 2, 0>(g, p, di, stream))
    switch (g.bits) {
        case 4: return g.topk == 8 ? RAC_TEAMS(4, 8) : RAC_TEAMS(4, 0);
        case 3: return g.topk == 8 ? RAC_TEAMS(3, 8) : RAC_TEAMS(3, 0);
        case 2: return g.topk == 8 ? RAC_TEAMS(2, 8) : RAC_TEAMS(2, 0);
    }
#undef RAC_TEAMS
    return RAC_EUNSUPPORTED;
}
static int launch_top(const Geometry &g, CodecParams &p, cudaStream_t stream) {
#define RAC_TOPB(B) (g.topk == 8 ? launch_top_bits<B, 8>(g, p, stream) : launch_top_bits<B, 0>(g, p, stream))
    switch (g.bits) {
        case 4: return RAC_TOPB(4);
        case 3: return RAC_TOPB(3);
        case 2: return RAC_TOPB(2);
    }
#undef RAC_TOPB
    return RAC_EUNSUPPORTED;
}

// The streaming kernel of one call.  REF (every token has a reference row: identity rows) drops the test per token; with x_hat it
// also keeps the thread's steps in registers, which is faster at every width (3 to 7 %, 8192 channels 40 %) but in one case: rows of
// 4 or 8 KB in tensors that L2 does not hold (131072 x 4096 583 us with REF, 528 without, 131072 x 2048 308 and 272; both forms are
// equal at 80 M channels; 3840 and 4352 channels 3 and 6 % faster with it, as everywhere else).  Register variants: 64 Ki registers
// hold two CTAs of 160 threads at 128 registers a thread beside a third, or four at 96.  Without x_hat four CTAs are the better
// ones; with x_hat the kernel reads both step tables every token, and at four CTAs per SM the shared-memory carve-out leaves too
// little L1 for them.
template <int BITS, bool TOPK, bool XHAT, int LPG, int D>
static int launch_stream_lpg(const Geometry &g, CodecParams &p, size_t smem, long long max_ctas, cudaStream_t stream) {
    const bool long_pow2 = XHAT && (g.d == 2048 || g.d == 4096) && p.T * g.d > 80'000'000;
    const bool allref = p.ref_row == nullptr && p.ref_base != nullptr && !long_pow2;
#define RAC_STREAM(M, R) \
    launch_persistent(encode_ws_kernel<BITS, TOPK, XHAT, M, false, LPG, D, R>, p, g.nthreads, smem, max_ctas, stream)
    if constexpr (XHAT) {
        if constexpr (!(TOPK && D != 0)) {   // (at that width, identity rows with outliers are always one launch)
            if (allref) return RAC_STREAM(2, true);
        }
        return RAC_STREAM(2, false);
    } else if constexpr (D != 0) {
        return allref ? RAC_STREAM(4, true) : RAC_STREAM(4, false);
    } else {
        return g.nthreads > 96 && g.nthreads <= 160 ? RAC_STREAM(4, false) : RAC_STREAM(2, false);
    }
#undef RAC_STREAM
}

// Widths 4096 and 5120 have variants with the record geometry compiled in; 4096 with outliers is always one launch (one_launch),
// and so is every call with outliers and without x_hat: what those would need is not instantiated.  With eight outliers 5120 comes
// here with gathered rows and a predictor (16384 tokens, groups of 128 137.4 us without the constants, 135.0 with; of 64 149.0 and 145.0),
// or in groups of 32, which have no constants and whose teams do not fit (launch_teams).
template <int BITS, bool TOPK, bool XHAT>
static int launch_stream(const Geometry &g, CodecParams &p, size_t smem, long long max_ctas, cudaStream_t stream) {
    if (p.tok_list || p.intra_base || p.coef_ext)   // the subset form has one variant: it is not the hot path
        return launch_persistent(encode_ws_kernel<BITS, TOPK, XHAT, 2, true, 0>, p, g.nthreads, smem, max_ctas, stream);
    if constexpr (!TOPK || XHAT) {
        if (g.d == 5120 && (!TOPK || g.topk == 8)) {
            if (g.lpg == 4) return launch_stream_lpg<BITS, TOPK, XHAT, 4, 5120>(g, p, smem, max_ctas, stream);
            if (g.lpg == 2) return launch_stream_lpg<BITS, TOPK, XHAT, 2, 5120>(g, p, smem, max_ctas, stream);
        }
        if constexpr (!TOPK) {
            if (g.d == 4096 && g.lpg == 4) return launch_stream_lpg<BITS, TOPK, XHAT, 4, 4096>(g, p, smem, max_ctas, stream);
            if (g.d == 4096 && g.lpg == 2) return launch_stream_lpg<BITS, TOPK, XHAT, 2, 4096>(g, p, smem, max_ctas, stream);
        }
        if (g.lpg == 4) return launch_stream_lpg<BITS, TOPK, XHAT, 4, 0>(g, p, smem, max_ctas, stream);
        if (g.lpg == 2) return launch_stream_lpg<BITS, TOPK, XHAT, 2, 0>(g, p, smem, max_ctas, stream);
        return launch_stream_lpg<BITS, TOPK, XHAT, 0, 0>(g, p, smem, max_ctas, stream);
    }
    return RAC_EUNSUPPORTED;
}

template <int BITS>
static int launch_stream_bits(const Geometry &g, CodecParams &p, size_t smem, long long max_ctas, cudaStream_t stream) {
    if (g.topk > 0)
        return p.X_hat ? launch_stream<BITS, true, true>(g, p, smem, max_ctas, stream)
                       : launch_stream<BITS, true, false>(g, p, smem, max_ctas, stream);
    return p.X_hat ? launch_stream<BITS, false, true>(g, p, smem, max_ctas, stream)
                   : launch_stream<BITS, false, false>(g, p, smem, max_ctas, stream);
}

// Encode: one launch (one_launch), or the streaming kernel and then, with outliers, the selection kernel.
static int launch_encode(const Geometry &g, CodecParams &p, long long max_ctas, cudaStream_t stream) {
    if (g.scale_mode == 1) return launch_encode_dyn(g, p, max_ctas, stream);
    const bool topk = g.topk > 0;
    const bool sub = p.tok_list || p.intra_base || p.coef_ext;
    if (topk && !sub) {
        const int rc = launch_teams(g, p, stream);
        if (rc != RAC_EUNSUPPORTED) return rc;
        if (one_launch(g, p)) return launch_top(g, p, stream);
    }
    p.stages = 2;
    const size_t smem = ws_smem_layout(g.d, g.rec, p.stages, topk).total;
    int rc = RAC_EUNSUPPORTED;
    switch (g.bits) {
        case 4: rc = launch_stream_bits<4>(g, p, smem, max_ctas, stream); break;
        case 3: rc = launch_stream_bits<3>(g, p, smem, max_ctas, stream); break;
        case 2: rc = launch_stream_bits<2>(g, p, smem, max_ctas, stream); break;
    }
    if (rc != RAC_OK || !topk) return rc;
    DeviceInfo di;
    rc = device_info(&di);
    if (rc != RAC_OK) return rc;
    // A warp per pair of tokens.  Many rounds of them, or a token list: three CTAs of eight warps (80 registers, 48 tokens per
    // SM); few rounds: four CTAs of seven warps (72 registers, 56 tokens).  With more work than one round, every warp gets the
    // same number of rounds (a grid of whole rounds, not a full grid with a ragged last round).
    // (x_hat, gathered rows, eight against seven warps, both launches: 131072 x 5120 846 / 850 us, 8000 x 8192 115 / 112 and 30000 x
    // 8192 392 / 391, 14000 x 5120 99 / 100)
    const bool wide = sub || p.T > (long long)di.sms * 3 * 8 * kOutPair * 6;
    const int wpc = wide ? 8 : 7;
    const long long per_cta = wpc * kOutPair;
    long long blocks = (p.T + per_cta - 1) / per_cta;
    const long long resident = (long long)di.sms * (wide ? 3 : 4);
    if (blocks > resident) {
        const long long rounds = (blocks + resident - 1) / resident;
        blocks = (blocks + rounds - 1) / rounds;
    }
    const int nth = g.d / 32;      // up to 128 threads the call is always one launch (one_launch)
    const unsigned nb = (unsigned)blocks, nt = wpc * 32;
#define RAC_OUT(NV, KT)                                                                    \
    (wide ? launch_after(outlier_kernel<NV, KT, false, 8>, nb, nt, 0, stream, p, g.bits)     \
          : launch_after(outlier_kernel<NV, KT, false, 7>, nb, nt, 0, stream, p, g.bits))
    if (sub) launch_after(outlier_kernel<8, 0, true, 8>, nb, nt, 0, stream, p, g.bits);
    else if (g.topk == 8) {
        if (nth <= 160) RAC_OUT(5, 8);
        else RAC_OUT(8, 8);
    } else {
        if (nth <= 160) RAC_OUT(5, 0);
        else RAC_OUT(8, 0);
    }
#undef RAC_OUT
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

static int launch_decode(const Geometry &g, CodecParams &p, cudaStream_t stream) {
    if (g.scale_mode == 1) return launch_decode_dyn(g, p, stream);
    p.stages = 2;
    DecSmem L = dec_smem_layout(g.d, g.rec, p.stages);
    const int kt = g.topk == 0 ? 0 : (g.topk <= 8 ? 8 : 16);
    const bool sub = p.tok_list || p.intra_base || p.coef_ext;
    // The streaming form is the faster one (131072 x 5120: 0.444 against 0.517 ms without outliers, 0.451 against
    // 0.491 ms with eight; 131072 x 4096: 0.37 against 0.43 and 0.40 against 0.46 ms).  The barrier form serves the
    // token-list / second-reference-buffer calls.
    const bool ws = !sub;
    const int wstages = (g.nthreads > 128 ? 3 : 2);
    DwSmem LW = dw_smem_layout(g.d, g.rec, wstages, kt > 0);
    if (ws) p.stages = wstages;
    const bool row1 = p.ref_row != nullptr || p.ref_base == nullptr;   // else every token has its reference row
#define RAC_DECW(B, K, W)                                                                                      \
    (row1 ? launch_persistent(decode_ws_kernel<B, K, false, true, W>, p, g.nthreads, LW.total, p.T, stream)   \
          : launch_persistent(decode_ws_kernel<B, K, false, false, W>, p, g.nthreads, LW.total, p.T, stream))
#define RAC_DEC(B, K)                                                                            \
    (sub ? launch_persistent(decode_kernel<B, K, true>, p, g.nthreads, L.total, p.T, stream)    \
     : ws ? (g.d == 5120 ? RAC_DECW(B, K, 5120) : RAC_DECW(B, K, 0)) \
         : launch_persistent(decode_kernel<B, K, false>, p, g.nthreads, L.total, p.T, stream))
    switch (g.bits * 100 + kt) {
        case 400: return RAC_DEC(4, 0);
        case 408: return RAC_DEC(4, 8);
        case 416: return RAC_DEC(4, 16);
        case 300: return RAC_DEC(3, 0);
        case 308: return RAC_DEC(3, 8);
        case 316: return RAC_DEC(3, 16);
        case 200: return RAC_DEC(2, 0);
        case 208: return RAC_DEC(2, 8);
        case 216: return RAC_DEC(2, 16);
    }
#undef RAC_DEC
#undef RAC_DECW
    return RAC_EUNSUPPORTED;
}

// Tokens whose reference is a row of the same prompt (ref_row >= first_intra_row) form the second wave; both lists come out in
// ascending token order.  Every CTA owns a range of per_cta tokens (a multiple of kSplitTokens) and counts the second-wave tokens
// before it by itself -- the rows are in L2, and what the CTAs read twice costs less than a launch or one CTA's walk over
// everything (131072 tokens 33 us in one CTA, 10 so).  A warp takes 128 consecutive tokens
// and reads them once: a count, one barrier, the lists (2048 tokens 3.9 us with a second reading, 1.7 so).
constexpr int kSplitTokens = 4096, kSplitCtas = 128;
__global__ void __launch_bounds__(1024) split_waves_kernel(const int32_t *ref_row, int T, long long first_intra_row, int per_cta,
                                                           int32_t *wave1, int32_t *wave2, int32_t *wave_count) {
    __shared__ int s_cnt[2][32];
    grid_launch_dependents();
    grid_dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lo = blockIdx.x * per_cta, hi = min(T, lo + per_cta);
    int n2 = 0;                       // second-wave tokens before the current 4096
    if (lo > 0) {
        int c = 0;
        for (int t = tid; t < lo; t += 16 * 1024) {
            int v[16];
#pragma unroll
            for (int u = 0; u < 16; u++) v[u] = ref_row[min(t + 1024 * u, lo - 1)];
#pragma unroll
            for (int u = 0; u < 16; u++) c += (t + 1024 * u < lo && v[u] >= first_intra_row) ? 1 : 0;
        }
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) s_cnt[1][warp] = c;
        __syncthreads();
        n2 = __reduce_add_sync(0xffffffffu, s_cnt[1][lane]);
    }
    for (int base = lo, buf = 0; base < hi; base += kSplitTokens, buf ^= 1) {
        const int t0 = base + warp * 128 + lane;
        int v[4];
        unsigned int second[4];
        int c = 0;
#pragma unroll
        for (int u = 0; u < 4; u++) v[u] = t0 + 32 * u < hi ? ref_row[t0 + 32 * u] : -1;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            second[u] = __ballot_sync(0xffffffffu, v[u] >= first_intra_row);
            c += __popc(second[u]);
        }
        if (lane == 0) s_cnt[buf][warp] = c;
        __syncthreads();              // (a buffer is written again only behind the next one's barrier)
        const int other = s_cnt[buf][lane];
        int at = n2 + __reduce_add_sync(0xffffffffu, lane < warp ? other : 0);
        n2 += __reduce_add_sync(0xffffffffu, other);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int t = t0 + 32 * u, before = at + __popc(second[u] & ((1u << lane) - 1u));
            if (t < hi) {
                if ((second[u] >> lane) & 1u) wave2[before] = t;
                else wave1[t - before] = t;
            }
            at += __popc(second[u]);
        }
    }
    if (hi == T && tid == 0) {
        wave_count[0] = T - n2;
        wave_count[1] = n2;
    }
}

// A subset of the tokens and a second reference buffer (the *_list entry points); all null/0 otherwise.
struct Subset {
    const int32_t *tok_list = nullptr;
    const int32_t *tok_count = nullptr;
    const void *intra_base = nullptr;
    long long intra_rows = 0;
    const uint32_t *coef_seg = nullptr;
    const int32_t *seg_of = nullptr;
};
static int apply_subset(const Subset &sub, CodecParams *p) {
    if ((sub.tok_list == nullptr) != (sub.tok_count == nullptr)) return RAC_EINVAL;
    if (sub.intra_rows < 0 || (sub.intra_rows > 0 && !sub.intra_base)) return RAC_EINVAL;
    if (sub.intra_base && !aligned16(sub.intra_base)) return RAC_EALIGN;
    if (p->ref_rows + sub.intra_rows > 0x7fffffffLL) return RAC_EUNSUPPORTED;
    p->tok_list = sub.tok_list;
    p->tok_count = sub.tok_count;
    p->intra_base = sub.intra_rows > 0 ? static_cast<const uint16_t *>(sub.intra_base) : nullptr;
    p->intra_rows = sub.intra_rows;
    p->coef_ext = sub.coef_seg;
    p->seg_of = sub.seg_of;
    return RAC_OK;
}

// test hook of rac_selftest_bounded_wait: bytes announced beyond what a stage's copies deliver
struct WaitTest {
    uint32_t extra_tx;
};

static int reconstruct_impl(const rac_codec_cfg *cfg, const void *payload, int64_t T, const void *ref_base,
                            int64_t ref_rows, const int32_t *ref_row, const void *gain, const void *bias,
                            const float *step, void *X_hat, uint32_t *dev_status, void *stream,
                            const Subset &sub = Subset(), const WaitTest *wt = nullptr) {
    Geometry g;
    int rc = make_geometry(cfg, &g);
    if (rc != RAC_OK) return rc;
    CodecParams p = {};
    rc = fill_common(g, &p, T, ref_base, ref_rows, ref_row, gain, bias, dev_status);
    if (rc != RAC_OK) return rc;
    rc = apply_subset(sub, &p);
    if (rc != RAC_OK) return rc;
    if ((g.coef_fmt == 1) != (sub.coef_seg != nullptr) || (sub.coef_seg != nullptr) != (sub.seg_of != nullptr)) return RAC_EINVAL;
    if (T == 0) return RAC_OK;
    if (!payload || !X_hat || (!step && g.scale_mode == 0)) return RAC_EINVAL;   // mode 1 reads no table
    if (!aligned16(payload) || !aligned16(X_hat) || (step && !aligned16(step))) return RAC_EALIGN;
    p.payload = const_cast<uint8_t *>(static_cast<const uint8_t *>(payload));
    p.X_hat = static_cast<uint16_t *>(X_hat);
    p.step = step;
    if (wt) p.test_extra_tx = wt->extra_tx;
    return launch_decode(g, p, static_cast<cudaStream_t>(stream));
}

}  // namespace rac

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
using namespace rac;

extern "C" {

const char *rac_version(void) { return "rac-b200 0.1.0 (sm_100a)"; }

const char *rac_strerror(int err) {
    switch (err) {
        case RAC_OK: return "ok";
        case RAC_EINVAL: return "invalid argument";
        case RAC_EALIGN: return "pointer not 16-byte aligned";
        case RAC_ESIZE: return "caller buffer too small";
        case RAC_EUNSUPPORTED: return "unsupported configuration";
        case RAC_ECUDA: return "CUDA runtime error";
    }
    return "unknown error";
}

size_t rac_record_bytes(const rac_codec_cfg *cfg) {
    Geometry g;
    return make_geometry(cfg, &g) == RAC_OK ? (size_t)g.rec : 0;
}

size_t rac_payload_bytes(const rac_codec_cfg *cfg, int64_t T) {
    if (T < 0) return 0;
    return rac_record_bytes(cfg) * (size_t)T;
}

// ---- header of a serialised payload (host only)
static uint32_t header_sum(const unsigned char *h) {
    uint32_t sum = 0;
    for (int i = 0; i < 14; i++) {
        uint32_t w;
        memcpy(&w, h + 4 * i, 4);
        sum += w;
    }
    return sum;
}

int rac_header_write(const rac_codec_cfg *cfg, int64_t T, void *header) {
    const size_t rec = rac_record_bytes(cfg);
    if (!header || rec == 0 || T < 0) return RAC_EINVAL;
    unsigned char h[RAC_HEADER_BYTES];
    memset(h, 0, sizeof h);
    memcpy(h, "RACP", 4);
    const uint16_t version = 1, size = RAC_HEADER_BYTES;
    memcpy(h + 4, &version, 2);
    memcpy(h + 6, &size, 2);
    memcpy(h + 8, &T, 8);
    const int32_t f[9] = {cfg->d, cfg->group, cfg->bits, cfg->topk, cfg->coef_fmt, cfg->scale_mode, cfg->flags,
                          cfg->qgroup, cfg->topk_group};
    memcpy(h + 16, f, sizeof f);
    const uint32_t rec32 = (uint32_t)rec;
    memcpy(h + 52, &rec32, 4);
    const uint32_t sum = header_sum(h);
    memcpy(h + 56, &sum, 4);
    memcpy(header, h, sizeof h);
    return RAC_OK;
}

int rac_header_parse(const void *header, rac_codec_cfg *cfg_out, int64_t *T_out) {
    if (!header || !cfg_out || !T_out) return RAC_EINVAL;
    const unsigned char *h = static_cast<const unsigned char *>(header);
    uint16_t version, size;
    uint32_t rec32, sum, tail;
    int64_t T;
    int32_t f[9];
    memcpy(&version, h + 4, 2);
    memcpy(&size, h + 6, 2);
    memcpy(&T, h + 8, 8);
    memcpy(f, h + 16, sizeof f);
    memcpy(&rec32, h + 52, 4);
    memcpy(&sum, h + 56, 4);
    memcpy(&tail, h + 60, 4);
    if (memcmp(h, "RACP", 4) != 0 || version != 1 || size != RAC_HEADER_BYTES || tail != 0 || sum != header_sum(h)) return RAC_EINVAL;
    rac_codec_cfg cfg;
    cfg.d = f[0]; cfg.group = f[1]; cfg.bits = f[2]; cfg.topk = f[3]; cfg.coef_fmt = f[4]; cfg.scale_mode = f[5];
    cfg.flags = f[6]; cfg.qgroup = f[7]; cfg.topk_group = f[8];
    const size_t rec = rac_record_bytes(&cfg);
    if (rec == 0 || rec != (size_t)rec32 || T < 0) return RAC_EINVAL;
    *cfg_out = cfg;
    *T_out = T;
    return RAC_OK;
}

size_t rac_encode_workspace_bytes(const rac_codec_cfg *cfg, int64_t T) {
    Geometry g;
    if (make_geometry(cfg, &g) != RAC_OK || T < 0) return 0;
    if (g.topk == 0) return 0;
    return (size_t)T * (size_t)(((g.d / 32) * 4 + 15) / 16 * 16);  // one 16-byte padded row of slab maxima per token
}

static bool ranges_overlap(const void *a, size_t na, const void *b, size_t nb) {
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(a), b0 = reinterpret_cast<uintptr_t>(b);
    return na > 0 && nb > 0 && a0 < b0 + nb && b0 < a0 + na;
}

static int encode_impl(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                       const int32_t *ref_row, const void *ref_gain, const void *ref_bias, const float *step,
                       const float *inv_step, void *payload, size_t payload_cap, void *X_hat, void *workspace,
                       size_t workspace_bytes, uint32_t *dev_status, void *stream, const Subset &sub = Subset(),
                       const WaitTest *wt = nullptr) {
    Geometry g;
    int rc = make_geometry(cfg, &g);
    if (rc != RAC_OK) return rc;
    CodecParams p = {};
    rc = fill_common(g, &p, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, dev_status);
    if (rc != RAC_OK) return rc;
    rc = apply_subset(sub, &p);
    if (rc != RAC_OK) return rc;
    if ((g.coef_fmt == 1) != (sub.coef_seg != nullptr) || (sub.coef_seg != nullptr) != (sub.seg_of != nullptr)) return RAC_EINVAL;
    if (T == 0) return RAC_OK;
    if (!X || !payload) return RAC_EINVAL;
    if (g.scale_mode == 0 && (!step || !inv_step)) return RAC_EINVAL;   // the static tables; mode 1 reads neither
    if (!aligned16(X) || !aligned16(payload) || (step && !aligned16(step)) || (inv_step && !aligned16(inv_step))) return RAC_EALIGN;
    if (X_hat && !aligned16(X_hat)) return RAC_EALIGN;
    if (payload_cap < (size_t)g.rec * (size_t)T) return RAC_ESIZE;
    if (X_hat && g.topk > 0 && g.scale_mode == 0) {
        // the outlier pass runs after the streaming pass has written x_hat and reads X and the reference rows
        // again: a token's x_hat must not land on X, nor on a reference row that this call still reads.  With
        // identity rows (ref_row == NULL) every token's reference row is the row it writes.
        const size_t out_bytes = (size_t)T * (size_t)g.d * 2;
        if (ranges_overlap(X_hat, out_bytes, X, out_bytes)) return RAC_EUNSUPPORTED;
        if (ref_base && !ref_row && ranges_overlap(X_hat, out_bytes, ref_base, (size_t)ref_rows * (size_t)g.d * 2))
            return RAC_EUNSUPPORTED;
    }
    const size_t need = rac_encode_workspace_bytes(cfg, T);
    if (need > 0) {
        if (!workspace) return RAC_EINVAL;
        if (!aligned16(workspace)) return RAC_EALIGN;
        if (workspace_bytes < need) return RAC_ESIZE;
    }
    p.X = static_cast<const uint16_t *>(X);
    p.payload = static_cast<uint8_t *>(payload);
    p.X_hat = static_cast<uint16_t *>(X_hat);
    p.step = step;
    p.inv_step = inv_step;
    p.tmax = static_cast<float *>(workspace);
    if (wt) p.test_extra_tx = wt->extra_tx;
    return launch_encode(g, p, T, static_cast<cudaStream_t>(stream));
}

int rac_encode(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
               const int32_t *ref_row, const void *ref_gain, const void *ref_bias, const float *step,
               const float *inv_step, void *payload, size_t payload_cap, void *workspace, size_t workspace_bytes,
               uint32_t *dev_status, void *stream) {
    return encode_impl(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload, payload_cap,
                       nullptr, workspace, workspace_bytes, dev_status, stream);
}

int rac_encode_reconstruct(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                           const int32_t *ref_row, const void *ref_gain, const void *ref_bias, const float *step,
                           const float *inv_step, void *payload, size_t payload_cap, void *X_hat, void *workspace,
                           size_t workspace_bytes, uint32_t *dev_status, void *stream) {
    if (T > 0 && !X_hat) return RAC_EINVAL;
    return encode_impl(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload, payload_cap,
                       X_hat, workspace, workspace_bytes, dev_status, stream);
}

int rac_selftest_bounded_wait(const rac_codec_cfg *cfg, int32_t which, const void *in, int64_t T, const void *ref_base,
                              int64_t ref_rows, const float *step, const float *inv_step, void *out, size_t out_cap,
                              void *workspace, size_t workspace_bytes, uint32_t *dev_status, void *stream) {
    if (T < 1 || T > (which == 2 ? 16384 : 1024) || !dev_status) return RAC_EINVAL;
    const WaitTest wt = {16u};   // every stage announces 16 bytes that never come
    if (which == 2) {
        const size_t rec = rac_record_bytes(cfg), pay = (size_t)T * rec;
        if (rec == 0 || !out) return RAC_EINVAL;
        if (out_cap < pay + (size_t)T * (size_t)cfg->d * 2) return RAC_ESIZE;
        return encode_impl(cfg, in, T, ref_base, ref_rows, nullptr, nullptr, nullptr, step, inv_step, out, pay,
                           static_cast<uint8_t *>(out) + pay, workspace, workspace_bytes, dev_status, stream, Subset(), &wt);
    }
    if (which == 0)
        return encode_impl(cfg, in, T, ref_base, ref_rows, nullptr, nullptr, nullptr, step, inv_step, out, out_cap, nullptr,
                           workspace, workspace_bytes, dev_status, stream, Subset(), &wt);
    if (which == 1) {
        const size_t need = rac_record_bytes(cfg) ? (size_t)T * (size_t)cfg->d * 2 : 0;
        if (need == 0 || out_cap < need) return need == 0 ? RAC_EINVAL : RAC_ESIZE;
        return reconstruct_impl(cfg, in, T, ref_base, ref_rows, nullptr, nullptr, nullptr, step, out, dev_status, stream,
                                Subset(), &wt);
    }
    return RAC_EINVAL;
}

int rac_decode_reconstruct(const rac_codec_cfg *cfg, const void *payload, int64_t T, const void *ref_base,
                           int64_t ref_rows, const int32_t *ref_row, const void *ref_gain, const void *ref_bias,
                           const float *step, void *X_hat, uint32_t *dev_status, void *stream) {
    return reconstruct_impl(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat, dev_status, stream);
}

int rac_sender_reconstruct(const rac_codec_cfg *cfg, const void *payload, int64_t T, const void *ref_base,
                           int64_t ref_rows, const int32_t *ref_row, const void *ref_gain, const void *ref_bias,
                           const float *step, void *X_hat, uint32_t *dev_status, void *stream) {
    return reconstruct_impl(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat, dev_status, stream);
}

int rac_encode_reconstruct_list(const rac_codec_cfg *cfg, const void *X, int64_t T, const int32_t *tok_list,
                                const int32_t *tok_count, const void *ref_base, int64_t ref_rows, const int32_t *ref_row,
                                const void *intra_base, int64_t intra_rows, const uint32_t *coef_seg, const int32_t *seg_of,
                                const void *ref_gain, const void *ref_bias,
                                const float *step, const float *inv_step, void *payload, size_t payload_cap, void *X_hat,
                                void *workspace, size_t workspace_bytes, uint32_t *dev_status, void *stream) {
    Subset sub;
    sub.tok_list = tok_list;
    sub.tok_count = tok_count;
    sub.intra_base = intra_base;
    sub.intra_rows = intra_rows;
    sub.coef_seg = coef_seg;
    sub.seg_of = seg_of;
    return encode_impl(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, inv_step, payload, payload_cap,
                       X_hat, workspace, workspace_bytes, dev_status, stream, sub);
}

int rac_decode_reconstruct_list(const rac_codec_cfg *cfg, const void *payload, int64_t T, const int32_t *tok_list,
                                const int32_t *tok_count, const void *ref_base, int64_t ref_rows, const int32_t *ref_row,
                                const void *intra_base, int64_t intra_rows, const uint32_t *coef_seg, const int32_t *seg_of,
                                const void *ref_gain, const void *ref_bias,
                                const float *step, void *X_hat, uint32_t *dev_status, void *stream) {
    Subset sub;
    sub.tok_list = tok_list;
    sub.tok_count = tok_count;
    sub.intra_base = intra_base;
    sub.intra_rows = intra_rows;
    sub.coef_seg = coef_seg;
    sub.seg_of = seg_of;
    return reconstruct_impl(cfg, payload, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, step, X_hat, dev_status, stream,
                            sub);
}

int rac_split_waves(const int32_t *ref_row, int64_t T, int64_t first_intra_row, int32_t *wave1, int32_t *wave2,
                    int32_t *wave_count, void *stream) {
    if (T < 0 || first_intra_row < 0 || !wave_count) return RAC_EINVAL;
    if (T >= (1ll << 30)) return RAC_EUNSUPPORTED;
    if (T > 0 && (!ref_row || !wave1 || !wave2)) return RAC_EINVAL;
    const long long pieces = (T + kSplitTokens - 1) / kSplitTokens;
    const int per_cta = (int)((pieces + kSplitCtas - 1) / kSplitCtas) * kSplitTokens;
    const unsigned ctas = T > 0 ? (unsigned)((T + per_cta - 1) / per_cta) : 1u;
    launch_after(split_waves_kernel, ctas, 1024, 0, static_cast<cudaStream_t>(stream), ref_row, (int)T, (long long)first_intra_row,
                 per_cta, wave1, wave2, wave_count);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

}  // extern "C"
