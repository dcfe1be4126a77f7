// Step tables, segment fit and reconstruction error (sm_100a): the passes that look at a whole call's tokens to produce
// a few numbers.
//
// Kernels: calib_kernel (per-channel sums of e^2, or -- for the segment fit -- the statistics of every (token, group)),
// calib_finalize_kernel (step tables from the sums), segment_fit_kernel + seg_of_kernel (Eq. 6 over several fitting
// positions), recon_error_kernel + recon_error_finalize_kernel (error of a sender-path run).
#include "rac_codec_dev.cuh"

namespace rac {

// ------------------------------------------------------------------------------------------------
// per-channel sums of e^2 (the residual of Eq. 7 with wire coefficients)
// ------------------------------------------------------------------------------------------------
// A warp owns 1024 consecutive channels (32 per lane) and strides over tokens by itself: two stages of its own, each
// filled by one bulk copy of the X row and one of the reference row, and no barrier between warps until the end.  The front
// end is the encoder's (slab loads, Eq. 6 statistics, wire coefficients); instead of codes, every lane accumulates e^2 of
// its channels, for tokens with a reference (table row 0) in registers, for tokens coded directly (row 1) in shared memory.
// The warps of a CTA own the same channels and add their sums up at the end, in warp order.  The partition of the tokens
// depends on the width only: `parts` CTAs per 1024 channels, chosen so that all CTAs are resident at once.
// One CTA of whole rows per partition (128 of them, four warps and a CTA barrier per token) ran 4096 x 2880 in 51 us, this
// form in 16 us: the rows were waiting for one another, not for memory.
// MOMENTS: the first pass of the segment fit instead -- the centred statistics of Eq. 6 of every (token, group)
// go to p.moments and nothing is accumulated.
constexpr int kCalWarps = 8;
constexpr int kCalStages = 2;
constexpr int kCalParts = 128;                 // most partitions of the tokens (the workspace is sized for them)
constexpr int kCalStageBytes = 4096;           // 2 KB of X, 2 KB of the reference
constexpr int kCalAccBytes = 33 * 32 * 4;      // 32 sums per lane, rows of 33 words so that both readings are conflict-free

struct CalSmem {
    int stage0, acc1, cnt, total;
};
__host__ __device__ constexpr CalSmem cal_smem_layout(bool moments) {
    CalSmem s{};
    s.stage0 = 128;                            // behind the mbarriers
    s.acc1 = s.stage0 + kCalWarps * kCalStages * kCalStageBytes;
    s.cnt = s.acc1 + (moments ? 0 : kCalWarps * kCalAccBytes);
    s.total = s.cnt + kCalWarps * 2 * 4;
    return s;
}
// chunks of 1024 channels, and partitions of the tokens: chunks * parts <= 296 CTAs (two on each of 148 SMs)
static int cal_chunks(int d) { return (d + 1023) / 1024; }
static int cal_parts(int d) { return 296 / cal_chunks(d) < kCalParts ? 296 / cal_chunks(d) : kCalParts; }

template <bool MOMENTS>
__global__ void __launch_bounds__(kCalWarps * 32, MOMENTS ? 3 : 2) calib_kernel(const CodecParams p, const int nchunk) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr CalSmem L = cal_smem_layout(MOMENTS);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rot = (lane >> 1) & 3;
    const int d = p.d;
    const int chunk = blockIdx.x % nchunk, part = blockIdx.x / nchunk, parts = gridDim.x / nchunk;
    const int slab = chunk * 32 + lane;
    const bool valid = slab * 32 < d;
    const uint32_t chunk_bytes = (uint32_t)min(2048, 2 * d - 2048 * chunk);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + warp * kCalStages * 8;
    const uint32_t stage0 = sbase + L.stage0 + warp * kCalStages * kCalStageBytes;
    if (lane == 0) {
        for (int s = 0; s < kCalStages; s++) mbar_init(bar0 + 8 * s, 1);
        mbar_init_fence();
    }
    float *acc1 = reinterpret_cast<float *>(smem + L.acc1 + warp * kCalAccBytes);
    if (!MOMENTS)
        for (int o = lane; o < 33 * 32; o += 32) acc1[o] = 0.f;
    __syncwarp();
    grid_dependency_wait();

    const long long first = part * kCalWarps + warp, stride = parts * kCalWarps;
    const int n_my = p.T > first ? (int)((p.T - first + stride - 1) / stride) : 0;
    auto raw_row_of = [&](int k) -> int {
        const long long t = first + k * stride;
        return p.ref_row ? __ldg(p.ref_row + t) : (int)t;
    };
    // all lanes learn the token's row; lane 0 starts its copies
    auto issue = [&](int k, int s, int raw) -> bool {
        const int row = resolve_row<false>(p, raw, lane == 0);
        if (lane == 0) {
            const long long t = first + k * stride;
            const uint32_t bar = bar0 + 8 * s, a = stage0 + s * kCalStageBytes;
            mbar_arrive_expect_tx(bar, row >= 0 ? 2 * chunk_bytes : chunk_bytes);
            bulk_load(a, p.X + t * d + chunk * 1024, chunk_bytes, bar);
            if (row >= 0) bulk_load(a + 2048, p.ref_base + (long long)row * d + chunk * 1024, chunk_bytes, bar);
        }
        return row >= 0;
    };
    bool ref_of[kCalStages] = {false, false};
    if (0 < n_my) ref_of[0] = issue(0, 0, raw_row_of(0));
    if (1 < n_my) ref_of[1] = issue(1, 1, raw_row_of(1));
    int next_raw = 2 < n_my ? raw_row_of(2) : 0;

    float acc0[32];
#pragma unroll
    for (int i = 0; i < 32; i++) acc0[i] = 0.f;
    int cnt_ref = 0, cnt_dir = 0;
    bool timed_out = false;

    // one token in stage s; returns false when its data did not arrive
    auto token = [&](int k, int s, uint32_t parity) -> bool {
        const uint32_t xs = stage0 + s * kCalStageBytes;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar0 + 8 * s, parity))) return false;
        const bool has_ref = ref_of[s];
        uint32_t xw[16], rw[16];     // lanes beyond the row hold zeros and form groups of their own
#pragma unroll
        for (int i = 0; i < 16; i++) { xw[i] = 0u; rw[i] = 0u; }
        if (valid) {
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t off = (uint32_t)(lane * 64 + ((j + rot) & 3) * 16);
                const uint4 w = lds128(xs + off);
                xw[4 * j + 0] = w.x; xw[4 * j + 1] = w.y; xw[4 * j + 2] = w.z; xw[4 * j + 3] = w.w;
                if (has_ref) {
                    const uint4 r = load_ref_words(xs + 2048 + off, p.gain, p.bias, chunk * 1024 + (int)(off >> 1));
                    rw[4 * j + 0] = r.x; rw[4 * j + 1] = r.y; rw[4 * j + 2] = r.z; rw[4 * j + 3] = r.w;
                }
            }
        }
        __syncwarp();                                       // the rows are in registers: the stage can be refilled
        if (k + kCalStages < n_my) {
            ref_of[s] = issue(k + kCalStages, s, next_raw);
            if (k + kCalStages + 1 < n_my) next_raw = raw_row_of(k + kCalStages + 1);
        }
        const long long tok = first + k * stride;
        u64 a2, b2;
        float4 st;
        if (!MOMENTS && p.coef_ext) {
            // shared coefficients: the residual of Eq. 7 with the words of the token's segment
            const uint32_t cw = valid ? p.coef_ext[(long long)p.seg_of[tok] * p.J + (slab >> p.lpg_shift)] : 0u;
            const float a = half_bits_to_float(cw & 0xffffu), b = half_bits_to_float(cw >> 16);
            a2 = pack2(a, a);
            b2 = pack2(b, b);
        } else {
            fit_group(xw, rw, has_ref, p.lpg, p.inv_group, 0xffffffffu, p.status, a2, b2, &st);
        }
        if (MOMENTS) {
            if (valid && (lane & (p.lpg - 1)) == 0) p.moments[tok * p.J + (slab >> p.lpg_shift)] = st;
        } else if (has_ref) {
            cnt_ref++;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                float e0, e1;
                unpack2(sub_pair(xw[i], pfma(a2, bf16x2_to_p(rw[i]), b2)), e0, e1);
                acc0[2 * i] = __fmaf_rn(e0, e0, acc0[2 * i]);
                acc0[2 * i + 1] = __fmaf_rn(e1, e1, acc0[2 * i + 1]);
            }
        } else {
            cnt_dir++;
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const int f = 8 * (((i >> 2) + rot) & 3) + 2 * (i & 3);    // channel within the slab
                float e0, e1;
                unpack2(sub_pair(xw[i], b2), e0, e1);                      // fma(alpha, 0, beta) = beta
                acc1[f * 33 + lane] = __fmaf_rn(e0, e0, acc1[f * 33 + lane]);
                acc1[(f + 1) * 33 + lane] = __fmaf_rn(e1, e1, acc1[(f + 1) * 33 + lane]);
            }
        }
        return true;
    };
    uint32_t parity = 0;
    for (int k = 0; k < n_my && !timed_out; k += 2) {
        timed_out = !token(k, 0, parity) || (k + 1 < n_my && !token(k + 1, 1, parity));
        parity ^= 1u;
    }
    if (timed_out) {
        if (lane == 0 && p.status) atomicOr(p.status, RAC_STATUS_TIMEOUT);
        // give copies that may still be in flight a bounded chance to land before the CTA retires
        for (int s = 0; s < kCalStages; s++) {
            mbar_wait_bounded(bar0 + 8 * s, 0);
            mbar_wait_bounded(bar0 + 8 * s, 1);
        }
    }
    if (MOMENTS) return;

    // sums of this CTA: row 0 goes to where the stages were, then the warps' sums are added in warp order
    int *cnt = reinterpret_cast<int *>(smem + L.cnt);
    if (lane == 0) {
        cnt[2 * warp] = cnt_ref;
        cnt[2 * warp + 1] = cnt_dir;
    }
    static_assert(kCalWarps * kCalAccBytes <= kCalWarps * kCalStages * kCalStageBytes, "row 0 fits where the stages were");
    __syncthreads();
    float *all0 = reinterpret_cast<float *>(smem + L.stage0);
    const float *all1 = reinterpret_cast<const float *>(smem + L.acc1);
#pragma unroll
    for (int i = 0; i < 32; i++) {
        const int f = 8 * (((i >> 3) + rot) & 3) + (i & 7);
        all0[warp * (kCalAccBytes / 4) + f * 33 + lane] = acc0[i];
    }
    __syncthreads();
    float *out = p.calib_partial + (long long)part * 2 * d + chunk * 1024;
    const int nc = min(1024, d - chunk * 1024);
    for (int c = threadIdx.x; c < nc; c += kCalWarps * 32) {
        const int at = (c & 31) * 33 + (c >> 5);
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int w = 0; w < kCalWarps; w++) {
            s0 += all0[w * (kCalAccBytes / 4) + at];
            s1 += all1[w * (kCalAccBytes / 4) + at];
        }
        out[c] = s0;
        out[d + c] = s1;
    }
    if (chunk == 0 && threadIdx.x < 2) {
        int n = 0;
        for (int w = 0; w < kCalWarps; w++) n += cnt[2 * w + threadIdx.x];
        reinterpret_cast<int *>(p.calib_partial + (long long)parts * 2 * d)[2 * part + threadIdx.x] = n;
    }
}

// Step tables from the per-partition sums: 32 channels per CTA, eight threads per channel, each adding every eighth
// partition in binary64, then the eight in order (a fixed summation order -> deterministic).  One thread per channel and
// all partitions in a row took 21 us at d = 2880 (a chain of 128 loads), eight with four loads at a time 5.4; all sixteen are loaded at once now (one trip).
constexpr int kFinSlices = 8;
__global__ void __launch_bounds__(32 * kFinSlices) calib_finalize_kernel(const float *partial, int parts, int d, int bits,
                                                                         float clip_sigmas, float *step, float *inv_step) {
    __shared__ double s_sum[kFinSlices][32];
    __shared__ int s_n;
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;      // d is a multiple of 32: a CTA stays within one table row
    const int row = c >= d;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    grid_launch_dependents();
    grid_dependency_wait();
    const int *cnt = reinterpret_cast<const int *>(partial + (long long)parts * 2 * d);
    double sum = 0.0;
    float v[kCalParts / kFinSlices];     // one trip
#pragma unroll
    for (int u = 0; u < kCalParts / kFinSlices; u++)
        v[u] = slice + u * kFinSlices < parts ? partial[(long long)(slice + u * kFinSlices) * 2 * d + c] : 0.f;
    if (threadIdx.x < parts) atomicAdd(&s_n, cnt[2 * threadIdx.x + row]);
#pragma unroll
    for (int u = 0; u < kCalParts / kFinSlices; u++) sum += (double)v[u];
    s_sum[slice][lane] = sum;
    __syncthreads();
    if (slice != 0) return;
    for (int k = 1; k < kFinSlices; k++) sum += s_sum[k][lane];
    const int n = s_n;
    float s = 0.f, is = 0.f;
    if (n > 0) {
        double qmax = (double)((1 << (bits - 1)) - 1);
        double want = (double)clip_sigmas * sqrt(sum / (double)n) / qmax;
        if (want > 0.0) {
            if (want > 65504.0) want = 65504.0;
            __half h = __double2half(want);
            if ((double)__half2float(h) < want) h = __ushort_as_half((unsigned short)(__half_as_ushort(h) + 1));  // round up
            s = __half2float(h);
            if (s != 0.f) is = __fdiv_rn(1.0f, s);
        }
    }
    step[c] = s;
    inv_step[c] = is;
}
static_assert(kCalParts <= 32 * kFinSlices, "one thread per partition reads the token counts");

// ------------------------------------------------------------------------------------------------
// Eq. 6 over several fitting positions: one coefficient pair per (segment of tokens, group)
// ------------------------------------------------------------------------------------------------
// Pass 1 (calib_kernel<true>, above) leaves the centred statistics of every (token, group).  Pass 2: one warp per
// (segment, group) merges them with the pairwise update of means and centred sums, in binary64 and in a fixed
// order (lane l takes tokens l, l+32, ... of the segment in order, then a shuffle tree), applies the
// zero-variance rule and rounds to the wire format.
struct Mom {
    double n, mr, mh, sxx, sxy;
};
__device__ __forceinline__ Mom mom_merge(const Mom &a, const Mom &b) {
    if (b.n == 0.0) return a;
    if (a.n == 0.0) return b;
    Mom o;
    o.n = a.n + b.n;
    const double dr = b.mr - a.mr, dh = b.mh - a.mh, w = b.n / o.n, f = a.n * w;
    o.mr = a.mr + dr * w;
    o.mh = a.mh + dh * w;
    o.sxx = a.sxx + b.sxx + dr * dr * f;
    o.sxy = a.sxy + b.sxy + dr * dh * f;
    return o;
}
__global__ void __launch_bounds__(256) segment_fit_kernel(const float4 *moments, const int32_t *seg_off, long long n_seg,
                                                          int J, int group, long long T, uint32_t *coef_seg) {
    grid_launch_dependents();
    grid_dependency_wait();
    const long long wid = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (wid >= n_seg * J) return;
    const long long k = wid / J;
    const int j = (int)(wid - k * J);
    long long t0 = seg_off[k], t1 = seg_off[k + 1];
    t0 = t0 < 0 ? 0 : (t0 > T ? T : t0);
    t1 = t1 < t0 ? t0 : (t1 > T ? T : t1);
    Mom m = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (long long t = t0 + lane; t < t1; t += 32) {
        const float4 s = moments[t * J + j];
        const Mom one = {(double)group, (double)s.x, (double)s.y, (double)s.z, (double)s.w};
        m = mom_merge(m, one);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {   // lane l absorbs lane l + o: earlier tokens stay on the left
        Mom b;
        b.n = __shfl_down_sync(0xffffffffu, m.n, o);
        b.mr = __shfl_down_sync(0xffffffffu, m.mr, o);
        b.mh = __shfl_down_sync(0xffffffffu, m.mh, o);
        b.sxx = __shfl_down_sync(0xffffffffu, m.sxx, o);
        b.sxy = __shfl_down_sync(0xffffffffu, m.sxy, o);
        if (lane + o < 32) m = mom_merge(m, b);
    }
    if (lane == 0) {
        double a = 0.0, b = m.mh;
        if (m.sxx > 1e-12 && fabs(m.sxy) < 65504.0 * m.sxx) {
            a = m.sxy / m.sxx;
            b = m.mh - a * m.mr;
        }
        a = fmin(fmax(a, -65504.0), 65504.0);
        b = fmin(fmax(b, -65504.0), 65504.0);
        const uint32_t a16 = __half_as_ushort(__double2half(a)), b16 = __half_as_ushort(__double2half(b));
        coef_seg[k * J + j] = a16 | (b16 << 16);
    }
}
// segment of every token: the last k with seg_off[k] <= t (empty segments have equal offsets and are skipped)
__global__ void seg_of_kernel(const int32_t *seg_off, long long n_seg, long long T, int32_t *seg_of) {
    grid_launch_dependents();
    grid_dependency_wait();
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= T) return;
    long long lo = 0, hi = n_seg;   // invariant: seg_off[lo] <= t (seg_off[0] = 0), answer in [lo, hi)
    while (hi - lo > 1) {
        const long long mid = (lo + hi) >> 1;
        if (seg_off[mid] <= t) lo = mid; else hi = mid;
    }
    seg_of[t] = (int32_t)lo;
}

// ------------------------------------------------------------------------------------------------
// reconstruction error of a sender-path run (input of the byte-cost side of calibration, Sec. IV-C)
// ------------------------------------------------------------------------------------------------
constexpr int kErrGrid = 592;     // fixed, so that the summation order does not depend on the device
constexpr int kErrThreads = 256;

struct ErrSum {
    double se, sx;
    float mx;
};
__device__ __forceinline__ void err_add(ErrSum &s, const uint4 &a, const uint4 &b) {
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const float x0 = __uint_as_float(aw[k] << 16), x1 = __uint_as_float(aw[k] & 0xffff0000u);
        const float y0 = __uint_as_float(bw[k] << 16), y1 = __uint_as_float(bw[k] & 0xffff0000u);
        const float d0 = __fsub_rn(x0, y0), d1 = __fsub_rn(x1, y1);   // exact or one rounding: both are bf16
        s.se += (double)d0 * (double)d0 + (double)d1 * (double)d1;
        s.sx += (double)x0 * (double)x0 + (double)x1 * (double)x1;
        s.mx = fmaxf(s.mx, fmaxf(fabsf(d0), fabsf(d1)));
    }
}
// Sums of a CTA by a fixed tree (the same order on every run): halves of the threads down to one; thread 0 holds them afterwards.
// The three levels above a warp's width are taken by the first warp behind one barrier, the rest by shuffles.
__device__ __forceinline__ void err_reduce(double &se, double &sx, double &mx) {
    __shared__ double s_se[kErrThreads], s_sx[kErrThreads], s_mx[kErrThreads];
    const int t = threadIdx.x;
    s_se[t] = se; s_sx[t] = sx; s_mx[t] = mx;
    __syncthreads();
    static_assert(kErrThreads == 256, "the tree below");
    if (t >= 32) return;
    auto top = [&](const double *v, auto join) {
        const double a = join(v[t], v[t + 128]), b = join(v[t + 64], v[t + 192]);
        const double c = join(v[t + 32], v[t + 160]), e = join(v[t + 96], v[t + 224]);
        return join(join(a, b), join(c, e));
    };
    auto add = [](double a, double b) { return a + b; };
    auto most = [](double a, double b) { return fmax(a, b); };
    se = top(s_se, add);
    sx = top(s_sx, add);
    mx = top(s_mx, most);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        se += __shfl_down_sync(0xffffffffu, se, o);
        sx += __shfl_down_sync(0xffffffffu, sx, o);
        mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, o));
    }
}
// partial[b] = (sum (x - x_hat)^2, sum x^2, max |x - x_hat|) over the 8-element chunks b, b + grid, ...; four chunks of a
// thread are loaded before the first is used
__global__ void __launch_bounds__(kErrThreads) recon_error_kernel(const uint4 *X, const uint4 *Xh, long long n8,
                                                                  double *partial) {
    grid_dependency_wait();
    constexpr long long stride = (long long)kErrGrid * kErrThreads;
    ErrSum s = {0.0, 0.0, 0.f};
    for (long long i = blockIdx.x * (long long)kErrThreads + threadIdx.x; i < n8; i += 4 * stride) {
        uint4 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const long long at = i + u * stride < n8 ? i + u * stride : i;      // loads without a branch
            a[u] = X[at];
            b[u] = Xh[at];
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i + u * stride < n8) err_add(s, a[u], b[u]);
    }
    double mx = (double)s.mx;
    err_reduce(s.se, s.sx, mx);
    if (threadIdx.x == 0) {
        partial[3 * blockIdx.x + 0] = s.se;
        partial[3 * blockIdx.x + 1] = s.sx;
        partial[3 * blockIdx.x + 2] = mx;
    }
}
// one CTA adds the partial sums: each thread every 256th, then the same tree (one thread for all 592 took 63 us, this takes 4 us)
__global__ void __launch_bounds__(kErrThreads) recon_error_finalize_kernel(const double *partial, double *out) {
    grid_launch_dependents();
    grid_dependency_wait();
    double se = 0.0, sx = 0.0, mx = 0.0;
    for (int b = threadIdx.x; b < kErrGrid; b += kErrThreads) {
        se += partial[3 * b];
        sx += partial[3 * b + 1];
        mx = fmax(mx, partial[3 * b + 2]);
    }
    err_reduce(se, sx, mx);
    if (threadIdx.x == 0) { out[0] = se; out[1] = sx; out[2] = mx; }
}

// Launches a form of calib_kernel: `ctas` CTAs per chunk of 1024 channels.
template <bool MOMENTS>
static int launch_calib(const CodecParams &p, int ctas, cudaStream_t stream) {
    constexpr CalSmem L = cal_smem_layout(MOMENTS);
    DeviceInfo di;
    int dev = 0, occ = 0;
    int rc = device_info(&di, &dev);
    if (rc != RAC_OK) return rc;
    if (L.total > di.max_smem_optin) return RAC_EUNSUPPORTED;
    rc = resident_ctas(reinterpret_cast<const void *>(calib_kernel<MOMENTS>), dev, kCalWarps * 32, L.total, &occ);
    if (rc != RAC_OK) return rc;
    const int chunks = cal_chunks(p.d);
    if (ctas == 0) {      // as many as are resident at once, and no more than there are tokens for
        ctas = di.sms * occ / chunks;
        const long long most = (p.T + kCalWarps - 1) / kCalWarps;
        if (ctas > most) ctas = (int)most;
        if (ctas < 1) ctas = 1;
    }
    launch_after(calib_kernel<MOMENTS>, (unsigned)(ctas * chunks), kCalWarps * 32, L.total, stream, p, chunks);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

}  // namespace rac

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
using namespace rac;

extern "C" {

size_t rac_fit_segments_workspace_bytes(const rac_codec_cfg *cfg, int64_t T) {
    Geometry g;
    if (make_geometry(cfg, &g) != RAC_OK || T < 0) return 0;
    return ((size_t)T * (size_t)g.J * sizeof(float4) + 15) / 16 * 16 + 16;
}

int rac_fit_segments(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                     const int32_t *ref_row, const void *ref_gain, const void *ref_bias, const int32_t *seg_off,
                     int64_t n_seg, uint32_t *coef_seg, int32_t *seg_of, void *workspace, size_t workspace_bytes,
                     uint32_t *dev_status, void *stream) {
    Geometry g;
    int rc = make_geometry(cfg, &g);
    if (rc != RAC_OK) return rc;
    CodecParams p = {};
    rc = fill_common(g, &p, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, dev_status);
    if (rc != RAC_OK) return rc;
    if (n_seg < 0 || n_seg >= (1ll << 30) || T >= (1ll << 31)) return RAC_EUNSUPPORTED;
    if (n_seg == 0) return T == 0 ? RAC_OK : RAC_EINVAL;
    if (!seg_off || !coef_seg || !workspace || (T > 0 && (!X || !seg_of))) return RAC_EINVAL;
    if (!aligned16(X) || !aligned16(workspace)) return RAC_EALIGN;
    if (workspace_bytes < rac_fit_segments_workspace_bytes(cfg, T)) return RAC_ESIZE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p.X = static_cast<const uint16_t *>(X);
    p.moments = static_cast<float4 *>(workspace);
    if (T > 0) {
        rc = launch_calib<true>(p, 0, st);
        if (rc != RAC_OK) return rc;
        launch_after(seg_of_kernel, (unsigned)((T + 255) / 256), 256, 0, st, seg_off, (long long)n_seg, (long long)T, seg_of);
    }
    const long long warps = n_seg * g.J;
    launch_after(segment_fit_kernel, (unsigned)((warps * 32 + 255) / 256), 256, 0, st, p.moments, seg_off, (long long)n_seg, g.J,
                 g.group, (long long)T, coef_seg);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

size_t rac_recon_error_workspace_bytes(void) { return (size_t)kErrGrid * 3 * sizeof(double); }

int rac_recon_error(const void *X, const void *X_hat, int64_t T, int32_t d, double *out, void *workspace,
                    size_t workspace_bytes, void *stream) {
    if (T < 0 || d <= 0 || !out || !workspace) return RAC_EINVAL;
    if (d % 8) return RAC_EUNSUPPORTED;
    if (T > 0 && (!X || !X_hat)) return RAC_EINVAL;
    if (!aligned16(X) || !aligned16(X_hat) || !aligned16(workspace) || (reinterpret_cast<uintptr_t>(out) & 7u)) return RAC_EALIGN;
    if (workspace_bytes < rac_recon_error_workspace_bytes()) return RAC_ESIZE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double *partial = static_cast<double *>(workspace);
    launch_after(recon_error_kernel, kErrGrid, kErrThreads, 0, st, static_cast<const uint4 *>(X), static_cast<const uint4 *>(X_hat),
                 (long long)T * d / 8, partial);
    launch_after(recon_error_finalize_kernel, 1, kErrThreads, 0, st, partial, out);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

size_t rac_calibrate_workspace_bytes(const rac_codec_cfg *cfg) {
    Geometry g;
    if (make_geometry(cfg, &g) != RAC_OK) return 0;
    return (size_t)kCalParts * 2 * (size_t)g.d * sizeof(float) + (size_t)kCalParts * 2 * sizeof(int);
}

static int calibrate_impl(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                          const int32_t *ref_row, const void *ref_gain, const void *ref_bias, const uint32_t *coef_seg,
                          const int32_t *seg_of, float clip_sigmas, float *step, float *inv_step, void *workspace,
                          size_t workspace_bytes, uint32_t *dev_status, void *stream) {
    Geometry g;
    int rc = make_geometry(cfg, &g);
    if (rc != RAC_OK) return rc;
    CodecParams p = {};
    rc = fill_common(g, &p, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, dev_status);
    if (rc != RAC_OK) return rc;
    if (g.scale_mode != 0) return RAC_EUNSUPPORTED;   // the tables belong to the static quantiser only
    if ((g.coef_fmt == 1) != (coef_seg != nullptr) || (coef_seg != nullptr) != (seg_of != nullptr)) return RAC_EINVAL;
    p.coef_ext = coef_seg;
    p.seg_of = seg_of;
    if (!step || !inv_step || !workspace || !(clip_sigmas > 0.f)) return RAC_EINVAL;
    if (T > 0 && !X) return RAC_EINVAL;
    if (!aligned16(X) || !aligned16(workspace) || !aligned16(step) || !aligned16(inv_step)) return RAC_EALIGN;
    if (workspace_bytes < rac_calibrate_workspace_bytes(cfg)) return RAC_ESIZE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    p.X = static_cast<const uint16_t *>(X);
    p.calib_partial = static_cast<float *>(workspace);
    // every CTA of the fixed grid writes its partials, also when it has no token
    const int parts = cal_parts(g.d);
    rc = launch_calib<false>(p, parts, st);
    if (rc != RAC_OK) return rc;
    launch_after(calib_finalize_kernel, (unsigned)(2 * g.d / 32), 32 * kFinSlices, 0, st, p.calib_partial, parts, g.d, g.bits,
                 clip_sigmas, step, inv_step);
    return cudaGetLastError() == cudaSuccess ? RAC_OK : RAC_ECUDA;
}

int rac_calibrate_steps(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                        const int32_t *ref_row, const void *ref_gain, const void *ref_bias, float clip_sigmas,
                        float *step, float *inv_step, void *workspace, size_t workspace_bytes, uint32_t *dev_status,
                        void *stream) {
    return calibrate_impl(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, nullptr, nullptr, clip_sigmas, step,
                          inv_step, workspace, workspace_bytes, dev_status, stream);
}

int rac_calibrate_steps_shared(const rac_codec_cfg *cfg, const void *X, int64_t T, const void *ref_base, int64_t ref_rows,
                               const int32_t *ref_row, const void *ref_gain, const void *ref_bias,
                               const uint32_t *coef_seg, const int32_t *seg_of, float clip_sigmas, float *step,
                               float *inv_step, void *workspace, size_t workspace_bytes, uint32_t *dev_status,
                               void *stream) {
    if (!coef_seg || !seg_of) return RAC_EINVAL;
    return calibrate_impl(cfg, X, T, ref_base, ref_rows, ref_row, ref_gain, ref_bias, coef_seg, seg_of, clip_sigmas, step,
                          inv_step, workspace, workspace_bytes, dev_status, stream);
}

}  // extern "C"
