// Three-channel first layer (7x7, stride 2, pad 3), whole output rows at a time, optionally fused with the 3x3 / stride-2 /
// pad-1 max-pool.
//
// conv_stem.cu builds the im2col operand of 128 pixels in shared memory: 90 KB of traffic per tile, more time than the
// MMAs take.  Here the operand is never built.  Input rows are stored with FOUR channels per pixel (the fourth zero), 8
// bytes each, so that output column q (stride 2) starts 16 q bytes into a row: eight consecutive columns are one core
// matrix of the unswizzled K-major layout, and the next two pixels of the window are the core matrix 16 bytes further on.
// The K-direction offset of the operand descriptor is therefore 16 bytes, core matrices overlap, and a kernel row is two
// MMAs (K = 32: eight pixels x four channels, the eighth pixel and the fourth channel meet zero weights) straight from the
// rows.  Widening a row costs one 16-byte store per two pixels, once per row instead of once per window.
//
// A CTA walks consecutive steps; a step is two output rows (2p, 2p + 1) of an image, i.e. one pooled row.
//   warps 0-3   input rows -> ring of widened rows (four new rows per step; loads run a step ahead)
//   warp 4      MMAs: per output row seven kernel rows x two, rows outside the image skipped, into one of two TMEM sets
//   warps 5-12  epilogue: bias, ReLU, one rounding; pooled: the running maximum with the row above (kept in registers from
//               the step before), through shared memory, then three columns to one and 16-byte stores along the row.
// Every pooled value is written once: no reductions in memory and nothing to clear first.  Every wait is bounded.
#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

using namespace tc;

namespace {

constexpr int kConvWarps = 4, kMmaWarp = kConvWarps, kFirstEpi = kConvWarps + 1, kEpiWarps = 8;
constexpr int kThreads = (kFirstEpi + kEpiWarps) * 32;
constexpr int kR = 7, kC = 3;
constexpr int kSlots = 24;                         // rows of the ring: a window of nine, and up to nine of the next step
constexpr int kWindow = 9;                         // input rows under a step
constexpr uint32_t kSmemLimit = 232448;
constexpr uint32_t kDescHi = (128u >> 4) | (1u << 14);   // SBO = 128 bytes, descriptor version bit

struct StemRowsParams {
    int N, H, W, K, P, Q, Mb, relu, y_bf16;
    int PP, PQ, pairs, n_steps;                    // pooled height / width; pixel pairs of a row; steps in all (images x row pairs)
    int spi;                                       // steps per image
    uint32_t pitch, line, off_b, off_stage, stage_bytes, off_bias, off_bar, smem_bytes, tmem_cols;
};

struct StemRowsBars {
    uint64_t in_full[2], in_empty[2], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
    uint32_t abort_flag;
};

__device__ __forceinline__ uint64_t desc64(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint4 max4(const uint4 &a, const uint4 &b)
{
    return make_uint4(max_bf16x2(a.x, b.x), max_bf16x2(a.y, b.y), max_bf16x2(a.z, b.z), max_bf16x2(a.w, b.w));
}
// barrier among the epilogue warps with a vote: true when every one of their threads says so
__device__ __forceinline__ bool epi_all(bool ok)
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %2, 0;\n\tbar.red.and.pred p, 1, %1, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(r) : "n"(kEpiWarps * 32), "r"((uint32_t)ok) : "memory");
    return r != 0u;
}

// The steps of a CTA in order.  `warm`: the step before the first one of an image's inside, computed for the row it hands
// on and not stored.
struct Steps {
    int at, end, spi;
    bool first, pool;
    int n, p;
    bool reset, store;
    __device__ Steps(int lo, int hi, int spi_, bool pool_) : at(lo), end(hi), spi(spi_), first(true), pool(pool_), n(0), p(0), reset(false), store(false) {}
    __device__ bool next()
    {
        if (at >= end) return false;
        n = at / spi; p = at - n * spi;
        if (first && pool && p > 0) { p -= 1; first = false; reset = true; store = false; return true; }
        reset = first || p == 0;
        first = false; store = true;
        ++at;
        return true;
    }
};

template <bool kPool>
__global__ void __launch_bounds__(kThreads, 1)
conv_stem_rows_kernel(const StemRowsParams p, const uint16_t *__restrict__ x, const uint8_t *__restrict__ blob,
                      const float *__restrict__ bias, void *__restrict__ y, uint32_t *ws)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *ring = smem;                             // [kSlots] rows of `pitch` bytes: pixel x at 8 (x + 3)
    uint8_t *bsm = smem + p.off_b;                    // [7 kernel rows][4 octets][K filters][8] bf16
    float *bias_s = reinterpret_cast<float *>(smem + p.off_bias);
    StemRowsBars *bars = reinterpret_cast<StemRowsBars *>(smem + p.off_bar);
    volatile uint32_t *abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lo = (int)((long long)p.n_steps * blockIdx.x / gridDim.x), hi = (int)((long long)p.n_steps * (blockIdx.x + 1) / gridDim.x);

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->in_full[s], kConvWarps); mbar_init(&bars->in_empty[s], 1);
            mbar_init(&bars->acc_full[s], 1); mbar_init(&bars->acc_empty[s], kEpiWarps);
        }
        bars->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    pdl_trigger();
    // borders of the ring's rows and the operand's unused places: zeros, once
    for (uint32_t o = tid * 16; o < p.off_stage; o += kThreads * 16) *reinterpret_cast<uint4 *>(smem + o) = make_uint4(0, 0, 0, 0);
    __syncthreads();
    {
        // weight of (tap (r, s), channel c, filter n) at k = s * 4 + c of kernel row r.  (The blob is never written by a
        // kernel that lets its successor start early: no need to wait for the kernel before this one.)
        const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
        const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_BLK]);
        const uint32_t *pairs = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
        const uint16_t *values = reinterpret_cast<const uint16_t *>(blob + hdr[BP_OFF_VALUES]);
        const int per_pair = p.Mb * kC;
        for (int fb = 0; fb < p.K / p.Mb; ++fb) {
            const uint32_t j0 = blk_off[fb], n = (blk_off[fb + 1] - j0) * per_pair;       // one channel block per filter block
#pragma unroll 4
            for (uint32_t e = tid; e < n; e += kThreads) {
                const uint32_t j = j0 + e / per_pair, rem = e % per_pair, f = rem / kC, c = rem - f * kC;
                const uint32_t tap = pairs[j] >> 16, r = tap / kR, sx = tap - r * kR;
                const uint16_t v = values[(size_t)j * per_pair + rem];
                const uint32_t kk = sx * 4 + c;
                if (r < (uint32_t)kR)                                                        // (not a 7x7 tap: ignored)
                    *reinterpret_cast<uint16_t *>(bsm + (((size_t)r * 4 + (kk >> 3)) * p.K + fb * p.Mb + f) * 16 + (kk & 7) * 2) = v;
            }
        }
    }
    pdl_wait();
    for (int i = tid; i < p.K; i += kThreads) bias_s[i] = bias ? bias[i] : 0.f;
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;

    if (warp < kConvWarps) {
        // ---- input rows: thread u widens pixel pair u, i.e. padded pixels 2u and 2u + 1 = input pixels 2u - 3 and 2u - 2,
        // twelve bytes that start two bytes before a word boundary ------------------------------------------------------
        const int words_in = 3 * p.W / 2, u = tid, g = 3 * u - 5;            // first word of the twelve (and two) bytes
        const bool on = u < p.pairs;
        const uint32_t *x32 = reinterpret_cast<const uint32_t *>(x);
        // rows w .. w + 3 of the window of (image n, first row y_lo): requested together
        auto request = [&](uint32_t (&a)[4][4], int n, int y_lo, int w) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int yy = y_lo + w + q;
                const bool in = on && w + q < kWindow && yy >= 0 && yy < p.H;
                const uint32_t *row = x32 + ((size_t)n * p.H + (in ? yy : 0)) * words_in;
#pragma unroll
                for (int k = 0; k < 4; ++k) a[q][k] = in && g + k >= 0 && g + k < words_in ? __ldg(row + g + k) : 0u;
            }
        };
        auto widen = [&](const uint32_t (&a)[4][4], uint32_t base, int w) {
            if (!on) return;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (w + q >= kWindow) break;
                uint32_t slot = base + (uint32_t)(w + q);
                if (slot >= (uint32_t)kSlots) slot -= kSlots;
                // six elements e0 .. e5 = bytes 2 .. 13 of the four words
                const uint32_t e01 = __funnelshift_r(a[q][0], a[q][1], 16), e23 = __funnelshift_r(a[q][1], a[q][2], 16),
                               e45 = __funnelshift_r(a[q][2], a[q][3], 16);
                *reinterpret_cast<uint4 *>(ring + slot * p.pitch + (uint32_t)u * 16u) =
                    make_uint4(e01, e23 & 0xFFFFu, (e23 >> 16) | (e45 << 16), e45 >> 16);
            }
        };
        Steps st(lo, hi, p.spi, kPool);
        uint32_t i = 0, base = 0, next[4][4];                                // step count; ring slot of the window's first row
        bool more = st.next();
        if (more) request(next, st.n, 4 * st.p - 3, kWindow - 4);           // the four rows every step brings, a step ahead
        while (more) {
            const int y_lo = 4 * st.p - 3;
            base = st.reset ? (i ? base + kWindow : 0u) : base + 4u;
            if (base >= (uint32_t)kSlots) base -= kSlots;
            if (i >= 2 && !mbar_wait(&bars->in_empty[i & 1u], ((i >> 1) & 1u) ^ 1u, abort_flag, ws, 0xB100)) break;
            if (st.reset) {                                                  // the other five rows of the window
                uint32_t a[4][4], b2[4][4];
                request(a, st.n, y_lo, 0);
                request(b2, st.n, y_lo, 1);
                widen(a, base, 0);
                widen(b2, base, 1);
            }
            widen(next, base, kWindow - 4);
            more = st.next();
            if (more) request(next, st.n, 4 * st.p - 3, kWindow - 4);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->in_full[i & 1u]);
            ++i;
        }
    } else if (warp == kMmaWarp) {
        // ---- MMAs ------------------------------------------------------------------------------------------------------
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16_f32(128, p.K);
            const uint32_t ring16 = (smem_u32(ring) >> 4) | (1u << 16), pitch16 = p.pitch >> 4;      // K-direction offset: 16 bytes
            const uint32_t b16 = (smem_u32(bsm) >> 4) | ((uint32_t)p.K << 16), brow16 = 4u * p.K;
            Steps st(lo, hi, p.spi, kPool);
            uint32_t i = 0, base = 0;
            bool ok = true;
            while (ok && st.next()) {
                base = st.reset ? (i ? base + kWindow : 0u) : base + 4u;
                if (base >= (uint32_t)kSlots) base -= kSlots;
                const uint32_t b = i & 1u, ph = (i >> 1) & 1u;
                if (i >= 2 && !mbar_wait(&bars->acc_empty[b], ph ^ 1u, abort_flag, ws, 0xB200)) break;
                if (!mbar_wait(&bars->in_full[b], ph, abort_flag, ws, 0xB210)) break;
                tc_fence_after_sync();
                for (int j = 0; j < 2; ++j) {
                    const uint32_t d = tmem_base + (b * 2u + j) * p.K;
                    const int y0 = 2 * (2 * st.p + j) - 3;                  // input row under kernel row 0
                    uint32_t acc = 0;
                    for (int r = 0; r < kR; ++r) {
                        if (y0 + r < 0 || y0 + r >= p.H) continue;           // zero padding
                        uint32_t slot = base + 2u * j + r;
                        if (slot >= (uint32_t)kSlots) slot -= kSlots;
                        const uint32_t a_lo = ring16 + slot * pitch16, b_lo = b16 + r * brow16;
                        mma_bf16_ss(d, desc64(a_lo), desc64(b_lo), idesc, acc);
                        mma_bf16_ss(d, desc64(a_lo + 2u), desc64(b_lo + 2u * p.K), idesc, 1u);
                        acc = 1u;
                    }
                }
                mma_commit(&bars->in_empty[b]);
                mma_commit(&bars->acc_full[b]);
                ++i;
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: warp -> TMEM lane quarter and every second 16-column chunk -----------------------------------------
        const int quarter = warp & 3, part = (warp - kFirstEpi) >> 2, q = quarter * 32 + lane, et = tid - kFirstEpi * 32;
        const int nch = p.K / 16;
        constexpr int kMaxOwn = 4;                       // chunks per warp (K <= 128)
        uint32_t saved[kMaxOwn][8];                      // the row above, packed
#pragma unroll
        for (int c = 0; c < kMaxOwn; ++c)
#pragma unroll
            for (int k = 0; k < 8; ++k) saved[c][k] = 0u;
        Steps st(lo, hi, p.spi, kPool);
        uint32_t i = 0;
        bool ok = true;
        while (st.next()) {
            const uint32_t b = i & 1u;
            uint8_t *stage = smem + p.off_stage + (kPool ? (size_t)b * p.stage_bytes : 0u);
            if (kPool && st.p == 0) {
#pragma unroll
                for (int c = 0; c < kMaxOwn; ++c)
#pragma unroll
                    for (int k = 0; k < 8; ++k) saved[c][k] = 0u;            // (nothing is negative after ReLU)
            }
            ok = mbar_wait(&bars->acc_full[b], (i >> 1) & 1u, abort_flag, ws, 0xB400);
            if (!__all_sync(0xFFFFFFFFu, ok)) ok = false;
            tc_fence_after_sync();
            const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + b * 2u * p.K;
#pragma unroll
            for (int c = 0; c < kMaxOwn; ++c) {
                const int ch = part + 2 * c;
                if (ch >= nch || !ok) break;
                uint32_t r0[16], r1[16];
                tmem_ld_x16(t_addr + ch * 16, r0);
                tmem_ld_x16(t_addr + p.K + ch * 16, r1);
                tmem_ld_wait();
                uint32_t o0[8], o1[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float b0 = bias_s[ch * 16 + 2 * k], b1 = bias_s[ch * 16 + 2 * k + 1];
                    o0[k] = cvt_bf16x2(__uint_as_float(r0[2 * k]) + b0, __uint_as_float(r0[2 * k + 1]) + b1);
                    o1[k] = cvt_bf16x2(__uint_as_float(r1[2 * k]) + b0, __uint_as_float(r1[2 * k + 1]) + b1);
                    if (p.relu) { o0[k] = relu_bf16x2(o0[k]); o1[k] = relu_bf16x2(o1[k]); }
                }
                if constexpr (kPool) {
                    // rows 2p - 1, 2p, 2p + 1 (the last one may not exist)
                    const bool has1 = 2 * st.p + 1 < p.P;
                    uint32_t m[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        m[k] = max_bf16x2(saved[c][k], o0[k]);
                        if (has1) m[k] = max_bf16x2(m[k], o1[k]);
                        saved[c][k] = o1[k];
                    }
                    // one line of 2 K bytes per column, 16-byte units XOR-ed with the column (conflict free)
                    uint8_t *line = stage + (size_t)q * p.line;
                    const uint32_t x7 = (uint32_t)(q & 7);
                    *reinterpret_cast<uint4 *>(line + (((uint32_t)(2 * ch) ^ x7) << 4)) = make_uint4(m[0], m[1], m[2], m[3]);
                    *reinterpret_cast<uint4 *>(line + (((uint32_t)(2 * ch + 1) ^ x7) << 4)) = make_uint4(m[4], m[5], m[6], m[7]);
                } else if (q < p.Q) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int row = 2 * st.p + j;
                        if (row >= p.P) continue;
                        const size_t o = (((size_t)st.n * p.P + row) * p.Q + q) * p.K + ch * 16;
                        if (p.y_bf16) {
                            uint4 *yp = reinterpret_cast<uint4 *>(static_cast<uint16_t *>(y) + o);
                            const uint32_t *v = j ? o1 : o0;
                            yp[0] = make_uint4(v[0], v[1], v[2], v[3]);
                            yp[1] = make_uint4(v[4], v[5], v[6], v[7]);
                        } else {
                            float4 *yp = reinterpret_cast<float4 *>(static_cast<float *>(y) + o);
                            const uint32_t *v = j ? r1 : r0;
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                float f[4];
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    f[k] = __uint_as_float(v[4 * h + k]) + bias_s[ch * 16 + 4 * h + k];
                                    if (p.relu) f[k] = fmaxf(f[k], 0.f);
                                }
                                yp[h] = make_float4(f[0], f[1], f[2], f[3]);
                            }
                        }
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->acc_empty[b]);
            if constexpr (kPool) {
                if (!epi_all(ok)) break;                 // (the staged row is complete; all eight warps go on, or stop, as one)
                if (st.store) {
                    // pooled column v = columns 2v - 1, 2v, 2v + 1
                    const int units = p.K / 8;
                    uint16_t *out = static_cast<uint16_t *>(y) + ((size_t)st.n * p.PP + st.p) * p.PQ * p.K;
                    for (int e = et; e < p.PQ * units; e += kEpiWarps * 32) {
                        const int v = e / units, u = e - v * units, c0 = 2 * v;
                        auto at = [&](int col) { return *reinterpret_cast<const uint4 *>(stage + (size_t)col * p.line + (((uint32_t)u ^ (uint32_t)(col & 7)) << 4)); };
                        uint4 m = at(c0);
                        if (c0 > 0) m = max4(m, at(c0 - 1));
                        if (c0 + 1 < p.Q) m = max4(m, at(c0 + 1));
                        *reinterpret_cast<uint4 *>(out + (size_t)v * p.K + u * 8) = m;
                    }
                }
            } else if (!ok) break;
            ++i;
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, p.tmem_cols);
    }
}

bool plan(const npas_conv_desc &d, const npas_bp_desc &bp, StemRowsParams &p, bool pool)
{
    if (d.x_dtype != NPAS_BF16 || bp.w_packed != NPAS_BF16) return false;
    if (d.C != kC || bp.Nb != kC || d.R != kR || d.S != kR || d.stride != 2 || d.pad != 3) return false;
    if (d.has_residual || d.K % 16 || d.K > 128 || d.K % bp.Mb || d.W % 2) return false;
    p.N = d.N; p.H = d.H; p.W = d.W; p.K = d.K; p.Mb = bp.Mb;
    p.P = (d.H + 2 * d.pad - d.R) / 2 + 1; p.Q = (d.W + 2 * d.pad - d.S) / 2 + 1;
    if (p.P < 1 || p.Q < 1 || p.Q > 128) return false;         // a whole output row is one MMA tile
    p.relu = d.relu; p.y_bf16 = d.y_dtype == NPAS_BF16;
    if (pool && (!d.relu || !p.y_bf16)) return false;          // (the running maximum starts from zero, on packed bf16 pairs)
    p.PP = (p.P - 1) / 2 + 1; p.PQ = (p.Q - 1) / 2 + 1;
    p.spi = (p.P + 1) / 2;                                     // = PP
    const long long steps = (long long)d.N * p.spi;
    if (steps > 0x3FFFFFFF) return false;
    p.n_steps = (int)steps;
    p.pairs = p.Q + 3;
    p.pitch = round_up((uint32_t)p.pairs * 16u, 128);
    p.line = round_up(2u * d.K, 128);
    p.off_b = kSlots * p.pitch + 1024u;                        // (an operand reads 128 columns, past the end of the last row)
    p.off_stage = round_up(p.off_b + (uint32_t)kR * 4u * d.K * 16u, 128);
    p.stage_bytes = 128u * p.line;
    p.off_bias = p.off_stage + (pool ? 2u * p.stage_bytes : 0u);
    p.off_bar = round_up(p.off_bias + d.K * 4u, 128);
    p.smem_bytes = p.off_bar + (uint32_t)sizeof(StemRowsBars) + 1024u;
    if (p.smem_bytes > kSmemLimit) return false;
    p.tmem_cols = 32;
    while ((int)p.tmem_cols < 4 * d.K) p.tmem_cols *= 2;
    return true;
}

}  // namespace

bool conv_stem_rows_supported(const npas_conv_desc &d, const npas_bp_desc &bp, bool pool)
{
    StemRowsParams p;
    return plan(d, bp, p, pool);
}

npas_status conv_stem_rows_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x, const void *blob, const float *bias,
                                  void *y, uint32_t *ws, cudaStream_t st, bool pool)
{
    StemRowsParams p;
    if (!plan(d, bp, p, pool)) return NPAS_ERR_UNSUPPORTED;
    auto go = [&](auto kernel) {
        if (allow_dynamic_smem(reinterpret_cast<const void *>(kernel), (int)kSmemLimit) != NPAS_OK) return cudaErrorUnknown;
        const int sms = sm_count(), grid = p.n_steps < sms ? p.n_steps : sms;
        return launch_pdl(kernel, dim3(grid), dim3(kThreads), p.smem_bytes, st, p, static_cast<const uint16_t *>(x),
                          static_cast<const uint8_t *>(blob), bias, y, ws);
    };
    const cudaError_t e = pool ? go(conv_stem_rows_kernel<true>) : go(conv_stem_rows_kernel<false>);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // namespace npas
