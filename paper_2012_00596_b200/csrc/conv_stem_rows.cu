// Three-channel first layer (7x7, stride 2, pad 3), whole output rows at a time, optionally fused with the 3x3 / stride-2 /
// pad-1 max-pool.
//
// conv_stem.cu builds the im2col operand of 128 pixels in shared memory: 90 KB of traffic per tile, more time than the
// MMAs take.  Here the operand is never built.  Input rows are stored with FOUR channels per pixel (the fourth is one), 8
// bytes each, so that output column q (stride 2) starts 16 q bytes into a row: eight consecutive columns are one core
// matrix of the unswizzled K-major layout, and the next two pixels of the window are the core matrix 16 bytes further on.
// The K-direction offset of the operand descriptor is therefore 16 bytes, core matrices overlap, and a kernel row is two
// MMAs (K = 32: eight pixels x four channels, the fourth channel meets the bias) straight from the rows.  Widening a row costs
// one 16-byte store per two pixels, once per row instead of once per window.
//
// The eighth pixel lies outside the window and its weights are zero, but zero times an infinity is not: the second MMA's second
// core matrix (pixels seven and eight) is read from a copy of the row in which the second pixel of every pair is zero, by a
// K-direction offset from one row to the other.  That costs 8 more bytes stored per two pixels, and no more operand reads.
//
// Shared memory is what bounds it (an MMA of K filters reads 4 KB of rows and 32 K bytes of weights, three times what its
// arithmetic takes), so the two output rows of a step share their operand: input row t of the window is kernel row t of the
// first and t - 2 of the second, and with the kernel rows of one parity stored in falling order the two filter sets are one
// operand of 2 K columns.  18 operand reads per step instead of 28.
//
// A CTA walks consecutive steps; a step is two output rows (2p, 2p + 1) of an image, i.e. one pooled row.
//   warps 0-3   input rows -> ring of widened rows (four new rows per step; loads run a step ahead)
//   warp 4      MMAs: nine input rows x two, rows outside the image are zeros, into one of two TMEM sets
//   warps 5-12  epilogue: ReLU, one rounding; pooled: after the maximum with the row above (kept in registers from
//               the step before: all of it is monotone, so one rounding serves the three rows), into one of two stages
//   warps 13-15 (pooled) three staged columns to one, 16-byte stores along the row.  Warps of their own: these loads queue
//               behind the operand reads of the MMAs, and the accumulators waited for them (1.8 k of 3.6 k clocks a step).
// 64 x 224 x 224, K = 64, pooled, launches back to back in a captured graph: 40.8 us (40.6 without the copy of the rows; 63 with
// separate operand reads, the bias from shared memory and pooling by the epilogue's warps).
// Every pooled value is written once: no reductions in memory and nothing to clear first.  Every wait is bounded.
#include <type_traits>

#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

using namespace tc;

namespace {

constexpr int kConvWarps = 4, kMmaWarp = kConvWarps, kFirstEpi = kConvWarps + 1, kEpiWarps = 8;
constexpr int kFirstPool = kFirstEpi + kEpiWarps, kPoolWarps = 3;
template <bool kPool> constexpr int kThreads = (kFirstPool + (kPool ? kPoolWarps : 0)) * 32;
constexpr int kR = 7, kC = 3;
constexpr int kSlots = 18;                         // rows of the ring: a window of nine, and up to nine of the next step
constexpr int kWindow = 9;                         // input rows under a step
constexpr uint32_t kOne = 0x3F800000u;              // bf16 one as the second of a pair
constexpr uint32_t kSmemLimit = 232448;
constexpr uint32_t kDescHi = (128u >> 4) | (1u << 14);   // SBO = 128 bytes, descriptor version bit

struct StemRowsParams {
    int N, H, W, K, P, Q, Mb, relu, y_bf16, early;  // early: the blob may be read before the wait (Launch::blob_ready)
    int PP, PQ, pairs, n_steps;                    // pooled height / width; pixel pairs of a row; steps in all (images x row pairs)
    int spi;                                       // steps per image
    uint32_t pitch, off_z, line, off_b, off_stage, stage_bytes, off_bar, smem_bytes, tmem_cols;
};

struct StemRowsBars {
    uint64_t in_full[2], in_empty[2], acc_full[2], acc_empty[2], stage_full[2], stage_empty[2];
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
__global__ void __launch_bounds__(kThreads<kPool>, 1)
conv_stem_rows_kernel(const StemRowsParams p, const uint16_t *__restrict__ x, const uint8_t *__restrict__ blob,
                      const float *__restrict__ bias, void *__restrict__ y, uint32_t *ws)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *ring = smem;                             // [kSlots] rows of `pitch` bytes: pixel x at 8 (x + 3); off_z further the same, odd x only
    uint8_t *bsm = smem + p.off_b;                    // [parity of the kernel row][4 octets][4 K: (6 | 5 - r) / 2, filter][8] bf16
    StemRowsBars *bars = reinterpret_cast<StemRowsBars *>(smem + p.off_bar);
    volatile uint32_t *abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lo = (int)((long long)p.n_steps * blockIdx.x / gridDim.x), hi = (int)((long long)p.n_steps * (blockIdx.x + 1) / gridDim.x);

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&bars->in_full[s], kConvWarps); mbar_init(&bars->in_empty[s], 1);
            mbar_init(&bars->acc_full[s], 1); mbar_init(&bars->acc_empty[s], kEpiWarps);
            mbar_init(&bars->stage_full[s], kEpiWarps); mbar_init(&bars->stage_empty[s], kPoolWarps);
        }
        bars->abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    pdl_trigger();
    // borders of the ring's rows and the operand's unused places: zeros, once
    for (uint32_t o = tid * 16; o < p.off_stage; o += kThreads<kPool> * 16) *reinterpret_cast<uint4 *>(smem + o) = make_uint4(0, 0, 0, 0);
    __syncthreads();
    {
        // weight of (tap (r, s), channel c, filter n) at k = s * 4 + c of kernel row r
        if (!p.early) pdl_wait();
        blob = behind_wait(blob);
        const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
        const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_BLK]);
        const uint32_t *pairs = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
        const uint16_t *values = reinterpret_cast<const uint16_t *>(blob + hdr[BP_OFF_VALUES]);
        const uint32_t per_pair = p.Mb * kC, nfb = p.K / p.Mb;
        auto put = [&](uint32_t tap, uint32_t n, uint32_t c, uint16_t v) {
            const uint32_t r = tap / kR, kk = (tap - r * kR) * 4 + c;
            if (r < (uint32_t)kR)                                                            // (not a 7x7 tap: ignored)
                *reinterpret_cast<uint16_t *>(bsm + ((((r & 1) * 4 + (kk >> 3)) * 4 + ((6 - r) >> 1)) * p.K + n) * 16 + (kk & 7) * 2) = v;
        };
        if (per_pair % 8 == 0) {
            // eight weights of a pair per thread: one load, no division per weight
            const uint32_t upp = per_pair / 8, n_units = __ldg(blk_off + nfb) * upp;
            for (uint32_t e = tid; e < n_units; e += kThreads<kPool>) {
                const uint32_t j = e / upp, rem = (e - j * upp) * 8, tap = __ldg(pairs + j) >> 16;
                const uint4 q = __ldg(reinterpret_cast<const uint4 *>(values + (size_t)j * per_pair + rem));
                uint32_t fb = 0;
                while (fb + 1 < nfb && __ldg(blk_off + fb + 1) <= j) ++fb;                           // one channel block per filter block
                const uint32_t v[4] = {q.x, q.y, q.z, q.w};
                uint32_t f = rem / kC, c = rem - f * kC;
                f += fb * p.Mb;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    put(tap, f, c, (uint16_t)(v[k >> 1] >> (16 * (k & 1))));
                    if (++c == (uint32_t)kC) { c = 0; ++f; }
                }
            }
        } else {
            for (uint32_t fb = 0; fb < nfb; ++fb) {
                const uint32_t j0 = blk_off[fb], n = (blk_off[fb + 1] - j0) * per_pair;
                for (uint32_t e = tid; e < n; e += kThreads<kPool>) {
                    const uint32_t j = j0 + e / per_pair, rem = e % per_pair, f = rem / kC;
                    put(__ldg(pairs + j) >> 16, fb * p.Mb + f, rem - f * kC, __ldg(values + (size_t)j * per_pair + rem));
                }
            }
        }
    }
    pdl_wait();
    x = behind_wait(x); bias = behind_wait(bias);
    // bias: the fourth channel of every pixel is one, and a window's pixels 2 .. 4 of kernel row 3 (never outside the image)
    // weigh it with the bias' upper, middle and lower eight bits, so that the sum is exact
    for (int f = tid; bias && f < p.K; f += kThreads<kPool>) {
        const float v = __ldg(bias + f);
        const bool finite = fabsf(v) <= 3.0e38f;
        const uint32_t hi16 = finite ? __float_as_uint(v) >> 16 : cvt_bf16x2(v, 0.f) & 0xFFFFu;
        const float rest = finite ? v - __uint_as_float(hi16 << 16) : 0.f;
        const uint32_t mid16 = __float_as_uint(rest) >> 16, lo16 = __float_as_uint(rest - __uint_as_float(mid16 << 16)) >> 16;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t kk = 4 * (2 + k) + 3;
            *reinterpret_cast<uint16_t *>(bsm + (((4 + (kk >> 3)) * 4 + 1) * p.K + f) * 16 + (kk & 7) * 2) = (uint16_t)(k == 0 ? hi16 : k == 1 ? mid16 : lo16);
        }
    }
    fence_proxy_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;

    if (warp < kConvWarps) {
        // ---- input rows: thread u - 1 widens pixel pair u, i.e. padded pixels 2u and 2u + 1 = input pixels 2u - 3 and 2u - 2,
        // twelve bytes that start two bytes before a word boundary.  (Pair 0 is padding; rows of 128 columns have one pair
        // more than there are threads, the last pixel and padding: four threads take one row's each.) --------------------
        const int words_in = 3 * p.W / 2, u = tid + 1, g = 3 * u - 5;        // first word of the twelve (and two) bytes
        const bool on = u < p.pairs, tail = p.Q == kConvWarps * 32 && tid < 4;
        const uint32_t *x32 = reinterpret_cast<const uint32_t *>(x);
        // rows w .. w + 3 of the window of (image n, first row y_lo): requested together
        auto request = [&](uint32_t (&a)[4][4], uint2 &last, int n, int y_lo, int w) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int yy = y_lo + w + q;
                const bool in = on && w + q < kWindow && yy >= 0 && yy < p.H;
                const uint32_t *row = x32 + ((size_t)n * p.H + (in ? yy : 0)) * words_in;
#pragma unroll
                for (int k = 0; k < 4; ++k) a[q][k] = in && g + k >= 0 && g + k < words_in ? __ldg(row + g + k) : 0u;
            }
            last = make_uint2(0u, 0u);
            if (tail && w + tid < kWindow && y_lo + w + tid >= 0 && y_lo + w + tid < p.H) {
                const uint32_t *end = x32 + ((size_t)n * p.H + y_lo + w + tid + 1) * words_in;
                last = make_uint2(__ldg(end - 2), __ldg(end - 1));
            }
        };
        auto widen = [&](const uint32_t (&a)[4][4], const uint2 &last, uint32_t base, int w) {
            if (tail && w + tid < kWindow) {
                uint32_t slot = base + (uint32_t)(w + tid);
                if (slot >= (uint32_t)kSlots) slot -= kSlots;
                uint8_t *at = ring + slot * p.pitch + (uint32_t)(p.Q + 1) * 16u;
                const uint32_t e01 = __funnelshift_r(last.x, last.y, 16), e2 = (last.y >> 16) | kOne;
                *reinterpret_cast<uint4 *>(at) = make_uint4(e01, e2, 0u, kOne);
                *reinterpret_cast<uint2 *>(at + p.off_z) = make_uint2(e01, e2);
            }
            if (!on) return;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (w + q >= kWindow) break;
                uint32_t slot = base + (uint32_t)(w + q);
                if (slot >= (uint32_t)kSlots) slot -= kSlots;
                // six elements e0 .. e5 = bytes 2 .. 13 of the four words
                const uint32_t e01 = __funnelshift_r(a[q][0], a[q][1], 16), e23 = __funnelshift_r(a[q][1], a[q][2], 16),
                               e45 = __funnelshift_r(a[q][2], a[q][3], 16);
                uint8_t *at = ring + slot * p.pitch + (uint32_t)u * 16u;
                *reinterpret_cast<uint4 *>(at) = make_uint4(e01, (e23 & 0xFFFFu) | kOne, (e23 >> 16) | (e45 << 16), (e45 >> 16) | kOne);
                *reinterpret_cast<uint2 *>(at + p.off_z) = make_uint2(e01, (e23 & 0xFFFFu) | kOne);
            }
        };
        Steps st(lo, hi, p.spi, kPool);
        uint2 next_last, l0, l1;
        uint32_t i = 0, base = 0, next[4][4];                                // step count; ring slot of the window's first row
        bool more = st.next();
        if (more) request(next, next_last, st.n, 4 * st.p - 3, kWindow - 4);   // the four rows every step brings, a step ahead
        while (more) {
            const int y_lo = 4 * st.p - 3;
            base = st.reset ? (i ? base + kWindow : 0u) : base + 4u;
            if (base >= (uint32_t)kSlots) base -= kSlots;
            if (i >= 2 && !mbar_wait(&bars->in_empty[i & 1u], ((i >> 1) & 1u) ^ 1u, abort_flag, ws, 0xB100)) break;
            if (st.reset) {                                                  // the other five rows of the window
                uint32_t a[4][4], b2[4][4];
                request(a, l0, st.n, y_lo, 0);
                request(b2, l1, st.n, y_lo, 1);
                widen(a, l0, base, 0);
                widen(b2, l1, base, 1);
            }
            widen(next, next_last, base, kWindow - 4);
            more = st.next();
            if (more) request(next, next_last, st.n, 4 * st.p - 3, kWindow - 4);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->in_full[i & 1u]);
            ++i;
        }
    } else if (warp == kMmaWarp) {
        // ---- MMAs ------------------------------------------------------------------------------------------------------
        if (elect_one()) {
            const uint32_t idesc1 = idesc_bf16_f32(128, p.K), idesc2 = idesc_bf16_f32(128, 2 * p.K);
            const uint32_t ring16 = smem_u32(ring) >> 4, pitch16 = p.pitch >> 4;
            const uint32_t lbo1 = 1u << 16, lbo2 = ((p.off_z >> 4) + 1u) << 16;      // K-direction offsets: the next pair, here and in the copy
            const uint32_t b16 = (smem_u32(bsm) >> 4) | ((uint32_t)(4 * p.K) << 16);
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
                const uint32_t d = tmem_base + b * 2u * p.K;
                // window row t: kernel row t of the first output row (t < 7), t - 2 of the second (t >= 2); a row that
                // both need goes first, so that one MMA starts both sums
#pragma unroll
                for (int k = 0; k < kWindow; ++k) {
                    const uint32_t t = k < 5 ? k + 2 : k < 7 ? k - 5 : k;
                    const bool both = t >= 2 && t < (uint32_t)kR;
                    const uint32_t r = t < (uint32_t)kR ? t : t - 2;         // the larger kernel row: the operand's first columns
                    uint32_t slot = base + t;
                    if (slot >= (uint32_t)kSlots) slot -= kSlots;
                    const uint32_t a_lo = ring16 + slot * pitch16, b_lo = b16 + ((r & 1) * 16 + ((6 - r) >> 1)) * p.K;
                    const uint32_t dt = t < (uint32_t)kR ? d : d + p.K, idesc = both ? idesc2 : idesc1;
                    mma_bf16_ss(dt, desc64(a_lo | lbo1), desc64(b_lo), idesc, k > 0);
                    mma_bf16_ss(dt, desc64((a_lo + 2u) | lbo2), desc64(b_lo + 8u * p.K), idesc, 1u);
                }
                mma_commit(&bars->in_empty[b]);
                mma_commit(&bars->acc_full[b]);
                ++i;
            }
        }
        __syncwarp();
    } else if (warp < kFirstPool) {
        // ---- epilogue: warp -> TMEM lane quarter and every second 16-column chunk -----------------------------------------
        const int quarter = warp & 3, part = (warp - kFirstEpi) >> 2, q = quarter * 32 + lane;
        const int nch = p.K / 16;
        constexpr int kMaxOwn = 4;                       // chunks per warp (K <= 128)
        float saved[kMaxOwn][16];                        // the row above (pooled)
        Steps st(lo, hi, p.spi, kPool);
        uint32_t i = 0;
        bool ok = true;
        while (st.next()) {
            const uint32_t b = i & 1u;
            uint8_t *stage = smem + p.off_stage + (kPool ? (size_t)b * p.stage_bytes : 0u);
            if (kPool && st.reset) {
#pragma unroll
                for (int c = 0; c < kMaxOwn; ++c)
#pragma unroll
                    for (int k = 0; k < 16; ++k) saved[c][k] = __uint_as_float(0xFF800000u);
            }
            ok = mbar_wait(&bars->acc_full[b], (i >> 1) & 1u, abort_flag, ws, 0xB400);
            if (kPool && ok && i >= 2) ok = mbar_wait(&bars->stage_empty[b], ((i >> 1) & 1u) ^ 1u, abort_flag, ws, 0xB410);
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
            tc_fence_after_sync();
            const uint32_t t_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + b * 2u * p.K;
#pragma unroll
            for (int c = 0; c < kMaxOwn; ++c) {
                const int ch = part + 2 * c;
                if (ch >= nch) break;
                uint32_t r0[16], r1[16];
                tmem_ld_x16(t_addr + ch * 16, r0);
                tmem_ld_x16(t_addr + p.K + ch * 16, r1);
                tmem_ld_wait();
                if constexpr (kPool) {
                    // rows 2p - 1, 2p, 2p + 1 (the last one may not exist)
                    const bool has1 = 2 * st.p + 1 < p.P;
                    float v[16];
                    uint32_t m[8];
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        v[k] = fmaxf(saved[c][k], __uint_as_float(r0[k]));
                        if (has1) v[k] = fmaxf(v[k], __uint_as_float(r1[k]));
                        saved[c][k] = __uint_as_float(r1[k]);
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) m[k] = relu_bf16x2(cvt_bf16x2(v[2 * k], v[2 * k + 1]));
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
                            const uint32_t *v = j ? r1 : r0;
                            uint32_t o2[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                o2[k] = cvt_bf16x2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1]));
                                if (p.relu) o2[k] = relu_bf16x2(o2[k]);
                            }
                            yp[0] = make_uint4(o2[0], o2[1], o2[2], o2[3]);
                            yp[1] = make_uint4(o2[4], o2[5], o2[6], o2[7]);
                        } else {
                            float4 *yp = reinterpret_cast<float4 *>(static_cast<float *>(y) + o);
                            const uint32_t *v = j ? r1 : r0;
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                float f[4];
#pragma unroll
                                for (int k = 0; k < 4; ++k) {
                                    f[k] = __uint_as_float(v[4 * h + k]);
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
            if (lane == 0) {
                mbar_arrive(&bars->acc_empty[b]);
                if (kPool) mbar_arrive(&bars->stage_full[b]);
            }
            ++i;
        }
    } else if constexpr (kPool) {
        // ---- pooling: thread -> 16-byte unit u of a line, every `vs`-th pooled column; column v = columns 2v - 1, 2v, 2v + 1
        const int pt = tid - kFirstPool * 32, units = p.K / 8, u = pt % units, v0 = pt / units, vs = kPoolWarps * 32 / units;
        const bool on = v0 < vs;
        Steps st(lo, hi, p.spi, kPool);
        uint32_t i = 0;
        while (st.next()) {
            const uint32_t b = i & 1u;
            const bool ok = mbar_wait(&bars->stage_full[b], (i >> 1) & 1u, abort_flag, ws, 0xB500);
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
            const uint8_t *stage = smem + p.off_stage + (size_t)b * p.stage_bytes;
            uint16_t *out = static_cast<uint16_t *>(y) + ((size_t)st.n * p.PP + st.p) * p.PQ * p.K + u * 8;
            auto at = [&](int col) { return *reinterpret_cast<const uint4 *>(stage + (size_t)col * p.line + (((uint32_t)u ^ (uint32_t)(col & 7)) << 4)); };
            const int v_end = on && st.store ? p.PQ : 0;
            // loads of a batch are in flight together and not branched around (a row of 56 columns, 64 filters: five at a time
            // 39.6 us for 64 images, three 44.5, one after the other 46; 32 columns fit three: 22.1 against 26.2)
            auto batches = [&](auto size) {
                constexpr int kBatch = decltype(size)::value;
                for (int vb = 0; vb < p.PQ; vb += kBatch * vs) {
                    uint4 m[kBatch];
#pragma unroll
                    for (int k = 0; k < kBatch; ++k) {
                        const int c0 = 2 * min(vb + v0 + k * vs, p.PQ - 1);
                        m[k] = max4(at(c0), max4(at(c0 > 0 ? c0 - 1 : c0), at(c0 + 1 < p.Q ? c0 + 1 : c0)));
                    }
                    if (vb + kBatch * vs >= p.PQ) {      // all read: the stage is free before the row is on its way
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&bars->stage_empty[b]);
                    }
#pragma unroll
                    for (int k = 0; k < kBatch; ++k) {
                        const int v = vb + v0 + k * vs;
                        if (v < v_end) *reinterpret_cast<uint4 *>(out + (size_t)v * p.K) = m[k];
                    }
                }
            };
            if (p.PQ <= 3 * vs) batches(std::integral_constant<int, 3>{});
            else batches(std::integral_constant<int, 5>{});
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
    if (pool && (!d.relu || !p.y_bf16)) return false;          // (rows beside the image count as nothing because nothing is negative)
    p.PP = (p.P - 1) / 2 + 1; p.PQ = (p.Q - 1) / 2 + 1;
    p.spi = (p.P + 1) / 2;                                     // = PP
    const long long steps = (long long)d.N * p.spi;
    if (steps > 0x3FFFFFFF) return false;
    p.n_steps = (int)steps;
    p.pairs = p.Q + 3;
    p.pitch = round_up((uint32_t)p.pairs * 16u, 128);
    p.line = round_up(2u * d.K, 128);
    p.off_z = kSlots * p.pitch;
    p.off_b = 2u * p.off_z + 1024u;                            // (an operand reads 128 columns, past the end of the last row)
    p.off_stage = round_up(p.off_b + 2u * 4u * 4u * d.K * 16u, 128);
    p.stage_bytes = 128u * p.line;
    p.off_bar = p.off_stage + (pool ? 2u * p.stage_bytes : 0u);
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
                                  void *y, uint32_t *ws, cudaStream_t st, bool pool, Launch how)
{
    StemRowsParams p;
    if (!plan(d, bp, p, pool)) return NPAS_ERR_UNSUPPORTED;
    p.early = how.blob_ready;
    auto go = [&](auto kernel, int threads) {
        if (allow_dynamic_smem(reinterpret_cast<const void *>(kernel), (int)kSmemLimit) != NPAS_OK) return cudaErrorUnknown;
        const int sms = sm_count(), grid = p.n_steps < sms ? p.n_steps : sms;
        return launch_pdl(how, kernel, dim3(grid), dim3(threads), p.smem_bytes, st, p, static_cast<const uint16_t *>(x),
                          static_cast<const uint8_t *>(blob), bias, y, ws);
    };
    const cudaError_t e = pool ? go(conv_stem_rows_kernel<true>, kThreads<true>) : go(conv_stem_rows_kernel<false>, kThreads<false>);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // namespace npas
