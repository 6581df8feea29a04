// Block-based pruned GEMM for few output tiles: the columns of X are split over the CTAs of a cluster.
//
// The persistent kernels (linear_dn.cu, linear_d2.cu) give every output tile to one CTA (or pair), which is right while
// there are tiles for every SM.  A layer of few rows has a handful of tiles, and its time is then one CTA walking the
// whole input width by itself: latency, with most of the chip idle.  Here KS CTAs of a cluster share a tile of up to
// 128 rows x BN columns: each multiplies its own range of 64-column steps of X with the blob's masked dense image
// (both by TMA, 128-byte swizzled) into its tensor memory, writes the rows of its fp32 partial sums into the shared
// memory of the CTAs that own them (row r belongs to CTA r / rpr), and after one cluster barrier every CTA adds the KS
// partial sums of its rows in rank order (fixed order: bitwise reproducible), adds bias and residual, applies ReLU,
// rounds once and stores 16 bytes per thread along the row.
//
// What bounds it: the latency of one pass through the chain (copy, MMA, exchange, barrier, store), so the first copies
// are as early as possible: in a chain of layers (`early`) the weights are requested before the programmatic wait, X right
// after it; only the rows that exist are copied.
#include "common.cuh"
#include "tc_pair.cuh"

namespace npas {

using namespace tc;

namespace {

constexpr int kEpiWarps = 8;
constexpr int kThreads = (2 + kEpiWarps) * 32;           // warp 0: copies, warp 1: MMAs, then the epilogue warps
constexpr int kRows = 128;
constexpr int kMaxStages = 8;
constexpr int kMaxSplit = 8;                              // portable cluster size
constexpr uint32_t kSmemLimit = 232448;
constexpr uint32_t kDescHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t kDescLboOne = 1u << 16;

struct LinSkParams {
    int M, I, O, BN, KS, nK, kpr, nMT, nNT, S, XR, rpr;   // kpr: steps per CTA; XR: rows of X per copy; rpr: rows a CTA owns
    int relu, y_bf16, early;                              // early: the blob may be read before the wait (Launch::blob_ready)
    uint32_t x_bytes, stage_bytes, red_pitch, off_red, off_bias, off_bar, smem_bytes, tmem_cols;
};

struct LinSkBars {
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t acc_full;
    uint32_t tmem_base;
    uint32_t abort_flag;
};

__device__ __forceinline__ uint64_t desc64(uint32_t lo) { return ((uint64_t)kDescHiSw128 << 32) | lo; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1)
linear_bb_sk_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w, const LinSkParams p,
                    const float *__restrict__ bias, const void *__restrict__ res, void *__restrict__ y, uint32_t *ws)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float *bias_s = reinterpret_cast<float *>(smem + p.off_bias);      // [BN]
    LinSkBars *bars = reinterpret_cast<LinSkBars *>(smem + p.off_bar);
    volatile uint32_t *abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_ctarank(), tile = blockIdx.x / p.KS;
    const int mt = tile / p.nNT, nt = tile - mt * p.nNT;
    const int k_lo = rank * p.kpr, k_n = max(0, min(p.nK - k_lo, p.kpr));
    const int rows = min(kRows, p.M - mt * kRows), cols = min(p.BN, p.O - nt * p.BN);

    if (tid == 0) {
        for (int s = 0; s < p.S; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
        mbar_init(&bars->acc_full, 1);
        bars->abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&tmap_x);
        prefetch_tensormap(&tmap_w);
        // the weights of the first ring of steps
        for (int k = 0; p.early && k < min(k_n, p.S); ++k) {
            mbar_arrive_expect_tx(&bars->full[k], p.stage_bytes);
            tma_load_2d(smem + (size_t)k * p.stage_bytes + p.x_bytes, &tmap_w, &bars->full[k], (k_lo + k) * 64, nt * p.BN);
        }
    }
    if (warp == 1) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    pdl_trigger();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    cluster_arrive();                  // this CTA is running: its shared memory may be written by the others
    pdl_wait();
    const int z = zero_behind_wait();

    if (warp >= 2)
        for (int i = tid - 64 + z; i < p.BN; i += kThreads - 64) bias_s[i] = (bias && i < cols) ? __ldg(bias + nt * p.BN + i) : 0.f;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t s = 0, lap = 0;
            for (int k = 0; k < k_n; ++k) {
                if (lap >= 1 && !mbar_wait(&bars->empty[s], (lap & 1u) ^ 1u, abort_flag, ws, 0x9100)) break;
                if (lap >= 1 || !p.early) {
                    mbar_arrive_expect_tx(&bars->full[s], p.stage_bytes);
                    tma_load_2d(smem + (size_t)s * p.stage_bytes + p.x_bytes, &tmap_w, &bars->full[s], (k_lo + k) * 64, nt * p.BN);
                }
                tma_load_2d(smem + (size_t)s * p.stage_bytes, &tmap_x, &bars->full[s], (k_lo + k) * 64, mt * kRows);
                if (++s == (uint32_t)p.S) { s = 0; ++lap; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = idesc_bf16_f32(128, p.BN);
            // (18 address bits: in the CTAs of a cluster a shared-memory address carries the CTA's rank above them)
            const uint32_t base16 = ((smem_u32(smem) & 0x3FFFFu) >> 4) | kDescLboOne, stage16 = p.stage_bytes >> 4;
            uint32_t s = 0, ph = 0, a_lo = base16;
            bool go = true;
            for (int k = 0; k < k_n; ++k) {
                if (!mbar_wait(&bars->full[s], ph, abort_flag, ws, 0x9300)) { go = false; break; }
                tc_fence_after_sync();
                const uint32_t b_lo = a_lo + (p.x_bytes >> 4);
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j)          // 16 columns = 32 bytes inside the swizzled row
                    mma_bf16_ss(tmem_base, desc64(a_lo + 2 * j), desc64(b_lo + 2 * j), idesc, (k > 0 || j > 0) ? 1u : 0u);
                mma_commit(&bars->empty[s]);
                a_lo += stage16;
                if (++s == (uint32_t)p.S) { s = 0; ph ^= 1u; a_lo = base16; }
            }
            if (go) mma_commit(&bars->acc_full);
        }
        __syncwarp();
    }
    cluster_wait();                    // every CTA of the cluster is running
    if (warp >= 2 && k_n > 0) {
        // partial sums -> the CTAs that own the rows: [rank][row][BN] floats, rows padded by 16 bytes (conflict free)
        const int quarter = warp & 3, part = (warp - 2) >> 2, m = quarter * 32 + lane;
        if (__all_sync(0xFFFFFFFFu, mbar_wait(&bars->acc_full, 0, abort_flag, ws, 0x9400))) {
            tc_fence_after_sync();
            const int owner = min(m / p.rpr, p.KS - 1), r = m - owner * p.rpr;
            const uint32_t dst = map_to_cta(smem_u32(smem + p.off_red), (uint32_t)owner) + (uint32_t)(rank * p.rpr + r) * p.red_pitch;
            for (int c0 = part * 16; c0 < p.BN; c0 += 16 * (kEpiWarps / 4)) {
                uint32_t v[16];
                __syncwarp();
                tmem_ld_x16(tmem_base + ((uint32_t)(quarter * 32) << 16) + c0, v);
                tmem_ld_wait();
                if (m < rows) {
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        st_cluster_v4(dst + (uint32_t)(c0 + 4 * h) * 4u, v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
                }
            }
        }
    }
    tc_fence_before_sync();
    cluster_arrive();
    cluster_wait();                    // all partial sums are in place; no CTA touches another's memory after this
    tc_fence_after_sync();
    if (warp == 1) tmem_dealloc(tmem_base, p.tmem_cols);
    if (*abort_flag) {
        // a role gave up: leave time for copies still in flight to land before the CTA retires
        const long long t0 = clock64();
        while (clock64() - t0 < 400000ll) { }
        return;
    }

    const int live = (p.nK + p.kpr - 1) / p.kpr;          // CTAs that had steps to do
    const int own = max(0, min(p.rpr, rows - rank * p.rpr)), oct = p.BN / 8;
    for (int i = tid; i < own * oct; i += kThreads) {
        const int r = i / oct, c0 = (i - r * oct) * 8;
        if (c0 >= cols) continue;
        const size_t o0 = (size_t)(mt * kRows + rank * p.rpr + r) * p.O + (size_t)(nt * p.BN + c0 + z);
        const uint8_t *src = smem + p.off_red + (size_t)r * p.red_pitch + (size_t)c0 * 4;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = 0.f;
        for (int s = 0; s < live; ++s, src += (size_t)p.rpr * p.red_pitch) {
            const float4 a = *reinterpret_cast<const float4 *>(src), b = *reinterpret_cast<const float4 *>(src + 16);
            v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
            v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += bias_s[c0 + j];
        if (p.y_bf16) {
            if (res) {
                const uint4 u = __ldg(reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(res) + o0));
                const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[2 * j] += __uint_as_float(w[j] << 16);
                    v[2 * j + 1] += __uint_as_float(w[j] & 0xFFFF0000u);
                }
            }
            uint32_t o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                o[j] = cvt_bf16x2(v[2 * j], v[2 * j + 1]);
                if (p.relu) o[j] = relu_bf16x2(o[j]);
            }
            *reinterpret_cast<uint4 *>(static_cast<uint16_t *>(y) + o0) = make_uint4(o[0], o[1], o[2], o[3]);
        } else {
            if (res) {
                const float4 *rp = reinterpret_cast<const float4 *>(static_cast<const float *>(res) + o0);
                const float4 a = __ldg(rp + 0), b = __ldg(rp + 1);
                v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
                v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
            }
            if (p.relu) {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = fmaxf(v[j], 0.f);
            }
            float4 *yp = reinterpret_cast<float4 *>(static_cast<float *>(y) + o0);
            yp[0] = make_float4(v[0], v[1], v[2], v[3]);
            yp[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
    }
}

// Microseconds of a launch by a model fitted to 307 measured (size, tile, split) points (standard error 11 %; M 1 to
// 6272, I 64 to 2048, O 64 to 2048): what every launch costs, the steps of one CTA, the partial sums that leave a CTA
// through its own and other shared memories, and the grid.
double modelled(const LinSkParams &p)
{
    return 1.9 + 0.18 * p.kpr + 0.57e-4 * p.XR * p.BN * 4. + 0.01 * p.nMT * p.nNT * p.KS;
}

// `variant`: column tile + (CTAs per tile << 16); with the upper half zero this kernel is only planned when `automatic`.
bool plan(const npas_linear_desc &d, const npas_bb_desc &bb, LinSkParams &p, int sms, bool automatic)
{
    if (d.x_dtype != NPAS_BF16 || bb.w_packed != NPAS_BF16) return false;
    if (d.I % 8 || d.O % 8) return false;                 // rows of X, W and Y start on 16-byte boundaries
    const int want_bn = d.variant & 0xFFFF, want_ks = (d.variant >> 16) & 0xFFFF;
    if (!automatic && !want_ks) return false;
    LinSkParams q = {};
    q.M = d.M; q.I = d.I; q.O = d.O;
    q.nK = (d.I + 63) / 64;
    q.nMT = (d.M + kRows - 1) / kRows;
    q.relu = d.relu; q.y_bf16 = d.y_dtype == NPAS_BF16;
    const int rows = d.M < kRows ? d.M : kRows;
    q.XR = (rows + 7) / 8 * 8;
    q.x_bytes = (uint32_t)q.XR * 128u;
    double best = 0.;
    bool found = false;
    for (int bn = 128; bn >= 16; bn /= 2) {
        if (want_bn && bn != want_bn) continue;
        if (!want_bn && bn > 16 && bn >= 2 * d.O) continue;
        for (int ks = kMaxSplit; ks >= 1; ks /= 2) {
            if (want_ks ? ks != want_ks : (ks > 1 && ks > q.nK)) continue;
            q.BN = bn; q.KS = ks;
            q.nNT = (d.O + bn - 1) / bn;
            const long long tiles = (long long)q.nMT * q.nNT;
            // one wave: clusters do not straddle groups of SMs, so the larger ones leave some unused (sixteen clusters of
            // eight took two waves: 8.8 us against 4.4 with clusters of four)
            if (tiles * ks > (ks == 8 && !want_ks ? sms * 3 / 4 : ks > 1 ? sms - sms / 8 : sms)) continue;
            q.kpr = (q.nK + ks - 1) / ks;
            q.rpr = (rows + ks - 1) / ks;
            q.stage_bytes = q.x_bytes + (uint32_t)bn * 128u;
            q.red_pitch = (uint32_t)bn * 4u + 16u;
            const uint32_t red = (uint32_t)ks * q.rpr * q.red_pitch;
            const uint32_t tail = kRows * 128u;          // an MMA reads 128 rows from the start of the last stage
            const uint32_t fixed = round_up(red > tail ? red : tail, 128) + (uint32_t)bn * 4u + (uint32_t)sizeof(LinSkBars) + 256u + 1024u;
            q.S = (int)((kSmemLimit - fixed) / q.stage_bytes);
            if (q.S > kMaxStages) q.S = kMaxStages;
            if (q.S > q.kpr) q.S = q.kpr;
            if (q.S < 1 || (q.S < 2 && q.kpr > 1)) continue;
            q.off_red = (uint32_t)q.S * q.stage_bytes;
            q.off_bias = q.off_red + round_up(red > tail ? red : tail, 128);
            q.off_bar = round_up(q.off_bias + (uint32_t)bn * 4u, 128);
            q.smem_bytes = q.off_bar + (uint32_t)sizeof(LinSkBars) + 1024u;
            q.tmem_cols = 32;
            while ((int)q.tmem_cols < bn) q.tmem_cols *= 2;
            const double cost = modelled(q);
            if (!found || cost < best) { best = cost; p = q; found = true; }
        }
    }
    return found;
}

bool planned(const npas_linear_desc &d, const npas_bb_desc &bb, LinSkParams &p, bool automatic)
{
    return cached_plan(d, bb, automatic, p, [&](LinSkParams &q) { return plan(d, bb, q, sm_count(), automatic); });
}

}  // namespace

bool linear_sk_supported(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    LinSkParams p;
    return planned(d, bb, p, false);
}

// Where the persistent kernels leave most SMs idle: fewer tiles of 128 x 128 than a quarter of the SMs.  Measured (this
// kernel against the better persistent one, both in a chain of layers): 49x2048 -> 512 3.9 against 9.9 us, 64x2048 -> 1000 4.4 against 9.8,
// 196x1024 -> 256 3.9 against 7.1, 784x512 -> 128 3.6 against 5.1, 1x128 -> 256 2.5 against 3.9; from about forty
// tiles on they draw level (6272x512 -> 128 5.8 against 5.3).  Up to 256 columns there is little to split and the gain
// is that of narrower tiles on more SMs: for a single row tile, or where 128 x 32 tiles fill a fifth of the chip.
bool linear_sk_preferred(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    if (d.variant) return false;
    const int sms = sm_count();
    const long long nMT = (d.M + kRows - 1) / kRows;
    if (nMT * ((d.O + 127) / 128) * 4 >= sms) return false;
    if (d.I <= 256 && nMT > 1 && nMT * ((d.O + 31) / 32) * 5 < sms) return false;
    LinSkParams p;
    return planned(d, bb, p, true);
}

// the shape an automatic choice of this kernel runs, as a `variant` (0: none)
int32_t linear_sk_variant(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    LinSkParams p;
    return planned(d, bb, p, true) ? p.BN | (p.KS << 16) : 0;
}

npas_status linear_sk_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x, const void *blob, const float *bias,
                             const void *res, void *y, uint32_t *ws, cudaStream_t st, Launch how)
{
    LinSkParams p;
    if (!planned(d, bb, p, true)) return NPAS_ERR_UNSUPPORTED;
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return NPAS_ERR_CUDA;
    const BbLayout L = bb_layout(bb);
    auto encode = [&](CUtensorMap *m, const void *base, uint64_t outer, uint32_t box_rows) {
        const cuuint64_t dims[2] = {(cuuint64_t)d.I, outer};
        const cuuint64_t strides[1] = {(cuuint64_t)d.I * 2};
        const cuuint32_t box[2] = {64, box_rows}, estr[2] = {1, 1};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap tmx, tmw;
    if (!encode(&tmx, x, (uint64_t)d.M, (uint32_t)p.XR) || !encode(&tmw, static_cast<const uint8_t *>(blob) + L.off_dense, (uint64_t)d.O, (uint32_t)p.BN))
        return NPAS_ERR_CUDA;
    if (allow_dynamic_smem(reinterpret_cast<const void *>(linear_bb_sk_kernel), (int)kSmemLimit) != NPAS_OK) return NPAS_ERR_CUDA;
    p.early = how.blob_ready;
    const cudaError_t e = launch_pdl_cluster(how, linear_bb_sk_kernel, dim3(p.nMT * p.nNT * p.KS), dim3(kThreads), p.KS, p.smem_bytes, st,
                                             tmx, tmw, p, bias, res, y, ws);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // namespace npas
