// Block-punched convolution from the blob's dense operand image for few output tiles: the input channels (and taps) are
// split over the CTAs of a cluster.
//
// The persistent kernels (conv_dn.cu, conv_d2.cu) give a tile of positions and filters to one CTA (or pair), whose time is
// then the whole chain of channels x taps MMAs: one 14x14x256 image ran on four CTAs for 13 us.  Here KS = KC x KT CTAs of
// a cluster share a tile of 128 positions x NT filters: each takes a range of channel blocks and a range of taps,
// accumulates in its own tensor memory, writes the rows of its fp32 partial sums into the shared memory of the CTAs that
// own them, and after one cluster barrier every CTA adds the KS partial sums of its rows in rank order (bitwise
// reproducible), adds bias and residual, applies ReLU, rounds once and stores 16 bytes per thread along the filters.
//
// Operands.  Activations: slabs of CB channels (64, 32 or 16, the widest that divides C; one 2 CB-byte row per padded
// position, swizzled by the row width) by one 4-D tensor copy, so that a tap is a start offset of whole rows; stride 2 with
// a 3x3 kernel and pad 1 takes four slabs, one per parity class, and computes only the wanted positions.  Weights: the
// blob's image through a 4-D tensor map (128-byte lines of a filter row, lines, filter groups, rows): a box of lines x
// groups x (chunk, tap, octet) rows lands as [tap][octet][NT filters][8], whatever the image's group width, so NT is any
// multiple of 16 that groups can make up (one MMA covers 176 filters where the image has groups of 16).
//
// What bounds it is the latency of the chain copy, MMAs, exchange, store: the weights are requested by a warp of their own, in
// a chain of layers before the programmatic wait (`early`), the slabs right behind it.
#include "common.cuh"
#include "tail_start.h"
#include "tc_pair.cuh"

namespace npas {

using namespace tc;

namespace {

constexpr int kEpiWarps = 8;
constexpr int kThreads = (3 + kEpiWarps) * 32;           // warp 0: slabs, warp 1: MMAs, warp 2: weights, then the epilogue warps
constexpr int kRows = 128;
constexpr int kMaxStages = 4;
constexpr int kMaxChunks = 4;                             // 16-channel chunks per stage (CB / 16)
constexpr int kMaxOwnChunks = 256;                        // chunks of a CTA whose tap unions are kept (beyond: every tap)
constexpr int kMaxTapsSk = 16;
constexpr int kMaxSplit = 8;                              // portable cluster size
constexpr uint32_t kSmemLimit = 232448;
constexpr uint32_t kDescHiB = (128u >> 4) | (1u << 14);   // no swizzle, SBO = 128 bytes, version bit

struct ConvSkParams {
    int N, K, P, Q, Po, Qo, sh, pad;                      // P, Q: positions the tiles walk; sh: store every (1 << sh)-th
    int nph, Wp, TR, tiles_per_img, n_tiles, slab_rows;
    int RS, nCh, CB, nBlk, NT, nFT, KC, KT, bpr, tpr;     // bpr: channel blocks per CTA; tpr: taps per CTA
    int GI, lines, S, rpr;
    int relu, y_bf16, use_taps, early;                    // early: the blob may be read before the wait (Launch::blob_ready)
    uint32_t desc_hi_a, slab_bytes, act_stride, w_chunk, stage_bytes, red_pitch, off_red, off_bias, off_bar, smem_bytes, tmem_cols;
    uint32_t shift16[kMaxTapsSk];                         // operand start of every tap inside a stage's slabs, 16-byte units
};

struct ConvSkBars {
    uint64_t a_full[kMaxStages], w_full[kMaxStages][kMaxChunks], empty[kMaxStages];
    uint64_t acc_full;
    uint32_t tmem_base;
    uint32_t abort_flag;
    uint32_t taps[kMaxOwnChunks];                         // union of the kept taps per chunk of this CTA
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *m, uint64_t *bar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1)
conv_bp_sk_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w, const ConvSkParams p,
                  const uint8_t *__restrict__ blob, const float *__restrict__ bias, const void *__restrict__ res,
                  void *__restrict__ y, uint32_t *ws)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float *bias_s = reinterpret_cast<float *>(smem + p.off_bias);      // [NT]
    ConvSkBars *bars = reinterpret_cast<ConvSkBars *>(smem + p.off_bar);
    volatile uint32_t *abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int KS = p.KC * p.KT, rank = (int)cluster_ctarank(), work = blockIdx.x / KS;
    // (the last tile of filters ends with the last one, tail_start.h, and leaves those it shares with the tile before to that one)
    const int tile = work / p.nFT, ft = work - tile * p.nFT, k0 = tail_start(ft * p.NT, p.NT, p.K), shared = ft * p.NT - k0;
    const int img = tile / p.tiles_per_img, y0 = (tile - img * p.tiles_per_img) * p.TR;
    const int kc = rank / p.KT, kt = rank - kc * p.KT;
    const int blk_lo = kc * p.bpr, n_blk = max(0, min(p.nBlk - blk_lo, p.bpr));
    const int t_lo = kt * p.tpr, n_tap = max(0, min(p.RS - t_lo, p.tpr));
    const int t_box = min(t_lo, p.RS - p.tpr);            // first tap of the weight boxes: they stay inside a chunk's rows
    const bool has_work = n_blk > 0 && n_tap > 0;
    const int cpb = p.CB / 16;

    if (tid == 0) {
        for (int s = 0; s < p.S; ++s) {
            mbar_init(&bars->a_full[s], 1);
            mbar_init(&bars->empty[s], 1);
            for (int c = 0; c < cpb; ++c) mbar_init(&bars->w_full[s][c], 1);
        }
        mbar_init(&bars->acc_full, 1);
        bars->abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&tmap_x);
        prefetch_tensormap(&tmap_w);
    }
    if (warp == 1) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    pdl_trigger();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    cluster_arrive();                  // this CTA is running: its shared memory may be written by the others
    if (!p.early) pdl_wait();
    blob = behind_wait(blob);

    if (warp == 2) {
        // ---- weights: one box per 16-channel chunk; the first ring of stages before anything else ------------------
        if (lane == 0 && has_work) {
            const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
            const uint32_t off_image = hdr[BP_OFF_IMAGE];
            if (off_image == 0u || (off_image & 2047u) || hdr[BP_GI] != (uint32_t)p.GI) {
                bars->abort_flag = 2;                     // not the image this was planned for: the other roles leave their waits
                if (atomicCAS(ws, 0u, 6u /* NPAS_ERR_BLOB */) == 0u) ws[1] = 0xA001;
            } else {
                const int row0 = (int)(off_image / (uint32_t)(p.GI * 16)), g0 = k0 / p.GI, line0 = (k0 - g0 * p.GI) / 8;
                uint32_t s = 0, lap = 0;
                for (int b = 0; b < n_blk; ++b) {
                    if (lap >= 1 && !mbar_wait(&bars->empty[s], (lap & 1u) ^ 1u, abort_flag, ws, 0xA100)) break;
                    uint8_t *dst = smem + (size_t)s * p.stage_bytes + (size_t)p.nph * p.act_stride;
                    for (int c = 0; c < cpb; ++c, dst += p.w_chunk) {
                        mbar_arrive_expect_tx(&bars->w_full[s][c], p.w_chunk);
                        tma_load_4d(dst, &tmap_w, &bars->w_full[s][c], 0, line0, g0, row0 + (((blk_lo + b) * cpb + c) * p.RS + t_box) * 2);
                    }
                    if (++s == (uint32_t)p.S) { s = 0; ++lap; }
                }
            }
        }
        __syncwarp();
    }
    const int own_chunks = min(n_blk * cpb, kMaxOwnChunks);
    if (warp == 1 && p.use_taps) {
        // (a tap that no block of the tile's groups keeps in a chunk multiplies zeros: skipped.  Fetched beside the weights)
        const uint32_t off_tapu = reinterpret_cast<const uint32_t *>(blob)[BP_OFF_TAPU];
        const uint32_t *tapu = reinterpret_cast<const uint32_t *>(blob + off_tapu);
        const int g0 = k0 / p.GI, ng = min((k0 + p.NT - 1) / p.GI, p.K / p.GI - 1) - g0 + 1;
        for (int i = lane; i < own_chunks; i += 32) bars->taps[i] = off_tapu ? 0u : 0xFFFFFFFFu;
        __syncwarp();
        if (off_tapu)
#pragma unroll 4
            for (int e = lane; e < own_chunks * ng; e += 32) {
                const int g = e / own_chunks, i = e - g * own_chunks;
                atomicOr(&bars->taps[i], __ldg(tapu + (g0 + g) * p.nCh + blk_lo * cpb + i));
            }
        __syncwarp();
    }
    pdl_wait();
    const int z = zero_behind_wait();
    if (warp > 2)
        for (int i = tid - 96 + z; i < p.NT; i += kThreads - 96) bias_s[i] = bias ? __ldg(bias + k0 + i) : 0.f;

    if (warp == 0) {
        // ---- slabs -----------------------------------------------------------------------------------------------
        if (lane == 0 && has_work) {
            uint32_t s = 0, lap = 0;
            for (int b = 0; b < n_blk; ++b) {
                if (lap >= 1 && !mbar_wait(&bars->empty[s], (lap & 1u) ^ 1u, abort_flag, ws, 0xA110)) break;
                uint8_t *dst = smem + (size_t)s * p.stage_bytes;
                mbar_arrive_expect_tx(&bars->a_full[s], (uint32_t)p.nph * p.slab_bytes);
                const int c0 = (blk_lo + b) * p.CB;
                if (p.nph == 1) tma_load_4d(dst, &tmap_x, &bars->a_full[s], c0, -p.pad, y0 - p.pad, img);
                else
                    for (int ph = 0; ph < 4; ++ph)            // the input pixels (2 i + ph / 2, 2 j + ph % 2), i from y0 - 1, j from -1
                        tma_load_4d(dst + (size_t)ph * p.act_stride, &tmap_x, &bars->a_full[s], c0, (ph & 1) - 2, 2 * (y0 - 1) + (ph >> 1), img);
                if (++s == (uint32_t)p.S) { s = 0; ++lap; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMAs ------------------------------------------------------------------------------------------------
        if (elect_one() && has_work) {
            const uint32_t idesc = idesc_bf16_f32(128, p.NT);
            // (18 address bits: in the CTAs of a cluster a shared-memory address carries the CTA's rank above them)
            const uint32_t base16 = (smem_u32(smem) & 0x3FFFFu) >> 4, stage16 = p.stage_bytes >> 4, wc16 = p.w_chunk >> 4;
            const uint64_t hi_a = (uint64_t)p.desc_hi_a << 32, hi_b = (uint64_t)kDescHiB << 32;
            const uint32_t b_hi = (uint32_t)p.NT << 16, b_step = 2u * p.NT, range = ((1u << n_tap) - 1u) << t_lo;
            uint32_t s = 0, ph = 0, first = 0;
            int ch = 0;
            bool go = true;
            for (int b = 0; b < n_blk && go; ++b) {
                if (!mbar_wait(&bars->a_full[s], ph, abort_flag, ws, 0xA300)) { go = false; break; }
                const uint32_t st16 = base16 + s * stage16;
                uint32_t a_lo = st16 | (1u << 16), b0 = (st16 + (uint32_t)p.nph * (p.act_stride >> 4)) | b_hi;
                for (int c = 0; c < cpb; ++c, ++ch, a_lo += 2u, b0 += wc16) {          // 16 channels = 32 bytes inside the swizzled row
                    if (!mbar_wait(&bars->w_full[s][c], ph, abort_flag, ws, 0xA310)) { go = false; break; }
                    tc_fence_after_sync();
                    uint32_t b_lo = b0 + (uint32_t)(t_lo - t_box) * b_step;
                    // (without a test per MMA when every tap of the range is kept, which random masks always do: the issuing
                    // thread's own instructions are on the critical path)
                    const uint32_t kept = (p.use_taps && ch < own_chunks ? bars->taps[ch] : 0xFFFFFFFFu) & range;
                    if (kept == range) {
                        for (int t = t_lo; t < t_lo + n_tap; ++t, b_lo += b_step) {
                            mma_bf16_ss(tmem_base, hi_a | (a_lo + p.shift16[t]), hi_b | b_lo, idesc, first);
                            first = 1u;
                        }
                    } else {
                        for (int t = t_lo; t < t_lo + n_tap; ++t, b_lo += b_step) {
                            if (!((kept >> t) & 1u) && (first || t > t_lo)) continue;      // (one MMA at least: it clears the accumulator)
                            mma_bf16_ss(tmem_base, hi_a | (a_lo + p.shift16[t]), hi_b | b_lo, idesc, first);
                            first = 1u;
                        }
                    }
                }
                mma_commit(&bars->empty[s]);
                if (++s == (uint32_t)p.S) { s = 0; ph ^= 1u; }
            }
            if (go) mma_commit(&bars->acc_full);
        }
        __syncwarp();
    }
    cluster_wait();                    // every CTA of the cluster is running
    if (warp > 2 && has_work) {
        // partial sums -> the CTAs that own the rows: [rank][row][NT] floats, rows padded by 16 bytes (conflict free)
        const int quarter = warp & 3, part = (warp - 3) >> 2, m = quarter * 32 + lane;
        if (__all_sync(0xFFFFFFFFu, mbar_wait(&bars->acc_full, 0, abort_flag, ws, 0xA400))) {
            tc_fence_after_sync();
            const int owner = m / p.rpr, r = m - owner * p.rpr, oy = m / p.Wp, ox = m - oy * p.Wp;
            const bool valid = oy < p.TR && y0 + oy < p.P && ox < p.Q && (((y0 + oy) | ox) & p.sh) == 0;
            const uint32_t dst = map_to_cta(smem_u32(smem + p.off_red), (uint32_t)owner) + (uint32_t)(rank * p.rpr + r) * p.red_pitch;
            for (int c0 = part * 16; c0 < p.NT; c0 += 16 * (kEpiWarps / 4)) {
                uint32_t v[16];
                __syncwarp();
                tmem_ld_x16(tmem_base + ((uint32_t)(quarter * 32) << 16) + c0, v);
                tmem_ld_wait();
                if (valid) {
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

    const int live = ((p.nBlk + p.bpr - 1) / p.bpr) * p.KT;          // CTAs that had work (every tap range has)
    const int oct = p.NT / 8;
    for (int i = tid; i < p.rpr * oct; i += kThreads) {
        const int r = i / oct, c0 = (i - r * oct) * 8, m = rank * p.rpr + r, oy = m / p.Wp, ox = m - oy * p.Wp, yy = y0 + oy;
        if (m >= kRows || c0 < shared || oy >= p.TR || yy >= p.P || ox >= p.Q || ((yy | ox) & p.sh)) continue;
        const size_t o0 = (((size_t)img * p.Po + (yy >> p.sh)) * p.Qo + (ox >> p.sh)) * p.K + (size_t)(k0 + c0 + z);
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

// CTAs that run at once: clusters do not straddle groups of SMs, so the larger ones leave some unused.
int at_once(int ks, int sms) { return ks > 4 ? sms * 3 / 4 : ks > 1 ? sms - sms / 8 : sms; }

// Microseconds of a launch by a model fitted to 455 measured (layer, filters, split) points of 29 layers (standard error
// 9 %; the shape it picks is within 1 % of the best measured one on average): what every launch costs, the MMAs of one CTA
// (50 cycles or half a cycle per filter), the bytes it takes in, the partial sums that leave it, and the grid; what a CTA
// does comes again with every wave.
double modelled(const ConvSkParams &p, int sms)
{
    const int ks = p.KC * p.KT;
    const double mma = (double)p.bpr * (p.CB / 16) * p.tpr * (p.NT > 100 ? p.NT * 0.5 : 50.) / 1900.;
    const double in = (double)p.bpr * (p.nph * p.slab_bytes + (double)(p.CB / 16) * p.w_chunk) * 1e-5;
    const long long ctas = (long long)p.n_tiles * p.nFT * ks, cap = at_once(ks, sms);
    const double waves = (double)((ctas + cap - 1) / cap);
    return 2.05 + waves * (0.94 * mma + 0.82 * in + 0.02 * p.NT + 0.14 * p.bpr + (ks > 1 ? 0.22 : 0.)) + 0.0107 * (ctas < cap ? ctas : cap);
}

// `variant`: filters per tile | channel ranges << 16 | tap ranges << 24; 0: the model's choice
bool plan(const npas_conv_desc &d, const npas_bp_desc &bp, ConvSkParams &p, int sms, bool one_wave)
{
    if (d.x_dtype != NPAS_BF16 || bp.w_packed != NPAS_BF16) return false;
    if ((d.stride != 1 && d.stride != 2) || d.pad < 0 || d.C % 16 || d.K % 16) return false;
    const int RS = d.R * d.S;
    if (RS > kMaxTapsSk) return false;
    ConvSkParams q = {};
    q.GI = (int)bp_layout(bp, 0).GI;
    if (q.GI < 16) return false;
    q.N = d.N; q.K = d.K; q.RS = RS; q.pad = d.pad;
    q.P = d.H + 2 * d.pad - d.R + 1; q.Q = d.W + 2 * d.pad - d.S + 1;
    if (q.P < 1 || q.Q < 1) return false;
    q.Po = (q.P - 1) / d.stride + 1; q.Qo = (q.Q - 1) / d.stride + 1;
    const bool phases = d.stride == 2 && d.R == 3 && d.S == 3 && d.pad == 1;     // (as in conv_d2.cu)
    q.nph = phases ? 4 : 1;
    q.sh = phases ? 0 : d.stride - 1;
    if (phases) { q.P = q.Po; q.Q = q.Qo; q.Wp = q.Qo + 1; }
    else q.Wp = d.W + 2 * d.pad;
    if (q.Wp > 128) return false;
    q.TR = q.P < 128 / q.Wp ? q.P : 128 / q.Wp;
    q.slab_rows = phases ? q.TR + 1 : q.TR + d.R - 1;
    if (q.slab_rows > 128) return false;
    q.tiles_per_img = (q.P + q.TR - 1) / q.TR;
    const long long n_tiles = (long long)d.N * q.tiles_per_img;
    if (n_tiles > (one_wave ? sms : 0xFFFFFF)) return false;
    q.n_tiles = (int)n_tiles;
    q.nCh = d.C / 16;
    q.CB = d.C % 64 == 0 ? 64 : d.C % 32 == 0 ? 32 : 16;
    q.nBlk = d.C / q.CB;
    q.relu = d.relu; q.y_bf16 = d.y_dtype == NPAS_BF16;
    const uint32_t row = (uint32_t)q.CB * 2u;                   // bytes of a position in a slab
    q.desc_hi_a = ((8u * row) >> 4) | (1u << 14) | ((q.CB == 64 ? 2u : q.CB == 32 ? 4u : 6u) << 29);
    q.slab_bytes = (uint32_t)q.slab_rows * q.Wp * row;
    const uint32_t reach = (128u + (uint32_t)(phases ? 1 : d.R - 1) * q.Wp + (phases ? 1 : d.S)) * row;   // a shifted operand reads 128 rows
    q.act_stride = round_up(reach > q.slab_bytes ? reach : q.slab_bytes, 1024);
    for (int t = 0; t < RS; ++t) {
        const int r = t / d.S, s = t % d.S;
        if (phases) {
            const int a = (r - 1) & 1, b = (s - 1) & 1, dr = r == 0 ? -1 : 0, ds = s == 0 ? -1 : 0;
            q.shift16[t] = (uint32_t)(a * 2 + b) * (q.act_stride >> 4) + (uint32_t)((dr + 1) * q.Wp + ds + 1) * (row >> 4);
        } else {
            q.shift16[t] = (uint32_t)(r * q.Wp + s) * (row >> 4);
        }
    }
    const int want_nt = d.variant & 0xFFFF, want_kc = (d.variant >> 16) & 0xFF, want_kt = (d.variant >> 24) & 0xFF;
    double best = 0.;
    bool found = false;
    for (int nt = 16; nt <= 128; nt += 16) {
        if (want_nt && nt != want_nt) continue;
        if (nt < q.GI ? q.GI % nt != 0 : nt % q.GI != 0) continue;
        if (!want_nt && nt > d.K) continue;
        const int tile = nt < d.K ? nt : d.K;                   // (a wider tile was asked for: all filters)
        for (int kc = 1; kc <= kMaxSplit && kc <= q.nBlk; ++kc)
            for (int kt = 1; kc * kt <= kMaxSplit && kt <= RS && kt <= 4; ++kt) {
                if ((want_kc && kc != want_kc) || (want_kt && kt != want_kt)) continue;
                q.NT = tile; q.nFT = (d.K + tile - 1) / tile; q.KC = kc; q.KT = kt;
                q.bpr = (q.nBlk + kc - 1) / kc; q.tpr = (RS + kt - 1) / kt;
                if ((kc - 1) * q.bpr >= q.nBlk || (kt - 1) * q.tpr >= RS) continue;     // a CTA without work
                const int ks = kc * kt;
                const long long ctas = n_tiles * q.nFT * ks;
                if (ctas > (one_wave ? at_once(ks, sms) : 0x3FFFFFFF)) continue;
                // the blob's tap unions (per image group and chunk) are read only where few enough blocks meet in a tile that a
                // third of the taps must be missing: the two dependent reads cost 0.5 to 2 us where nothing else hides them
                const int wide = tile > q.GI ? tile : q.GI, blocks = ((wide + bp.Mb - 1) / bp.Mb) * ((16 + bp.Nb - 1) / bp.Nb);
                q.use_taps = bp.max_taps > 0 && blocks * bp.max_taps * 3 <= RS * 2;
                q.lines = (tile < q.GI ? tile : q.GI) / 8;
                q.rpr = (kRows + ks - 1) / ks;
                q.w_chunk = 2u * q.tpr * tile * 16u;
                q.stage_bytes = round_up((uint32_t)q.nph * q.act_stride + (uint32_t)(q.CB / 16) * q.w_chunk, 1024);
                q.red_pitch = (uint32_t)tile * 4u + 16u;
                const uint32_t red = round_up((uint32_t)ks * q.rpr * q.red_pitch, 128);
                const uint32_t fixed = red + round_up((uint32_t)tile * 4u, 128) + (uint32_t)sizeof(ConvSkBars) + 1024u + 128u;
                if (fixed + q.stage_bytes > kSmemLimit) continue;
                q.S = (int)((kSmemLimit - fixed) / q.stage_bytes);
                if (q.S > q.bpr) q.S = q.bpr;
                if (q.S > kMaxStages) q.S = kMaxStages;
                if ((uint32_t)q.S * q.stage_bytes >= (1u << 18)) continue;               // descriptor addresses are 14 bits of 16 bytes
                q.off_red = (uint32_t)q.S * q.stage_bytes;
                q.off_bias = q.off_red + red;
                q.off_bar = q.off_bias + round_up((uint32_t)tile * 4u, 128);
                q.smem_bytes = q.off_bar + (uint32_t)sizeof(ConvSkBars) + 1024u;
                q.tmem_cols = 32;
                while ((int)q.tmem_cols < tile) q.tmem_cols *= 2;
                const double cost = modelled(q, sms);
                if (!found || cost < best) { best = cost; p = q; found = true; }
            }
    }
    return found;
}

bool planned(const npas_conv_desc &d, const npas_bp_desc &bp, ConvSkParams &p, bool one_wave)
{
    return cached_plan(d, bp, one_wave, p, [&](ConvSkParams &q) { return plan(d, bp, q, sm_count(), one_wave); });
}

}  // namespace

bool conv_sk_supported(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvSkParams p;
    return planned(d, bp, p, false);
}

// Measured against the persistent kernels (this one, then the better of the two, both in a chain of layers): 14x14x256 -> 256 one image 4.8 against
// 9.9 us, four 6.7 against 10.1, eight 8.1 against 10.2; 7x7x512 -> 512 5.8 against 14.6; 7x27x29x96 -> 160 7.8 against 8.3;
// 54x6x33x160 -> 32 (108 position tiles) 8.0 against 6.9.  So: one wave, and no more position tiles than half the SMs.
// Strided 3x3 layers off multiples of 64 channels or filters come here unless the pair kernel's wide form is modelled faster
// (conv_d2.cu): the single-CTA kernel computes every position (12x19x50x144 -> 208 8.9 against 36 us); the others, when
// there are channels to split, one wave, and the pair kernel is not modelled faster (14x14x512 -> 512 5.8 against 17.1 us;
// 59x17x48x512 -> 64 38.6 against 19.3).
// The plan is part of the answer: what is launched is what was compared.
static bool choose(const npas_conv_desc &d, const npas_bp_desc &bp, ConvSkParams &p)
{
    const int sms = sm_count();
    if (d.variant) return false;
    const bool phases = d.stride == 2 && d.R == 3 && d.S == 3 && d.pad == 1;
    if (phases && (d.C % 64 || d.K % 64)) return planned(d, bp, p, false);
    const bool pairs = conv_d2_supported(d, bp);
    if (planned(d, bp, p, true) && (phases ? p.nBlk > 1 && modelled(p, sms) <= conv_dense_modelled(d, bp) : p.n_tiles * 2 <= sms)) return true;
    // several waves: against independent CTAs, whose tile is as narrow as the image's groups (11x15x25x416 -> 464 51 against 63 us)
    return d.stride == 1 && !pairs && planned(d, bp, p, false) && 1.05 * modelled(p, sms) < conv_dense_modelled(d, bp);
}

static bool chosen(const npas_conv_desc &d, const npas_bp_desc &bp, ConvSkParams &p)
{
    return cached_plan(d, bp, 0, p, [&](ConvSkParams &q) { return choose(d, bp, q); });
}

bool conv_sk_preferred(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvSkParams p;
    return chosen(d, bp, p);
}

// A stride-1 layer of this kernel's range that the pair kernel does sooner, by the models of both: many channels on just under
// half a wave of position tiles, where one wave leaves too few CTAs to split the chain (6x30x30x512 -> 128 21.0 us here, 15.1
// on pairs; 39x6x7x512 -> 128 15.6 and 14.2).
bool conv_sk_slower(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvSkParams p;
    return !d.variant && d.stride == 1 && planned(d, bp, p, true) && modelled(p, sm_count()) > conv_dense_modelled(d, bp);
}

// microseconds of the form that an automatic choice of this kernel would run; where it would not, more than any other takes
double conv_sk_modelled(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvSkParams p;
    return chosen(d, bp, p) ? modelled(p, sm_count()) : 1e30;
}

static int32_t shape_of(const ConvSkParams &p) { return p.NT | (p.KC << 16) | (p.KT << 24); }

// the shape an automatic choice of this kernel runs, as a `variant` (0: none)
int32_t conv_sk_variant(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvSkParams p;
    return chosen(d, bp, p) ? shape_of(p) : 0;
}

// Shapes worth timing, as `variant`s: those that the model (9 % standard error) puts within a quarter of its best one, where that
// is not modelled half as slow again as the other dense-image kernels.
int conv_sk_shapes(const npas_conv_desc &d, const npas_bp_desc &bp, int32_t *variants, int cap)
{
    npas_conv_desc q = d;
    q.variant = 0;
    ConvSkParams p;
    const int sms = sm_count();
    if (!planned(q, bp, p, false)) return 0;
    const double best = modelled(p, sms);
    if (best > 1.5 * conv_dense_modelled(q, bp)) return 0;
    int n = 0;
    for (int nt = 16; nt <= 128 && nt <= d.K; nt += 16)
        for (int kc = 1; kc <= kMaxSplit; ++kc)
            for (int kt = 1; kc * kt <= kMaxSplit && kt <= 4; ++kt) {
                q.variant = nt | (kc << 16) | (kt << 24);
                if (n < cap && plan(q, bp, p, sms, false) && modelled(p, sms) <= 1.25 * best) variants[n++] = q.variant;
            }
    return n;
}

npas_status conv_sk_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x, const void *blob, const float *bias,
                           const void *res, void *y, uint32_t *ws, cudaStream_t st, Launch how)
{
    ConvSkParams p;
    if (d.variant ? !planned(d, bp, p, false) : !chosen(d, bp, p)) return NPAS_ERR_UNSUPPORTED;
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return NPAS_ERR_CUDA;
    // X[N][H][W][C] as (C, W, H, N): a box of CB channels x Wp columns x slab rows (every other pixel for a parity class)
    CUtensorMap tmx, tmw;
    const cuuint64_t dims[4] = {(cuuint64_t)d.C, (cuuint64_t)d.W, (cuuint64_t)d.H, (cuuint64_t)d.N};
    const cuuint64_t strides[3] = {(cuuint64_t)d.C * 2, (cuuint64_t)d.W * d.C * 2, (cuuint64_t)d.H * d.W * d.C * 2};
    const cuuint32_t step = p.nph == 4 ? 2 : 1;
    const cuuint32_t box[4] = {(cuuint32_t)p.CB, (cuuint32_t)p.Wp * step, (cuuint32_t)p.slab_rows * step, 1}, estr[4] = {1, step, step, 1};
    const CUtensorMapSwizzle sw = p.CB == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : p.CB == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    if (enc(&tmx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return NPAS_ERR_CUDA;
    // The blob's image as (64 elements of a line, lines of a group's row, groups, rows of all (chunk, tap, octet)).  The map
    // covers the blob from its start (where the image begins only the header knows) and is given the length of a blob that
    // keeps everything; the kernel asks for rows of the image only, which every blob of this description holds in full.
    const uint32_t all_pairs = (uint32_t)(bp.K / bp.Mb) * (uint32_t)(bp.C / bp.Nb) * (uint32_t)p.RS, grow = (uint32_t)p.GI * 16u;
    const cuuint64_t wdims[4] = {64, (cuuint64_t)(p.GI / 8), (cuuint64_t)(d.K / p.GI), (cuuint64_t)(bp_layout(bp, all_pairs).total / grow)};
    const cuuint64_t wstr[3] = {128, (cuuint64_t)p.nCh * p.RS * 2u * grow, grow};
    const cuuint32_t wbox[4] = {64, (cuuint32_t)p.lines, (cuuint32_t)(p.NT < p.GI ? 1 : p.NT / p.GI), (cuuint32_t)(2 * p.tpr)}, wes[4] = {1, 1, 1, 1};
    if (enc(&tmw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(blob), wdims, wstr, wbox, wes, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return NPAS_ERR_CUDA;
    if (allow_dynamic_smem(reinterpret_cast<const void *>(conv_bp_sk_kernel), (int)kSmemLimit) != NPAS_OK) return NPAS_ERR_CUDA;
    const int KS = p.KC * p.KT;
    p.early = how.blob_ready;
    const cudaError_t e = launch_pdl_cluster(how, conv_bp_sk_kernel, dim3(p.n_tiles * p.nFT * KS), dim3(kThreads), KS, p.smem_bytes, st, tmx, tmw, p,
                                             static_cast<const uint8_t *>(blob), bias, res, y, ws);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // namespace npas
