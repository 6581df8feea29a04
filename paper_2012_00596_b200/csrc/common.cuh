// Shared host/device helpers of the library: blob header views, bf16 conversion, launch
// accounting and argument checks.  Nothing here is visible through the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>
#include <atomic>

#include "npas.h"

namespace npas {

constexpr uint32_t kMagicBP = 0x5042504Eu;  // 'NPBP'
constexpr uint32_t kMagicBB = 0x4242504Eu;  // 'NPBB'
constexpr uint32_t kVersion = 4;
constexpr uint32_t kAbiVersion = 1;

// Field indices of the 32-word blob headers (layout documented in npas.h).
enum BpHdr { BP_MAGIC, BP_VERSION, BP_DTYPE, BP_K, BP_C, BP_R, BP_S, BP_MB, BP_NB, BP_NFB, BP_NCB,
             BP_NPAIRS, BP_OFF_BLK, BP_OFF_PAIRS, BP_OFF_VALUES, BP_TOTAL, BP_G, BP_OFF_IMAGE, BP_OFF_TAPU, BP_GI,
             BP_OFF_KTOFF, BP_OFF_KT, BP_GS, BP_NKT };
enum BbHdr { BB_MAGIC, BB_VERSION, BB_DTYPE, BB_O, BB_I, BB_BO, BB_BI, BB_NBO, BB_NBI, BB_NVALS,
             BB_OFF_CNT, BB_OFF_ROWS, BB_OFF_COLS, BB_OFF_VOFF, BB_OFF_VALUES, BB_TOTAL, BB_KP, BB_OFF_TILES,
             BB_OFF_DENSE };
constexpr uint32_t kVersionBB = 3;

// Section offsets of a block-punched blob, computed on the host from the descriptor and nPairs.
// Microseconds of the GEMM kernels with both operands by TMA, columns in tiles of `bn`, on CTAs (128 rows a tile) or on CTA
// pairs (256 rows): fitted to 583 measured points (110 random layers, four widths on CTAs and three on pairs; standard error
// 8 and 7 %; the width and kernel it picks take 0.6 % more than the best measured on average, 8 % at worst).  Rounds of tiles
// x (K steps, a part of which grows with the width, and the epilogue), and the bytes that cross DRAM.  Wide tiles read the
// input less often, narrow ones fill a last round better: 42389 x 1920 -> 256 takes 52 us on CTAs and 40 on pairs,
// 9089 x 384 -> 576 12 us in tiles of 64 and 8 in tiles of 192, 1619 x 128 -> 512 5.5 us in tiles of 256 and 3.9 of 64.
inline double linear_modelled(const npas_linear_desc &d, int bn, bool pair, int sms)
{
    const int nK = (d.I + 63) / 64, nMT = (d.M + 127) / 128, nNT = (d.O + bn - 1) / bn, cap = pair ? sms / 2 : sms;
    const double tiles = (double)(pair ? (nMT + 1) / 2 : nMT) * nNT, r = (double)(((long long)tiles + cap - 1) / (cap > 0 ? cap : 1));
    const double out = (d.has_residual ? 2. : 1.) * (d.y_dtype == NPAS_BF16 ? 1. : 2.);
    const double mb = 2e-6 * ((double)d.M * d.I + out * d.M * d.O + (double)d.I * d.O);
    return pair ? 3.32 + r * (nK * (0.0973 + 0.00067 * bn) + 0.0017 * bn * out + 0.43) + 0.061 * mb
                : 3.02 + r * (nK * (0.1706 + 0.00070 * bn) + 0.0026 * bn * out + 0.14) + 0.037 * mb + 1.8e-7 * tiles * nK * (128 + bn);
}

struct BpLayout {
    uint32_t nFB, nCB, nPairs, G, es;
    uint32_t off_blk, off_pairs, off_values, total;
    uint32_t off_image, off_tapu, GI;          // dense operand image (bf16, C % 16 == 0 only; else 0)
    uint32_t off_ktoff, off_kt, GS, nKt, nGrp;  // kept 16-channel tiles by (chunk, filter group, tap); else 0
};
struct BbLayout {
    uint32_t nBo, nBi, nBlk, es;
    uint32_t off_cnt, off_rows, off_cols, off_voff, off_dense, off_values;  // total needs nVals
};

__host__ __device__ inline uint32_t round_up(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }
__host__ __device__ inline uint32_t dtype_size(int dt) { return dt == NPAS_F32 ? 4u : 2u; }

__host__ __device__ inline BpLayout bp_layout(const npas_bp_desc &d, uint32_t nPairs)
{
    BpLayout L;
    L.nFB = d.K / d.Mb; L.nCB = d.C / d.Nb; L.nPairs = nPairs;
    L.G = (d.Nb % 8 == 0) ? 8 : d.Nb;
    L.es = dtype_size(d.w_packed);
    L.off_blk = 128;
    L.off_pairs = round_up(L.off_blk + 4 * (L.nFB * L.nCB + 1), 128);
    L.off_values = round_up(L.off_pairs + 4 * nPairs, 128);
    L.total = L.off_values + round_up(nPairs * d.Mb * d.Nb * L.es, 128);
    // filters per group of the operand image: the largest power of two <= 128 that divides K
    L.GI = 128;
    while (d.K % L.GI) L.GI >>= 1;
    L.off_image = 0; L.off_tapu = 0;
    if (d.w_packed == NPAS_BF16 && d.C % 16 == 0) {
        L.off_image = round_up(L.total, 2048);     // on a multiple of a 128-filter row, so that tensor maps over the blob can count in rows
        L.off_tapu = L.off_image + round_up((uint32_t)d.K * d.R * d.S * d.C * 2u, 128);
        L.total = L.off_tapu + round_up((uint32_t)(d.K / L.GI) * (d.C / 16) * 4u, 128);
    }
    // kept weights as tiles of Mb filters x 16 channels, grouped for the kept-only tensor-core kernel
    uint32_t fgw = 256;
    while (d.K % fgw) fgw >>= 1;
    L.off_ktoff = 0; L.off_kt = 0; L.GS = 0; L.nKt = 0; L.nGrp = 0;
    if (d.w_packed == NPAS_BF16 && d.Mb % 16 == 0 && d.Nb % 16 == 0 && d.R * d.S <= 16 && fgw % d.Mb == 0) {
        L.GS = fgw / d.Mb;
        L.nGrp = d.K / fgw;
        L.nKt = nPairs * (d.Nb / 16);
        L.off_ktoff = L.total;
        L.off_kt = L.off_ktoff + round_up(4u * ((uint32_t)(d.C / 16) * L.nGrp + 1u), 128);
        L.total = L.off_kt + round_up(L.nKt * (uint32_t)d.Mb * 32u, 128);
    }
    return L;
}

inline BbLayout bb_layout(const npas_bb_desc &d)
{
    BbLayout L;
    L.nBo = d.O / d.Bo; L.nBi = d.I / d.Bi; L.nBlk = L.nBo * L.nBi;
    L.es = dtype_size(d.w_packed);
    L.off_cnt = 128;
    L.off_rows = round_up(L.off_cnt + 2 * L.nBlk, 128);
    L.off_cols = round_up(L.off_rows + d.Bo * L.nBlk, 128);
    L.off_voff = round_up(L.off_cols + d.Bi * L.nBlk, 128);
    L.off_dense = round_up(L.off_voff + 4 * (L.nBlk + 1), 128);
    L.off_values = L.off_dense + round_up((uint32_t)d.O * d.I * L.es, 128);
    return L;
}

// float32 -> bf16 bits, round to nearest even on the bit pattern; NaN keeps sign / upper payload.
__host__ __device__ inline uint16_t f32_bits_to_bf16(uint32_t b)
{
    if ((b & 0x7F800000u) == 0x7F800000u && (b & 0x007FFFFFu) != 0u)
        return (uint16_t)((b >> 16) | 0x0040u);
    return (uint16_t)((b + 0x7FFFu + ((b >> 16) & 1u)) >> 16);
}
__device__ inline float bf16_bits_to_f32(uint16_t h) { return __uint_as_float(((uint32_t)h) << 16); }

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline npas_status check_bp_desc(const npas_bp_desc *d)
{
    if (!d) return NPAS_ERR_NULL;
    if (d->K <= 0 || d->C <= 0 || d->R <= 0 || d->S <= 0 || d->Mb <= 0 || d->Nb <= 0) return NPAS_ERR_SHAPE;
    if (d->K % d->Mb || d->C % d->Nb || d->R * d->S > 64) return NPAS_ERR_SHAPE;
    if (d->C >= 65536 || d->Mb > 4096 || d->Nb > 4096 || d->max_taps < 0) return NPAS_ERR_SHAPE;
    if ((uint64_t)d->K * d->R * d->S * (uint64_t)d->C > (1ull << 28)) return NPAS_ERR_SHAPE;   // blob offsets are 32-bit
    if ((d->w_in != NPAS_F32 && d->w_in != NPAS_BF16) || (d->w_packed != NPAS_F32 && d->w_packed != NPAS_BF16))
        return NPAS_ERR_DTYPE;
    if (d->w_in == NPAS_BF16 && d->w_packed == NPAS_F32) return NPAS_ERR_DTYPE;
    return NPAS_OK;
}

inline npas_status check_bb_desc(const npas_bb_desc *d)
{
    if (!d) return NPAS_ERR_NULL;
    if (d->O <= 0 || d->I <= 0 || d->Bo <= 0 || d->Bi <= 0) return NPAS_ERR_SHAPE;
    if (d->Bo > 64 || d->Bi > 64 || d->O % d->Bo || d->I % d->Bi || d->max_cols < 0) return NPAS_ERR_SHAPE;
    if ((uint64_t)d->O * (uint64_t)d->I > (1ull << 27)) return NPAS_ERR_SHAPE;      // blob offsets are 32-bit
    if ((d->w_in != NPAS_F32 && d->w_in != NPAS_BF16) || (d->w_packed != NPAS_F32 && d->w_packed != NPAS_BF16))
        return NPAS_ERR_DTYPE;
    if (d->w_in == NPAS_BF16 && d->w_packed == NPAS_F32) return NPAS_ERR_DTYPE;
    return NPAS_OK;
}

// Process-wide count of kernels launched by this library.
std::atomic<uint64_t> &launch_counter();
inline void count_launch(uint64_t n = 1) { launch_counter().fetch_add(n, std::memory_order_relaxed); }

inline npas_status launch_status()
{
    return cudaGetLastError() == cudaSuccess ? NPAS_OK : NPAS_ERR_CUDA;
}

// Multiprocessors of the current device.
int sm_count();

// Plans (tile shapes, shared-memory layouts, the kernel chosen) follow from the two descriptors, the device's SM count and
// `tag` alone, and a program calls the same layers again and again: each thread keeps the last ones it made, one per slot
// of a small table (a call on a known layer then spends about 20 ns here instead of up to 2 us of search).
template <typename P, typename D, typename B, typename F>
inline bool cached_plan(const D &d, const B &b, int tag, P &p, F make)
{
    static_assert(sizeof(D) % 4 == 0 && sizeof(B) % 4 == 0, "descriptors are 32-bit words");
    struct Entry { D d; B b; int sms, tag; bool used, ok; P p; };
    constexpr uint32_t kSlots = 64;
    static thread_local Entry table[kSlots];
    const int sms = sm_count();
    uint32_t h = 2166136261u ^ (uint32_t)tag;
    for (const uint32_t *w = reinterpret_cast<const uint32_t *>(&d), *e = w + sizeof(D) / 4; w != e; ++w) h = (h ^ *w) * 16777619u;
    for (const uint32_t *w = reinterpret_cast<const uint32_t *>(&b), *e = w + sizeof(B) / 4; w != e; ++w) h = (h ^ *w) * 16777619u;
    Entry &t = table[(h ^ (h >> 16)) % kSlots];
    if (!t.used || t.sms != sms || t.tag != tag || memcmp(&t.d, &d, sizeof(D)) || memcmp(&t.b, &b, sizeof(B))) {
        t.used = false;
        t.ok = make(t.p);
        t.d = d; t.b = b; t.sms = sms; t.tag = tag;
        t.used = true;
    }
    if (t.ok) p = t.p;
    return t.ok;
}
npas_status allow_dynamic_smem(const void *kernel, int bytes);     // once per (kernel, device)

// How a compute kernel follows what is ahead of it in its stream (launch_pdl in tc_common.cuh has the rule).
struct Launch {
    bool plain = false;            // after everything ahead of it has ended, instead of as a programmatic dependent
    bool blob_ready = false;       // nothing has written the blob since before a launch of this chain that was `plain`
};

// Words of the caller's workspace.
enum WsWord { WS_STATUS = 0, WS_DETAIL = 1 };

// ---- kernels implemented in the other translation units (host launchers) ------------------------
npas_status conv_simt_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                             const void *blob, const float *bias, const void *res, void *y,
                             cudaStream_t st, Launch how);
bool conv_tc_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
npas_status conv_tc_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y,
                           uint32_t *ws, cudaStream_t st);
bool conv_stem_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_stem_pool_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
npas_status conv_stem_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                             const void *blob, const float *bias, void *y, uint32_t *ws, cudaStream_t st,
                             bool pool, Launch how);
bool conv_stem_rows_supported(const npas_conv_desc &d, const npas_bp_desc &bp, bool pool);
npas_status conv_stem_rows_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x, const void *blob,
                                  const float *bias, void *y, uint32_t *ws, cudaStream_t st, bool pool, Launch how);
bool conv_dn_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
npas_status conv_dn_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y,
                           uint32_t *ws, cudaStream_t st, Launch how);
bool conv_sk_preferred(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_sk_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
int32_t conv_sk_variant(const npas_conv_desc &d, const npas_bp_desc &bp);
int conv_sk_shapes(const npas_conv_desc &d, const npas_bp_desc &bp, int32_t *variants, int cap);
npas_status conv_sk_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y,
                           uint32_t *ws, cudaStream_t st, Launch how);
bool conv_d2_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_d2_preferred(const npas_conv_desc &d, const npas_bp_desc &bp);
double conv_dense_modelled(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_sk_slower(const npas_conv_desc &d, const npas_bp_desc &bp);
double conv_sk_modelled(const npas_conv_desc &d, const npas_bp_desc &bp);
double conv_d2_wide_modelled(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_d2_wide_preferred(const npas_conv_desc &d, const npas_bp_desc &bp);
int32_t conv_d2_wide_variant();
npas_status conv_d2_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y,
                           uint32_t *ws, cudaStream_t st, Launch how, bool wide);
bool conv_kr_supported(const npas_conv_desc &d, const npas_bp_desc &bp);
bool conv_kr_preferred(const npas_conv_desc &d, const npas_bp_desc &bp);
npas_status conv_kr_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y,
                           uint32_t *ws, cudaStream_t st, Launch how);
npas_status linear_simt_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                               const void *blob, const float *bias, const void *res, void *y, cudaStream_t st, Launch how);
bool linear_dn_supported(const npas_linear_desc &d, const npas_bb_desc &bb);
float linear_dn_cost(const npas_linear_desc &d, const npas_bb_desc &bb);
npas_status linear_dn_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                             const void *blob, const float *bias, const void *res, void *y, uint32_t *ws,
                             cudaStream_t st, Launch how);
bool linear_sk_supported(const npas_linear_desc &d, const npas_bb_desc &bb);
bool linear_sk_preferred(const npas_linear_desc &d, const npas_bb_desc &bb);
int32_t linear_sk_variant(const npas_linear_desc &d, const npas_bb_desc &bb);
npas_status linear_sk_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                             const void *blob, const float *bias, const void *res, void *y, uint32_t *ws,
                             cudaStream_t st, Launch how);
bool linear_d2_supported(const npas_linear_desc &d, const npas_bb_desc &bb);
float linear_d2_cost(const npas_linear_desc &d, const npas_bb_desc &bb);
npas_status linear_d2_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                             const void *blob, const float *bias, const void *res, void *y, uint32_t *ws,
                             cudaStream_t st, Launch how);
bool linear_two_preferred(const npas_linear_desc &a, const npas_linear_desc &b);
npas_status linear_two_launch(const npas_linear_desc &a, const npas_bb_desc &bba, const npas_linear_desc &b, const npas_bb_desc &bbb, const void *x,
                              const void *blob1, const float *bias1, const void *res, void *y1, const void *blob2, const float *bias2, void *y2,
                              uint32_t *ws, cudaStream_t st, Launch how);
bool linear_tc_supported(const npas_linear_desc &d, const npas_bb_desc &bb);
npas_status linear_tc_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                             const void *blob, const float *bias, const void *res, void *y, uint32_t *ws,
                             cudaStream_t st);

}  // namespace npas
