// Packers and mask helpers: dense weights + block masks <-> the blobs described in npas.h.
// These run once per layer (offline with respect to inference; in a search, once per candidate layer).  All index output
// is integer work and all value output is a bit copy or a single round-to-nearest-even conversion.  A blob is written
// once, section by section, zeros included: one CTA scans the masks, then a grid writes the sections 16 bytes per thread.
// (Clearing the blob first and placing two-byte values one by one took twice the bytes and partial writes: 512x3x3x512 with
// 16x8 blocks 14 us of placing after 10 of scanning.)
//
// Two callers.  The C calls are given a blob and do not know what the masks on the device keep: the scan writes header,
// offsets and the bytes between the sections, and the grid reads the sections' places from the header.  The binding allocates
// the blob itself and needs its size first: the scan ("plan") reads the caller's words once, keeps a copy of them and the
// prefix sums in scratch memory, and posts the two counts that the size follows from as one word of page-locked memory, as
// soon as they are known; the grid then has everything from its arguments and the scratch memory, and its last CTAs
// write header, offsets and gaps.  What counts there is the way to the host and back.
#include "common.cuh"
#include "internal_api.h"
#include "tc_common.cuh"

#include <type_traits>

namespace npas {

// ------------------------------------------------------------------------------------------------
// Exclusive prefix sum of `count(i)` for i < n into out[0..n] by ONE block of 1024 threads, four consecutive items per
// thread and step.
template <typename F>
__device__ void block_exclusive_scan(uint32_t n, F count, uint32_t *out, uint32_t *smem /* 33 words */)
{
    const uint32_t t = threadIdx.x, lane = t & 31, wid = t >> 5;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < n; base += 4096) {
        const uint32_t i0 = base + 4 * t;
        uint32_t c[4], sum = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) { c[j] = i0 + j < n ? count(i0 + j) : 0u; sum += c[j]; }
        uint32_t up = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, up, d); if (lane >= (uint32_t)d) up += v; }
        if (lane == 31) smem[wid] = up;
        __syncthreads();
        if (wid == 0) {
            uint32_t w = smem[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, w, d); if (lane >= (uint32_t)d) w += v; }
            smem[lane] = w;
        }
        __syncthreads();
        uint32_t run = carry + up - sum + (wid ? smem[wid - 1] : 0u);
#pragma unroll
        for (int j = 0; j < 4; ++j) { if (i0 + j < n) out[i0 + j] = run; run += c[j]; }
        carry += smem[31];
        __syncthreads();
    }
    if (t == 0) out[n] = carry;
    __syncthreads();
}

// zeros in [lo, hi) of the blob (offsets are even)
__device__ void zero_gap(uint8_t *blob, uint32_t lo, uint32_t hi)
{
    for (uint32_t o = lo + 2 * threadIdx.x; o < hi; o += 2 * blockDim.x) *reinterpret_cast<uint16_t *>(blob + o) = 0;
}

__device__ __forceinline__ uint64_t live_bits(int n) { return n == 64 ? ~0ull : ((1ull << n) - 1); }

template <typename TIn, typename TOut> __device__ __forceinline__ TOut convert(TIn v)
{
    if constexpr (sizeof(TIn) == sizeof(TOut)) return v;
    else return f32_bits_to_bf16(v);
}

// A mask word of the caller's, read once (another stream may be changing it).
__device__ __forceinline__ uint64_t load_once(const uint64_t *p) { return *reinterpret_cast<const volatile uint64_t *>(p); }

// The counts a blob's size follows from, in one word: bit 63 says that they are there, `most` lies above bit 32.
__device__ __forceinline__ void post_counts(unsigned long long *host, uint32_t total, uint32_t most)
{
    *reinterpret_cast<volatile unsigned long long *>(host) = (1ull << 63) | ((unsigned long long)most << 32) | total;
}

// largest value of a block of 1024 threads (32 words of shared memory)
__device__ __forceinline__ uint32_t block_max(uint32_t v, uint32_t *smem)
{
    v = __reduce_max_sync(0xFFFFFFFFu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) smem[threadIdx.x >> 5] = v;
    __syncthreads();
    return __reduce_max_sync(0xFFFFFFFFu, smem[threadIdx.x & 31]);
}

// ---- block-punched ---------------------------------------------------------------------------

constexpr uint32_t kScanCounts = 32768;                  // blocks whose counts the scan keeps in shared memory

__device__ void bp_write_header(uint32_t *hdr, const npas_bp_desc &d, const BpLayout &L)
{
    hdr[BP_OFF_IMAGE] = L.off_image; hdr[BP_OFF_TAPU] = L.off_tapu; hdr[BP_GI] = L.GI;
    hdr[BP_OFF_KTOFF] = L.off_ktoff; hdr[BP_OFF_KT] = L.off_kt; hdr[BP_GS] = L.GS; hdr[BP_NKT] = L.nKt;
    hdr[BP_MAGIC] = kMagicBP;
    hdr[BP_VERSION] = kVersion; hdr[BP_DTYPE] = d.w_packed;
    hdr[BP_K] = d.K; hdr[BP_C] = d.C; hdr[BP_R] = d.R; hdr[BP_S] = d.S; hdr[BP_MB] = d.Mb; hdr[BP_NB] = d.Nb;
    hdr[BP_NFB] = L.nFB; hdr[BP_NCB] = L.nCB; hdr[BP_NPAIRS] = L.nPairs;
    hdr[BP_OFF_BLK] = 128; hdr[BP_OFF_PAIRS] = L.off_pairs; hdr[BP_OFF_VALUES] = L.off_values;
    hdr[BP_TOTAL] = L.total; hdr[BP_G] = L.G;
}

// zeros between the sections, and behind the last one (by one CTA)
__device__ void bp_zero_gaps(uint8_t *blob, uint32_t blob_bytes, const npas_bp_desc &d, const BpLayout &L)
{
    const uint32_t nBlk = L.nFB * L.nCB, values_end = L.off_values + L.nPairs * d.Mb * d.Nb * L.es;
    zero_gap(blob, L.off_blk + 4 * (nBlk + 1), L.off_pairs);
    zero_gap(blob, L.off_pairs + 4 * L.nPairs, L.off_values);
    zero_gap(blob, values_end, L.off_image ? L.off_image : L.total);
    if (L.off_image) {
        const uint32_t tapu_end = L.off_tapu + (uint32_t)(d.K / L.GI) * (d.C / 16) * 4u;
        zero_gap(blob, L.off_image + (uint32_t)d.K * d.R * d.S * d.C * 2u, L.off_tapu);
        zero_gap(blob, tapu_end, L.off_kt ? L.off_ktoff : L.total);
    }
    if (L.off_kt) {
        zero_gap(blob, L.off_ktoff + 4 * ((uint32_t)(d.C / 16) * L.nGrp + 1), L.off_kt);
        zero_gap(blob, L.off_kt + L.nKt * d.Mb * 32u, L.total);
    }
    zero_gap(blob, L.total, blob_bytes & ~1u);
    if (threadIdx.x == 0 && (blob_bytes & 1u)) blob[blob_bytes - 1] = 0;
}

// tiles per (16-channel chunk, group of GS filter blocks), chunk major, as prefix sums; counts of the blocks in cnt_s, or from the masks
__device__ void bp_scan_tiles(const npas_bp_desc &d, const BpLayout &L, const uint8_t *cnt_s, const uint64_t *masks, uint32_t *kt_off, uint32_t *sm)
{
    const uint32_t nCh = d.C / 16, cpb = d.Nb / 16;
    const uint64_t live = live_bits(d.R * d.S);
    block_exclusive_scan(nCh * L.nGrp, [&](uint32_t i) {
        const uint32_t ch = i / L.nGrp, g = i % L.nGrp, cb = ch / cpb;
        uint32_t n = 0;
        for (uint32_t fb = g * L.GS; fb < (g + 1) * L.GS; ++fb) {
            const uint32_t b = fb * L.nCB + cb;
            n += b < kScanCounts ? cnt_s[b] : (uint32_t)__popcll(masks[b] & live);
        }
        return n; }, kt_off, sm);
}

__global__ void __launch_bounds__(1024)
bp_scan_kernel(npas_bp_desc d, const uint64_t *__restrict__ tap_mask, uint8_t *blob, uint32_t blob_bytes)
{
    __shared__ uint32_t sm[33];
    __shared__ uint8_t cnt_s[kScanCounts];               // kept taps per block (for the second scan)
    tc::pdl_trigger();                                   // the section writers may fetch weights and masks meanwhile
    const uint32_t nBlk = (uint32_t)(d.K / d.Mb) * (d.C / d.Nb);
    const uint64_t live = live_bits(d.R * d.S);
    uint32_t *hdr = reinterpret_cast<uint32_t *>(blob);
    uint32_t *blk_off = reinterpret_cast<uint32_t *>(blob + 128);
    if (threadIdx.x < 32) hdr[threadIdx.x] = 0;
    block_exclusive_scan(nBlk, [&](uint32_t i) {
        const uint32_t c = (uint32_t)__popcll(tap_mask[i] & live);
        if (i < kScanCounts) cnt_s[i] = (uint8_t)c;
        return c; }, blk_off, sm);
    const BpLayout L = bp_layout(d, blk_off[nBlk]);
    if (L.total > blob_bytes) {
        // A blob that does not fit keeps magic 0 and every section offset 0 (only the size that
        // would have been needed is recorded); the later kernels write nothing.
        if (threadIdx.x == 0) hdr[BP_TOTAL] = L.total;
        return;
    }
    if (threadIdx.x == 0) bp_write_header(hdr, d, L);
    bp_zero_gaps(blob, blob_bytes, d, L);
    if (L.off_kt) bp_scan_tiles(d, L, cnt_s, tap_mask, reinterpret_cast<uint32_t *>(blob + L.off_ktoff), sm);
}

// What the plan of a block-punched layer leaves in scratch memory.
struct BpScratch {
    uint64_t *masks; uint32_t *blk_off, *kt_off;
    size_t bytes;
};
static BpScratch bp_scratch(const npas_bp_desc &d, void *base)
{
    const BpLayout L = bp_layout(d, 0);
    const size_t nBlk = (size_t)L.nFB * L.nCB, off_blk = (nBlk * 8 + 15) / 16 * 16, off_kt = off_blk + (nBlk + 1 + 3) / 4 * 16;
    uint8_t *b = static_cast<uint8_t *>(base);
    return {reinterpret_cast<uint64_t *>(b), reinterpret_cast<uint32_t *>(b + off_blk), reinterpret_cast<uint32_t *>(b + off_kt),
            off_kt + ((size_t)(d.C / 16) * L.nGrp + 1) * 4};
}

// (L: the layout without pairs; what this kernel needs of it does not depend on them)
__global__ void __launch_bounds__(1024)
bp_plan_kernel(npas_bp_desc d, BpLayout L, const uint64_t *words, BpScratch s, unsigned long long *host)
{
    __shared__ uint32_t sm[33];
    __shared__ uint8_t cnt_s[kScanCounts];
    const uint32_t nBlk = L.nFB * L.nCB;
    const uint64_t live = live_bits(d.R * d.S);
    uint32_t most = 0;
    tc::pdl_wait();
    block_exclusive_scan(nBlk, [&](uint32_t i) {
        const uint64_t m = load_once(words + i);
        const uint32_t c = (uint32_t)__popcll(m & live);
        s.masks[i] = m;
        most = max(most, c);
        if (i < kScanCounts) cnt_s[i] = (uint8_t)c;
        return c; }, s.blk_off, sm);
    most = block_max(most, sm);
    if (threadIdx.x == 0) post_counts(host, s.blk_off[nBlk], most);
    __syncthreads();
    if (L.off_kt) bp_scan_tiles(d, L, cnt_s, s.masks, s.kt_off, sm);
}

// Blobs without derived sections (fp32, or C % 16 != 0): one CTA per block (fb, cb) writes the block's pair words and
// gathers its kept weights in the order of the destination.
template <typename TIn, typename TOut>
__global__ void bp_gather_kernel(npas_bp_desc d, const TIn *__restrict__ w, const uint64_t *__restrict__ tap_mask,
                                 uint8_t *blob)
{
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
    if (hdr[BP_MAGIC] != kMagicBP) return;
    const uint32_t nCB = d.C / d.Nb, b = blockIdx.x, fb = b / nCB, cb = b % nCB;
    const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + 128);
    uint32_t *pairs = reinterpret_cast<uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
    TOut *vals = reinterpret_cast<TOut *>(blob + hdr[BP_OFF_VALUES]);
    const uint32_t G = hdr[BP_G], Mb = d.Mb, Nb = d.Nb;
    uint64_t bits = tap_mask[b] & live_bits(d.R * d.S);
    for (uint32_t j = blk_off[b]; bits; ++j, bits &= bits - 1) {
        const uint32_t tap = __ffsll((long long)bits) - 1;
        if (threadIdx.x == 0) pairs[j] = cb | (tap << 16);
        for (uint32_t e = threadIdx.x; e < Mb * Nb; e += blockDim.x) {
            const uint32_t cg = e / (Mb * G), f = (e / G) % Mb, cl = e % G, c = cg * G + cl;
            vals[(size_t)j * Mb * Nb + e] = convert<TIn, TOut>(w[((size_t)(fb * Mb + f) * (d.R * d.S) + tap) * d.C + cb * Nb + c]);
        }
    }
}

// SUB consecutive weights as bf16 bits, packed two to a word (SUB = 1: in the low half)
template <int SUB> struct Packed { uint32_t w[SUB >= 2 ? SUB / 2 : 1]; };
template <int SUB> __device__ __forceinline__ Packed<SUB> load_packed(const uint16_t *p)
{
    Packed<SUB> r;
    if constexpr (SUB == 8) { const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p)); r.w[0] = u.x; r.w[1] = u.y; r.w[2] = u.z; r.w[3] = u.w; }
    else if constexpr (SUB == 4) { const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p)); r.w[0] = u.x; r.w[1] = u.y; }
    else r.w[0] = __ldg(p);
    return r;
}
template <int SUB> __device__ __forceinline__ Packed<SUB> load_packed(const uint32_t *p)
{
    Packed<SUB> r;
    if constexpr (SUB == 1) r.w[0] = f32_bits_to_bf16(__ldg(p));
    else {
#pragma unroll
        for (int h = 0; h < SUB / 4; ++h) {
            const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p) + h);
            r.w[2 * h] = (uint32_t)f32_bits_to_bf16(u.x) | ((uint32_t)f32_bits_to_bf16(u.y) << 16);
            r.w[2 * h + 1] = (uint32_t)f32_bits_to_bf16(u.z) | ((uint32_t)f32_bits_to_bf16(u.w) << 16);
        }
    }
    return r;
}
template <int SUB> __device__ __forceinline__ void store_packed(uint16_t *p, const Packed<SUB> &r)
{
    if constexpr (SUB == 8) *reinterpret_cast<uint4 *>(p) = make_uint4(r.w[0], r.w[1], r.w[2], r.w[3]);
    else if constexpr (SUB == 4) *reinterpret_cast<uint2 *>(p) = make_uint2(r.w[0], r.w[1]);
    else *p = (uint16_t)r.w[0];
}

// Blobs with the derived sections.  A thread owns one 16-byte unit of the operand image (filter, tap, eight channels), in
// the image's order, so that image stores are whole lines; what it keeps also goes, SUB channels at a time, to the packed
// values and to the tile section.  SUB = 8 when a block's channels are whole octets (then a unit lies in one block), else
// 4 or 1.  The CTAs behind the last unit write the tap unions, a warp per (filter group, 16-channel chunk), and after a plan
// the ones behind those write header, offsets and gaps.
// PLANNED: the layout is whole, masks and prefix sums are in scratch memory, nothing is read before the plan has ended; else
// they are in the blob, which the scan ahead of this kernel may still be writing.
template <typename TIn, int SUB, bool PLANNED>
__global__ void __launch_bounds__(256)
bp_expand_kernel(npas_bp_desc d, BpLayout L, const TIn *__restrict__ w, const uint64_t *__restrict__ tap_mask, const uint32_t *__restrict__ blk_plan,
                 const uint32_t *__restrict__ kt_plan, uint8_t *blob, uint32_t blob_bytes, uint32_t unit_ctas, uint32_t union_ctas)
{
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
    const uint32_t RS = d.R * d.S, nCh = d.C / 16, Mb = d.Mb, Nb = d.Nb, nCB = L.nCB, GI = L.GI, lane = threadIdx.x & 31;
    const uint64_t live = live_bits((int)RS);
    if constexpr (PLANNED) {
        tc::pdl_wait();
        w = tc::behind_wait(w); tap_mask = tc::behind_wait(tap_mask); blk_plan = tc::behind_wait(blk_plan); kt_plan = tc::behind_wait(kt_plan);
        if (blockIdx.x >= unit_ctas + union_ctas) {
            const uint32_t n = L.nFB * L.nCB + 1, n_kt = L.off_kt ? nCh * L.nGrp + 1 : 0, cta = blockIdx.x - unit_ctas - union_ctas;
            uint32_t *blk = reinterpret_cast<uint32_t *>(blob + L.off_blk), *kt = reinterpret_cast<uint32_t *>(blob + L.off_ktoff);
            if (cta == 0) {
                if (threadIdx.x < 32) {
                    reinterpret_cast<uint32_t *>(blob)[threadIdx.x] = 0;
                    __syncwarp();
                    if (threadIdx.x == 0) bp_write_header(reinterpret_cast<uint32_t *>(blob), d, L);
                }
                bp_zero_gaps(blob, blob_bytes, d, L);
            }
#pragma unroll 4
            for (uint32_t i = cta * 256u + threadIdx.x; i < n + n_kt; i += (gridDim.x - unit_ctas - union_ctas) * 256u) {
                if (i < n) blk[i] = blk_plan[i];
                else kt[i - n] = kt_plan[i - n];
            }
            return;
        }
    }
    if (blockIdx.x >= unit_ctas) {
        const uint32_t item = (blockIdx.x - unit_ctas) * 8 + (threadIdx.x >> 5);
        if (item >= (d.K / GI) * nCh) return;
        const uint32_t gi = item / nCh, ch = item - gi * nCh;
        const uint32_t fb_lo = gi * GI / Mb, n_fb = ((gi + 1) * GI - 1) / Mb - fb_lo + 1, cb_lo = ch * 16 / Nb, n_cb = (ch * 16 + 15) / Nb - cb_lo + 1;
        uint32_t u = 0;
        for (uint32_t i = lane; i < n_fb * n_cb; i += 32) {
            const uint64_t m = tap_mask[(size_t)(fb_lo + i / n_cb) * nCB + cb_lo + i % n_cb] & live;
            if (m) u |= RS > 32 ? 0xFFFFFFFFu : (uint32_t)m;
        }
        u = __reduce_or_sync(0xFFFFFFFFu, u);
        tc::pdl_wait();
        if (lane == 0 && (PLANNED || hdr[BP_MAGIC] == kMagicBP)) reinterpret_cast<uint32_t *>(blob + (PLANNED ? L.off_tapu : hdr[BP_OFF_TAPU]))[item] = u;
        return;
    }
    const uint32_t u = blockIdx.x * 256u + threadIdx.x, units = (uint32_t)d.K * RS * (d.C / 8);
    const uint32_t gsh = 31 - __clz(GI), kl = u & (GI - 1), v = u >> gsh, oct = v & 1, x = v >> 1;
    const uint32_t y = x / RS, tap = x - y * RS, gi = y / nCh, ch = y - gi * nCh;
    const uint32_t k = gi * GI + kl, c0 = ch * 16 + oct * 8, fb = k / Mb, f = k - fb * Mb;
    const bool in = u < units;
    // masks and weights first (they do not depend on the scan, which may still be running), after a plan all there is to load
    uint64_t bits[8 / SUB], m2 = 0;
    uint32_t first[8 / SUB], kt0 = 0;
    Packed<SUB> r[8 / SUB];
    bool kept8 = false;
    const uint32_t GS = L.GS, grp = SUB == 8 && GS ? fb / GS : 0, cb0 = c0 / Nb;
#pragma unroll
    for (int h = 0; h < 8 / SUB; ++h) {
        const size_t b = (size_t)fb * nCB + (c0 + h * SUB) / Nb;
        bits[h] = in ? tap_mask[b] & live : 0ull;
        if constexpr (PLANNED) first[h] = in ? blk_plan[b] : 0u;
    }
    if (SUB == 8 && GS && in) {
        if (lane < GS) m2 = tap_mask[(size_t)(grp * GS + lane) * nCB + cb0] & live;
        if constexpr (PLANNED) kt0 = kt_plan[ch * L.nGrp + grp];
    }
#pragma unroll
    for (int h = 0; h < 8 / SUB; ++h)
        if ((bits[h] >> tap) & 1ull) {
            kept8 = true;
            r[h] = load_packed<SUB>(w + ((size_t)k * RS + tap) * d.C + c0 + h * SUB);
        }
    tc::pdl_wait();
    if (!PLANNED && hdr[BP_MAGIC] != kMagicBP) return;
    uint32_t *pairs = reinterpret_cast<uint32_t *>(blob + (PLANNED ? L.off_pairs : hdr[BP_OFF_PAIRS]));
    uint16_t *vals = reinterpret_cast<uint16_t *>(blob + (PLANNED ? L.off_values : hdr[BP_OFF_VALUES]));
    const uint32_t G = L.G;
    if constexpr (!PLANNED) {
        const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + 128);
#pragma unroll
        for (int h = 0; h < 8 / SUB; ++h)
            if ((bits[h] >> tap) & 1ull) first[h] = blk_off[(size_t)fb * nCB + (c0 + h * SUB) / Nb];
    }
    Packed<8> img;
    img.w[0] = img.w[1] = img.w[2] = img.w[3] = 0;
#pragma unroll
    for (int h = 0; h < 8 / SUB; ++h) {
        if (!((bits[h] >> tap) & 1ull)) continue;
        const uint32_t c = c0 + h * SUB, cb = c / Nb, cc = c - cb * Nb;
        if constexpr (SUB == 1) img.w[h >> 1] |= r[h].w[0] << (16 * (h & 1));
        else {
#pragma unroll
            for (int j = 0; j < SUB / 2; ++j) img.w[h * (SUB / 2) + j] = r[h].w[j];
        }
        const uint32_t j = first[h] + (uint32_t)__popcll(bits[h] & ((1ull << tap) - 1ull));
        if (f == 0 && cc == 0) pairs[j] = cb | (tap << 16);
        store_packed<SUB>(vals + ((size_t)(j * (Nb / G) + cc / G) * Mb + f) * G + cc % G, r[h]);
    }
    if (in) store_packed<8>(reinterpret_cast<uint16_t *>(blob + (PLANNED ? L.off_image : hdr[BP_OFF_IMAGE])) + (size_t)u * 8, img);
    if constexpr (SUB == 8) {
        // the tile of (chunk, tap, filter block): behind the tiles of lower taps of the whole group and those of the
        // group's lower blocks that keep this tap.  (A warp holds filters of one group and one tap: with tiles, GI is at
        // least 16, and two octets of 16 filters are a warp.)
        const uint32_t off_kt = PLANNED ? L.off_kt : hdr[BP_OFF_KT];
        if (off_kt && __any_sync(0xFFFFFFFFu, in)) {
            const uint32_t below = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popcll(m2 & ((1ull << tap) - 1ull)));
            const uint32_t keep = __ballot_sync(0xFFFFFFFFu, (m2 >> tap) & 1ull);
            if (kept8) {
                if constexpr (!PLANNED) kt0 = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_KTOFF])[ch * L.nGrp + grp];
                const size_t tile = (size_t)kt0 + below + __popc(keep & ((1u << (fb - grp * GS)) - 1u));
                store_packed<8>(reinterpret_cast<uint16_t *>(blob + off_kt) + tile * Mb * 16 + (((f / 8) * 2 + oct) * 8 + f % 8) * 8, img);
            }
        }
    }
}
template <typename T>
__global__ void bp_scatter_kernel(npas_bp_desc d, const uint8_t *__restrict__ blob, T *w_out, uint64_t *tap_mask_out)
{
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
    const uint32_t nCB = d.C / d.Nb, b = blockIdx.x, fb = b / nCB, cb = b % nCB;
    const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_BLK]);
    const uint32_t *pairs = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
    const T *vals = reinterpret_cast<const T *>(blob + hdr[BP_OFF_VALUES]);
    const uint32_t G = hdr[BP_G], Mb = d.Mb, Nb = d.Nb;
    uint64_t bits = 0;
    for (uint32_t j = blk_off[b]; j < blk_off[b + 1]; ++j) {
        const uint32_t tap = pairs[j] >> 16;
        if (tap >= (uint32_t)(d.R * d.S)) continue;            // (no tap of the layer: ignored)
        bits |= 1ull << tap;
        if (!w_out) continue;
        for (uint32_t e = threadIdx.x; e < Mb * Nb; e += blockDim.x) {
            const uint32_t cg = e / (Mb * G), f = (e / G) % Mb, cl = e % G, c = cg * G + cl;
            w_out[((size_t)(fb * Mb + f) * (d.R * d.S) + tap) * d.C + cb * Nb + c] = vals[(size_t)j * Mb * Nb + e];
        }
    }
    if (tap_mask_out && threadIdx.x == 0) tap_mask_out[b] = bits;
}

// dense 0/1 mask [K][R][S][C] -> per-block tap bitsets; counts blocks that break the scheme.
__global__ void bp_mask_from_dense_kernel(npas_bp_desc d, const uint8_t *__restrict__ m, uint64_t *tap_mask,
                                          int32_t *violations)
{
    const uint32_t nCB = d.C / d.Nb, b = blockIdx.x, fb = b / nCB, cb = b % nCB, RS = d.R * d.S;
    auto kernel_bits = [&](uint32_t f, uint32_t c) {
        uint64_t bits = 0;
        for (uint32_t t = 0; t < RS; ++t)
            if (m[((size_t)(fb * d.Mb + f) * RS + t) * d.C + cb * d.Nb + c]) bits |= 1ull << t;
        return bits;
    };
    const uint64_t ref = kernel_bits(0, 0);
    int bad = 0;
    for (uint32_t e = threadIdx.x; e < (uint32_t)(d.Mb * d.Nb); e += blockDim.x)
        bad |= kernel_bits(e / d.Nb, e % d.Nb) != ref;
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        tap_mask[b] = ref;
        if (bad) atomicAdd(violations, 1);
    }
}

// ---- block-based -----------------------------------------------------------------------------

// What follows from the counts.
struct BbTail { uint32_t nVals, Kp, off_tiles, tiles_end, total; };
__host__ __device__ inline BbTail bb_tail(const npas_bb_desc &d, const BbLayout &L, uint32_t nVals, uint32_t most)
{
    BbTail t;
    t.nVals = nVals;
    t.Kp = round_up(most, 16u) < 16u ? 16u : round_up(most, 16u);            // largest kept-column count, rounded up to 16
    t.off_tiles = L.off_values + round_up(nVals * L.es, 128);
    t.tiles_end = t.off_tiles + L.nBlk * t.Kp * (uint32_t)d.Bo * L.es;
    t.total = round_up(t.tiles_end, 128);
    return t;
}

__device__ void bb_write_header(uint32_t *hdr, const npas_bb_desc &d, const BbLayout &L, const BbTail &t)
{
    hdr[BB_MAGIC] = kMagicBB;
    hdr[BB_KP] = t.Kp; hdr[BB_OFF_TILES] = t.off_tiles; hdr[BB_OFF_DENSE] = L.off_dense;
    hdr[BB_VERSION] = kVersionBB; hdr[BB_DTYPE] = d.w_packed;
    hdr[BB_O] = d.O; hdr[BB_I] = d.I; hdr[BB_BO] = d.Bo; hdr[BB_BI] = d.Bi;
    hdr[BB_NBO] = L.nBo; hdr[BB_NBI] = L.nBi; hdr[BB_NVALS] = t.nVals;
    hdr[BB_OFF_CNT] = L.off_cnt; hdr[BB_OFF_ROWS] = L.off_rows; hdr[BB_OFF_COLS] = L.off_cols;
    hdr[BB_OFF_VOFF] = L.off_voff; hdr[BB_OFF_VALUES] = L.off_values; hdr[BB_TOTAL] = t.total;
}

// zeros between the sections (the lists are bytes, so single bytes here), and behind the last one (by one CTA)
__device__ void bb_zero_gaps(uint8_t *blob, uint32_t blob_bytes, const npas_bb_desc &d, const BbLayout &L, const BbTail &t)
{
    const uint32_t gaps[7][2] = {{L.off_cnt + 2 * L.nBlk, L.off_rows}, {L.off_rows + d.Bo * L.nBlk, L.off_cols},
                                 {L.off_cols + d.Bi * L.nBlk, L.off_voff}, {L.off_voff + 4 * (L.nBlk + 1), L.off_dense},
                                 {L.off_dense + (uint32_t)d.O * d.I * L.es, L.off_values}, {L.off_values + t.nVals * L.es, t.off_tiles},
                                 {t.tiles_end, blob_bytes}};
    for (int g = 0; g < 7; ++g)
        for (uint32_t o = gaps[g][0] + threadIdx.x; o < gaps[g][1]; o += blockDim.x) blob[o] = 0;
}

__global__ void __launch_bounds__(1024)
bb_scan_kernel(npas_bb_desc d, const uint64_t *__restrict__ row_keep,
               const uint64_t *__restrict__ col_keep, uint8_t *blob, uint32_t blob_bytes, BbLayout L)
{
    __shared__ uint32_t sm[33];
    tc::pdl_trigger();                                     // the section writers may fetch weights and masks meanwhile
    const uint64_t rlive = live_bits(d.Bo), clive = live_bits(d.Bi);
    uint32_t *hdr = reinterpret_cast<uint32_t *>(blob);
    uint32_t *voff = reinterpret_cast<uint32_t *>(blob + L.off_voff);
    if (threadIdx.x < 32) hdr[threadIdx.x] = 0;
    uint32_t most = 0;                                     // largest kept-column count
    block_exclusive_scan(L.nBlk, [&](uint32_t i) {
        const uint32_t nc = (uint32_t)__popcll(col_keep[i] & clive);
        most = max(most, nc);
        return round_up((uint32_t)__popcll(row_keep[i] & rlive) * nc, 8u); }, voff, sm);
    const BbTail T = bb_tail(d, L, voff[L.nBlk], block_max(most, sm));
    if (T.total > blob_bytes) {                            // magic and offsets stay 0: nothing is written
        if (threadIdx.x == 0) hdr[BB_TOTAL] = T.total;
        return;
    }
    if (threadIdx.x == 0) bb_write_header(hdr, d, L, T);
    bb_zero_gaps(blob, blob_bytes, d, L, T);
}

// What the plan of a block-based layer leaves in scratch memory.
struct BbScratch {
    uint64_t *rows, *cols; uint32_t *voff;
    size_t bytes;
};
static BbScratch bb_scratch(const BbLayout &L, void *base)
{
    uint8_t *b = static_cast<uint8_t *>(base);
    const size_t words = (size_t)L.nBlk * 8;
    return {reinterpret_cast<uint64_t *>(b), reinterpret_cast<uint64_t *>(b + words), reinterpret_cast<uint32_t *>(b + 2 * words), 2 * words + ((size_t)L.nBlk + 1) * 4};
}

__global__ void __launch_bounds__(1024)
bb_plan_kernel(npas_bb_desc d, uint32_t nBlk, const uint64_t *row_words, const uint64_t *col_words, BbScratch s, unsigned long long *host)
{
    __shared__ uint32_t sm[33];
    const uint64_t rlive = live_bits(d.Bo), clive = live_bits(d.Bi);
    uint32_t most = 0;
    tc::pdl_wait();
    block_exclusive_scan(nBlk, [&](uint32_t i) {
        const uint64_t r = load_once(row_words + i), c = load_once(col_words + i);
        const uint32_t nc = (uint32_t)__popcll(c & clive);
        s.rows[i] = r; s.cols[i] = c;
        most = max(most, nc);
        return round_up((uint32_t)__popcll(r & rlive) * nc, 8u); }, s.voff, sm);
    most = block_max(most, sm);
    if (threadIdx.x == 0) post_counts(host, s.voff[nBlk], most);
}

// One CTA per block: the block's weights are staged once, then its part of every section is written whole, zeros
// included, in the section's own order, in 16-byte pieces where the geometry allows (the values always: every block's start
// on a multiple of eight).  PLANNED: counts in T, masks and value offsets in scratch memory, and the CTA behind the last
// block writes the header and the gaps; else they are in the blob, which the scan ahead of this kernel may still be writing.
template <typename TIn, typename TOut, bool PLANNED>
__global__ void __launch_bounds__(256)
bb_gather_kernel(npas_bb_desc d, const TIn *__restrict__ w, const uint64_t *__restrict__ row_keep,
                 const uint64_t *__restrict__ col_keep, const uint32_t *__restrict__ voff_plan, uint8_t *blob, uint32_t blob_bytes, BbLayout L, BbTail T)
{
    constexpr uint32_t kV = 16 / sizeof(TOut), kP = 64 + kV;      // elements per 16 bytes; rows of the staged block, 16-byte aligned, on different banks
    __shared__ __align__(16) TOut blk_s[64 * kP];
    __shared__ uint8_t rows[64], cols[64];
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
    const uint32_t b = blockIdx.x, t = threadIdx.x, lane = t & 31, wid = t >> 5;
    if constexpr (PLANNED) {
        tc::pdl_wait();
        w = tc::behind_wait(w); row_keep = tc::behind_wait(row_keep); col_keep = tc::behind_wait(col_keep); voff_plan = tc::behind_wait(voff_plan);
    }
    if (PLANNED && b == L.nBlk) {
        uint32_t *h = reinterpret_cast<uint32_t *>(blob);
        if (t < 32) {
            h[t] = 0;
            __syncwarp();
            if (t == 0) {
                bb_write_header(h, d, L, T);
                reinterpret_cast<uint32_t *>(blob + L.off_voff)[L.nBlk] = T.nVals;
            }
        }
        bb_zero_gaps(blob, blob_bytes, d, L, T);
        return;
    }
    const uint32_t bo = b / L.nBi, bi = b % L.nBi, Bo = d.Bo, Bi = d.Bi;
    const TIn *src = w + (size_t)bo * Bo * d.I + (size_t)bi * Bi;
    TOut *dense = reinterpret_cast<TOut *>(blob + L.off_dense) + (size_t)bo * Bo * d.I + (size_t)bi * Bi;
    TIn v[8][2];                                           // (all loads in flight together)
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i)
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t r = wid + 8 * i, c = lane + 32 * h;
            v[i][h] = r < Bo && c < Bi ? __ldg(src + (size_t)r * d.I + c) : (TIn)0;
        }
    const uint64_t rk = row_keep[b] & live_bits(d.Bo), ck = col_keep[b] & live_bits(d.Bi);
    uint32_t v0 = 0;
    if constexpr (PLANNED) v0 = voff_plan[b];
    const uint32_t nr = __popcll(rk), nc = __popcll(ck);
    if (t < 64) {
        // rank of bit t among the set bits = its slot in the ascending list
        const uint64_t below = t == 0 ? 0ull : (~0ull >> (64 - t));
        if (t < Bo && (rk >> t) & 1) rows[__popcll(rk & below)] = (uint8_t)t;
        if (t < Bi && (ck >> t) & 1) cols[__popcll(ck & below)] = (uint8_t)t;
    }
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i)
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t r = wid + 8 * i, c = lane + 32 * h;
            blk_s[r * kP + c] = ((rk >> r) & (ck >> c) & 1ull) ? convert<TIn, TOut>(v[i][h]) : (TOut)0;
        }
    tc::pdl_wait();
    __syncthreads();
    uint32_t Kp = T.Kp, off_tiles = T.off_tiles;
    if constexpr (!PLANNED) {
        if (hdr[BB_MAGIC] != kMagicBB) return;
        Kp = hdr[BB_KP]; off_tiles = hdr[BB_OFF_TILES];
        v0 = reinterpret_cast<const uint32_t *>(blob + L.off_voff)[b];
    }
    if (Bi % kV == 0 && d.I % kV == 0) {
        const uint32_t per = Bi / kV;
        for (uint32_t e = t; e < Bo * per; e += 256) {
            const uint32_t r = e / per, c = (e - r * per) * kV;
            *reinterpret_cast<uint4 *>(dense + (size_t)r * d.I + c) = *reinterpret_cast<const uint4 *>(blk_s + r * kP + c);
        }
    } else {
#pragma unroll 8
        for (uint32_t r = wid; r < Bo; r += 8)
#pragma unroll
            for (uint32_t h = 0; h < 2; ++h) {
                const uint32_t c = lane + 32 * h;
                if (c < Bi) dense[(size_t)r * d.I + c] = blk_s[r * kP + c];
            }
    }
    if (t < Bo) blob[L.off_rows + b * Bo + t] = t < nr ? rows[t] : 0xFF;
    if (t < Bi) blob[L.off_cols + b * Bi + t] = t < nc ? cols[t] : 0xFF;
    if (t == 0) { blob[L.off_cnt + 2 * b] = (uint8_t)nr; blob[L.off_cnt + 2 * b + 1] = (uint8_t)nc; }
    if (PLANNED && t == 0) reinterpret_cast<uint32_t *>(blob + L.off_voff)[b] = v0;
    // 16 bytes from a list of elements
    auto gather16 = [&](TOut *dst, auto element) {
        TOut o[kV];
#pragma unroll
        for (uint32_t j = 0; j < kV; ++j) o[j] = element(j);
        if constexpr (sizeof(TOut) == 2)
            *reinterpret_cast<uint4 *>(dst) = make_uint4(o[0] | ((uint32_t)o[1] << 16), o[2] | ((uint32_t)o[3] << 16),
                                                         o[4] | ((uint32_t)o[5] << 16), o[6] | ((uint32_t)o[7] << 16));
        else *reinterpret_cast<uint4 *>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
    };
    // values [kept row][kept column], then zeros up to a multiple of eight elements
    TOut *vals = reinterpret_cast<TOut *>(blob + L.off_values) + v0;
    const uint32_t nv = nr * nc;
    for (uint32_t e = t * kV; e < round_up(nv, 8); e += 256 * kV) {
        uint32_t r = nc ? e / nc : 0, c = e - r * nc;
        gather16(vals + e, [&](uint32_t j) {
            const TOut x = e + j < nv ? blk_s[rows[r] * kP + cols[c]] : (TOut)0;
            if (++c == nc) { c = 0; ++r; }
            return x; });
    }
    // the operand image [Kp/8][Bo][8]: kept columns compacted, kept rows in place, zeros elsewhere
    TOut *tile = reinterpret_cast<TOut *>(blob + off_tiles) + (size_t)b * Kp * Bo;
    for (uint32_t e = t; e < Kp / kV * Bo; e += 256) {
        const uint32_t x = e / (8 / kV), h = e - x * (8 / kV), q = x / Bo, r = x - q * Bo, c = q * 8 + h * kV;
        const bool row_on = (rk >> r) & 1ull;
        gather16(tile + (size_t)x * 8 + h * kV, [&](uint32_t j) { return row_on && c + j < nc ? blk_s[r * kP + cols[c + j]] : (TOut)0; });
    }
}

// One CTA per block: the dense block is put together in shared memory and written whole, zeros included.
template <typename T>
__global__ void __launch_bounds__(256)
bb_scatter_kernel(npas_bb_desc d, const uint8_t *__restrict__ blob, T *w_out, uint64_t *rk_out,
                  uint64_t *ck_out, BbLayout L)
{
    constexpr uint32_t kV = 16 / sizeof(T), kP = 64 + kV;
    __shared__ __align__(16) T blk_s[64 * kP];
    __shared__ uint8_t rows[64], cols[64];
    const uint32_t b = blockIdx.x, bo = b / L.nBi, bi = b % L.nBi, t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const uint32_t Bo = d.Bo, Bi = d.Bi;
    if (w_out)
        for (uint32_t e = t; e < 64 * kP / kV; e += 256) reinterpret_cast<uint4 *>(blk_s)[e] = make_uint4(0, 0, 0, 0);
    tc::pdl_wait();
    blob = tc::behind_wait(blob);
    // (counts, lists and the values' place do not depend on one another: one round trip; entries behind a list's end are masked here)
    const uint16_t cnt = *reinterpret_cast<const uint16_t *>(blob + L.off_cnt + 2 * b);
    const uint8_t my_row = t < Bo ? blob[L.off_rows + b * Bo + t] : 0, my_col = t < Bi ? blob[L.off_cols + b * Bi + t] : 0;
    const uint32_t v0 = reinterpret_cast<const uint32_t *>(blob + L.off_voff)[b];
    const uint32_t nr = min((uint32_t)cnt & 0xFFu, Bo), nc = min((uint32_t)cnt >> 8, Bi);
    const T *vals = reinterpret_cast<const T *>(blob + L.off_values) + v0;
    // all values on their way: eight rows of two halves per warp
    T x[8][2];
    if (w_out) {
#pragma unroll
        for (uint32_t i = 0; i < 8; ++i)
#pragma unroll
            for (uint32_t h = 0; h < 2; ++h) x[i][h] = wid + 8 * i < nr && lane + 32 * h < nc ? vals[(wid + 8 * i) * nc + lane + 32 * h] : (T)0;
    }
    if (t < Bo) rows[t] = t < nr ? my_row & 63 : 0;
    if (t < Bi) cols[t] = t < nc ? my_col & 63 : 0;
    __syncthreads();
    if (wid == 0) {
        // the lists as bit sets
        uint64_t rk = 0, ck = 0;
        for (uint32_t i = lane; i < nr; i += 32) rk |= 1ull << rows[i];
        for (uint32_t i = lane; i < nc; i += 32) ck |= 1ull << cols[i];
        const uint32_t r0 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)rk), r1 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(rk >> 32));
        const uint32_t c0 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)ck), c1 = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(ck >> 32));
        if (lane == 0 && rk_out) rk_out[b] = (uint64_t)r0 | ((uint64_t)r1 << 32);
        if (lane == 0 && ck_out) ck_out[b] = (uint64_t)c0 | ((uint64_t)c1 << 32);
    }
    if (!w_out) return;
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i)
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h)
            if (wid + 8 * i < nr && lane + 32 * h < nc) blk_s[rows[wid + 8 * i] * kP + cols[lane + 32 * h]] = x[i][h];
    __syncthreads();
    T *out = w_out + (size_t)bo * Bo * d.I + (size_t)bi * Bi;
    if (Bi % kV == 0 && d.I % kV == 0) {
        const uint32_t per = Bi / kV;
        for (uint32_t e = t; e < Bo * per; e += 256) {
            const uint32_t r = e / per, c = (e - r * per) * kV;
            *reinterpret_cast<uint4 *>(out + (size_t)r * d.I + c) = *reinterpret_cast<const uint4 *>(blk_s + r * kP + c);
        }
    } else {
        for (uint32_t r = wid; r < Bo; r += 8)
            for (uint32_t c = lane; c < Bi; c += 32) out[(size_t)r * d.I + c] = blk_s[r * kP + c];
    }
}

__global__ void bb_mask_from_dense_kernel(npas_bb_desc d, const uint8_t *__restrict__ m, uint64_t *row_keep,
                                          uint64_t *col_keep, int32_t *violations, uint32_t nBi)
{
    __shared__ uint64_t rowbits[64];
    const uint32_t b = blockIdx.x, bo = b / nBi, bi = b % nBi, t = threadIdx.x;
    uint64_t mine = 0;
    if (t < (uint32_t)d.Bo)
        for (uint32_t c = 0; c < (uint32_t)d.Bi; ++c)
            if (m[(size_t)(bo * d.Bo + t) * d.I + bi * d.Bi + c]) mine |= 1ull << c;
    rowbits[t] = mine;
    __syncthreads();
    uint64_t ck = 0, rk = 0;
    for (uint32_t r = 0; r < (uint32_t)d.Bo; ++r) { ck |= rowbits[r]; if (rowbits[r]) rk |= 1ull << r; }
    const int bad = __syncthreads_or(t < (uint32_t)d.Bo && mine != 0 && mine != ck);
    if (t == 0) {
        row_keep[b] = rk; col_keep[b] = ck;
        if (bad) atomicAdd(violations, 1);
    }
}

// The size a blob needs is known only on the device (it depends on the masks there).  The scan
// kernel leaves the magic word 0 when the caller's buffer is too small; read it back and say so.
static npas_status packed_fits(const void *blob, int magic_word, uint32_t magic, cudaStream_t st)
{
    uint32_t m = 0;
    if (cudaMemcpyAsync(&m, static_cast<const uint32_t *>(blob) + magic_word, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    return m == magic ? NPAS_OK : NPAS_ERR_BUFFER_TOO_SMALL;
}

}  // namespace npas

using namespace npas;

// ================================================================================================
extern "C" {

npas_status npas_internal_bp_size(const npas_bp_desc *d, uint64_t n_pairs, size_t *blob_bytes)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (n_pairs * d->Mb * d->Nb * 4 > 0x7FFFFFFFull) return NPAS_ERR_SHAPE;
    *blob_bytes = bp_layout(*d, (uint32_t)n_pairs).total;
    return NPAS_OK;
}

npas_status npas_pack_bp_size(const npas_bp_desc *d, const uint64_t *tap_mask_host, size_t *blob_bytes)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!tap_mask_host || !blob_bytes) return NPAS_ERR_NULL;
    const uint64_t live = d->R * d->S == 64 ? ~0ull : ((1ull << (d->R * d->S)) - 1);
    uint64_t n = 0;
    for (int i = 0; i < (d->K / d->Mb) * (d->C / d->Nb); ++i) n += __builtin_popcountll(tap_mask_host[i] & live);
    return npas_internal_bp_size(d, n, blob_bytes);
}

// The section writers of a blob with derived sections.  plan: what npas_internal_plan_bp left, or null (then masks and a blob
// that the scan ahead writes).
static cudaError_t bp_expand_launch(const npas_bp_desc &d, const BpLayout &L, const void *w, const uint64_t *masks, const BpScratch *plan, uint8_t *blob,
                                    uint32_t blob_bytes, cudaStream_t st)
{
    const uint32_t units = (uint32_t)d.K * d.R * d.S * (d.C / 8), unit_ctas = (units + 255) / 256;
    const uint32_t union_ctas = ((uint32_t)(d.K / L.GI) * (d.C / 16) + 7) / 8;
    const uint32_t front = L.nFB * L.nCB + 1 + (L.off_kt ? (uint32_t)(d.C / 16) * L.nGrp + 1 : 0);
    const uint32_t grid = unit_ctas + union_ctas + (plan ? (front + 2047) / 2048 : 0);
    auto go = [&](auto sub, auto *wp) {
        using TIn = std::remove_const_t<std::remove_pointer_t<decltype(wp)>>;
        if (plan)
            return tc::launch_pdl({}, bp_expand_kernel<TIn, sub.value, true>, dim3(grid), dim3(256), 0, st, d, L, wp, masks,
                                  (const uint32_t *)plan->blk_off, (const uint32_t *)plan->kt_off, blob, blob_bytes, unit_ctas, union_ctas);
        return tc::launch_pdl({}, bp_expand_kernel<TIn, sub.value, false>, dim3(grid), dim3(256), 0, st, d, L, wp, masks, (const uint32_t *)nullptr,
                              (const uint32_t *)nullptr, blob, blob_bytes, unit_ctas, union_ctas);
    };
    auto by_width = [&](auto *wp) {
        if (d.Nb % 8 == 0) return go(std::integral_constant<int, 8>{}, wp);
        if (d.Nb % 4 == 0) return go(std::integral_constant<int, 4>{}, wp);
        return go(std::integral_constant<int, 1>{}, wp);
    };
    return d.w_in == NPAS_F32 ? by_width(static_cast<const uint32_t *>(w)) : by_width(static_cast<const uint16_t *>(w));
}

npas_status npas_internal_pack_bp(const npas_bp_desc *d, const void *w, const uint64_t *tap_mask, void *blob,
                                  size_t blob_bytes, void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!w || !tap_mask || !blob) return NPAS_ERR_NULL;
    if (!aligned16(w) || !aligned16(blob) || (reinterpret_cast<uintptr_t>(tap_mask) & 7)) return NPAS_ERR_ALIGNMENT;
    const BpLayout L = bp_layout(*d, 0);
    if (blob_bytes < L.total || blob_bytes > 0xFFFFFFFFull) return NPAS_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint32_t nBlk = (d->K / d->Mb) * (d->C / d->Nb);
    uint8_t *b8 = static_cast<uint8_t *>(blob);
    bp_scan_kernel<<<1, 1024, 0, st>>>(*d, tap_mask, b8, (uint32_t)blob_bytes);
    const uint32_t *w32 = static_cast<const uint32_t *>(w);
    const uint16_t *w16 = static_cast<const uint16_t *>(w);
    if (L.off_image) {
        if (bp_expand_launch(*d, L, w, tap_mask, nullptr, b8, (uint32_t)blob_bytes, st) != cudaSuccess) return NPAS_ERR_CUDA;
    } else if (d->w_packed == NPAS_F32)
        bp_gather_kernel<uint32_t, uint32_t><<<nBlk, 128, 0, st>>>(*d, w32, tap_mask, b8);
    else if (d->w_in == NPAS_F32)
        bp_gather_kernel<uint32_t, uint16_t><<<nBlk, 128, 0, st>>>(*d, w32, tap_mask, b8);
    else
        bp_gather_kernel<uint16_t, uint16_t><<<nBlk, 128, 0, st>>>(*d, w16, tap_mask, b8);
    count_launch(2);
    return launch_status();
}

npas_status npas_internal_plan_bp_bytes(const npas_bp_desc *d, size_t *bytes)
{
    npas_status s = check_bp_desc(d);
    if (s == NPAS_OK) *bytes = bp_scratch(*d, nullptr).bytes;
    return s;
}

npas_status npas_internal_plan_bp(const npas_bp_desc *d, const uint64_t *words, void *scratch, uint64_t *host, void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!words || !scratch || !host) return NPAS_ERR_NULL;
    if (!aligned16(scratch) || (reinterpret_cast<uintptr_t>(words) & 7)) return NPAS_ERR_ALIGNMENT;
    void *mapped = nullptr;
    if (cudaHostGetDevicePointer(&mapped, host, 0) != cudaSuccess) return NPAS_ERR_CUDA;
    const cudaError_t e = tc::launch_pdl({}, bp_plan_kernel, dim3(1), dim3(1024), 0, static_cast<cudaStream_t>(stream), *d, bp_layout(*d, 0), words,
                                         bp_scratch(*d, scratch), static_cast<unsigned long long *>(mapped));
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status npas_internal_pack_bp_planned(const npas_bp_desc *d, const void *w, void *scratch, uint64_t n_pairs, void *blob, size_t blob_bytes, void *stream)
{
    size_t need = 0;
    npas_status s = npas_internal_bp_size(d, n_pairs, &need);
    if (s != NPAS_OK) return s;
    if (!w || !scratch || !blob) return NPAS_ERR_NULL;
    if (!aligned16(w) || !aligned16(blob) || !aligned16(scratch)) return NPAS_ERR_ALIGNMENT;
    if (blob_bytes < need || blob_bytes > 0xFFFFFFFFull) return NPAS_ERR_BUFFER_TOO_SMALL;
    const BpLayout L = bp_layout(*d, (uint32_t)n_pairs);
    const BpScratch plan = bp_scratch(*d, scratch);
    if (!L.off_image) return npas_internal_pack_bp(d, w, plan.masks, blob, blob_bytes, stream);
    if (bp_expand_launch(*d, L, w, plan.masks, &plan, static_cast<uint8_t *>(blob), (uint32_t)blob_bytes, static_cast<cudaStream_t>(stream)) != cudaSuccess) return NPAS_ERR_CUDA;
    count_launch();
    return launch_status();
}

npas_status npas_pack_bp(const npas_bp_desc *d, const void *w, const uint64_t *tap_mask, void *blob,
                         size_t blob_bytes, void *stream)
{
    npas_status s = npas_internal_pack_bp(d, w, tap_mask, blob, blob_bytes, stream);
    return s == NPAS_OK ? packed_fits(blob, BP_MAGIC, kMagicBP, static_cast<cudaStream_t>(stream)) : s;
}

npas_status npas_unpack_bp(const npas_bp_desc *d, const void *blob, size_t blob_bytes, void *w_out,
                           uint64_t *tap_mask_out, void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!blob) return NPAS_ERR_NULL;
    if (!aligned16(blob) || (w_out && !aligned16(w_out))) return NPAS_ERR_ALIGNMENT;
    if (blob_bytes < bp_layout(*d, 0).total) return NPAS_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t nW = (size_t)d->K * d->R * d->S * d->C;
    if (w_out && cudaMemsetAsync(w_out, 0, nW * dtype_size(d->w_packed), st) != cudaSuccess) return NPAS_ERR_CUDA;
    const uint32_t nBlk = (d->K / d->Mb) * (d->C / d->Nb);
    const uint8_t *b8 = static_cast<const uint8_t *>(blob);
    if (d->w_packed == NPAS_F32)
        bp_scatter_kernel<uint32_t><<<nBlk, 128, 0, st>>>(*d, b8, static_cast<uint32_t *>(w_out), tap_mask_out);
    else
        bp_scatter_kernel<uint16_t><<<nBlk, 128, 0, st>>>(*d, b8, static_cast<uint16_t *>(w_out), tap_mask_out);
    count_launch();
    return launch_status();
}

npas_status npas_mask_bp_from_dense(const npas_bp_desc *d, const uint8_t *m, uint64_t *tap_mask,
                                    int32_t *violations, void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!m || !tap_mask || !violations) return NPAS_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(violations, 0, 4, st) != cudaSuccess) return NPAS_ERR_CUDA;
    bp_mask_from_dense_kernel<<<(d->K / d->Mb) * (d->C / d->Nb), 128, 0, st>>>(*d, m, tap_mask, violations);
    count_launch();
    int32_t v = 0;
    if (cudaMemcpyAsync(&v, violations, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    return v ? NPAS_ERR_MASK_STRUCTURE : NPAS_OK;
}

npas_status npas_internal_bb_size(const npas_bb_desc *d, uint64_t n_vals, uint32_t max_cols, size_t *blob_bytes)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    const BbLayout L = bb_layout(*d);
    const uint32_t Kp = round_up(max_cols, 16u) < 16u ? 16u : round_up(max_cols, 16u);
    if (n_vals * 4 > 0x3FFFFFFFull || (uint64_t)L.nBlk * Kp * d->Bo * L.es > 0x3FFFFFFFull) return NPAS_ERR_SHAPE;
    *blob_bytes = bb_tail(*d, L, (uint32_t)n_vals, max_cols).total;
    return NPAS_OK;
}

npas_status npas_pack_bb_size(const npas_bb_desc *d, const uint64_t *rk, const uint64_t *ck, size_t *blob_bytes)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!rk || !ck || !blob_bytes) return NPAS_ERR_NULL;
    const uint64_t rlive = d->Bo == 64 ? ~0ull : ((1ull << d->Bo) - 1), clive = d->Bi == 64 ? ~0ull : ((1ull << d->Bi) - 1);
    const uint32_t nBlk = (uint32_t)(d->O / d->Bo) * (uint32_t)(d->I / d->Bi);
    uint64_t n = 0;
    uint32_t mx = 0;
    for (uint32_t i = 0; i < nBlk; ++i) {
        const uint32_t nc = (uint32_t)__builtin_popcountll(ck[i] & clive);
        n += round_up((uint32_t)__builtin_popcountll(rk[i] & rlive) * nc, 8u);
        mx = mx > nc ? mx : nc;
    }
    return npas_internal_bb_size(d, n, mx, blob_bytes);
}

// The section writers of a block-based blob.  voff_plan: value offsets that npas_internal_plan_bb left (then T is whole), or null
static cudaError_t bb_gather_launch(const npas_bb_desc &d, const BbLayout &L, const void *w, const uint64_t *rk, const uint64_t *ck, const uint32_t *voff_plan,
                                    const BbTail &T, uint8_t *blob, uint32_t blob_bytes, cudaStream_t st)
{
    auto go = [&](auto out, auto *wp) {
        using TIn = std::remove_const_t<std::remove_pointer_t<decltype(wp)>>;
        using TOut = decltype(out);
        if (voff_plan)
            return tc::launch_pdl({}, bb_gather_kernel<TIn, TOut, true>, dim3(L.nBlk + 1), dim3(256), 0, st, d, wp, rk, ck, voff_plan, blob, blob_bytes, L, T);
        return tc::launch_pdl({}, bb_gather_kernel<TIn, TOut, false>, dim3(L.nBlk), dim3(256), 0, st, d, wp, rk, ck, voff_plan, blob, blob_bytes, L, T);
    };
    if (d.w_packed == NPAS_F32) return go(uint32_t{}, static_cast<const uint32_t *>(w));
    return d.w_in == NPAS_F32 ? go(uint16_t{}, static_cast<const uint32_t *>(w)) : go(uint16_t{}, static_cast<const uint16_t *>(w));
}

npas_status npas_internal_pack_bb(const npas_bb_desc *d, const void *w, const uint64_t *rk, const uint64_t *ck,
                                  void *blob, size_t blob_bytes, void *stream)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!w || !rk || !ck || !blob) return NPAS_ERR_NULL;
    if (!aligned16(w) || !aligned16(blob)) return NPAS_ERR_ALIGNMENT;
    const BbLayout L = bb_layout(*d);
    if (blob_bytes < L.off_values || blob_bytes > 0xFFFFFFFFull) return NPAS_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t *b8 = static_cast<uint8_t *>(blob);
    bb_scan_kernel<<<1, 1024, 0, st>>>(*d, rk, ck, b8, (uint32_t)blob_bytes, L);
    const cudaError_t e = bb_gather_launch(*d, L, w, rk, ck, nullptr, BbTail{}, b8, (uint32_t)blob_bytes, st);
    count_launch(2);
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status npas_internal_plan_bb_bytes(const npas_bb_desc *d, size_t *bytes)
{
    npas_status s = check_bb_desc(d);
    if (s == NPAS_OK) *bytes = bb_scratch(bb_layout(*d), nullptr).bytes;
    return s;
}

npas_status npas_internal_plan_bb(const npas_bb_desc *d, const uint64_t *rows, const uint64_t *cols, void *scratch, uint64_t *host, void *stream)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!rows || !cols || !scratch || !host) return NPAS_ERR_NULL;
    if (!aligned16(scratch) || (reinterpret_cast<uintptr_t>(rows) & 7) || (reinterpret_cast<uintptr_t>(cols) & 7)) return NPAS_ERR_ALIGNMENT;
    void *mapped = nullptr;
    if (cudaHostGetDevicePointer(&mapped, host, 0) != cudaSuccess) return NPAS_ERR_CUDA;
    const BbLayout L = bb_layout(*d);
    const cudaError_t e = tc::launch_pdl({}, bb_plan_kernel, dim3(1), dim3(1024), 0, static_cast<cudaStream_t>(stream), *d, L.nBlk, rows, cols, bb_scratch(L, scratch),
                                         static_cast<unsigned long long *>(mapped));
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status npas_internal_pack_bb_planned(const npas_bb_desc *d, const void *w, void *scratch, uint64_t n_vals, uint32_t max_cols, void *blob,
                                          size_t blob_bytes, void *stream)
{
    size_t need = 0;
    npas_status s = npas_internal_bb_size(d, n_vals, max_cols, &need);
    if (s != NPAS_OK) return s;
    if (!w || !scratch || !blob) return NPAS_ERR_NULL;
    if (!aligned16(w) || !aligned16(blob) || !aligned16(scratch)) return NPAS_ERR_ALIGNMENT;
    if (blob_bytes < need || blob_bytes > 0xFFFFFFFFull) return NPAS_ERR_BUFFER_TOO_SMALL;
    const BbLayout L = bb_layout(*d);
    const BbScratch plan = bb_scratch(L, scratch);
    const cudaError_t e = bb_gather_launch(*d, L, w, plan.rows, plan.cols, plan.voff, bb_tail(*d, L, (uint32_t)n_vals, max_cols), static_cast<uint8_t *>(blob),
                                           (uint32_t)blob_bytes, static_cast<cudaStream_t>(stream));
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status npas_pack_bb(const npas_bb_desc *d, const void *w, const uint64_t *rk, const uint64_t *ck,
                         void *blob, size_t blob_bytes, void *stream)
{
    npas_status s = npas_internal_pack_bb(d, w, rk, ck, blob, blob_bytes, stream);
    return s == NPAS_OK ? packed_fits(blob, BB_MAGIC, kMagicBB, static_cast<cudaStream_t>(stream)) : s;
}

npas_status npas_unpack_bb(const npas_bb_desc *d, const void *blob, size_t blob_bytes, void *w_out,
                           uint64_t *rk_out, uint64_t *ck_out, void *stream)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!blob) return NPAS_ERR_NULL;
    if (!aligned16(blob) || (w_out && !aligned16(w_out))) return NPAS_ERR_ALIGNMENT;
    const BbLayout L = bb_layout(*d);
    if (blob_bytes < L.off_values) return NPAS_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const uint8_t *b8 = static_cast<const uint8_t *>(blob);
    const cudaError_t e = d->w_packed == NPAS_F32
        ? tc::launch_pdl({}, bb_scatter_kernel<uint32_t>, dim3(L.nBlk), dim3(256), 0, st, *d, b8, static_cast<uint32_t *>(w_out), rk_out, ck_out, L)
        : tc::launch_pdl({}, bb_scatter_kernel<uint16_t>, dim3(L.nBlk), dim3(256), 0, st, *d, b8, static_cast<uint16_t *>(w_out), rk_out, ck_out, L);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status npas_mask_bb_from_dense(const npas_bb_desc *d, const uint8_t *m, uint64_t *rk, uint64_t *ck,
                                    int32_t *violations, void *stream)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!m || !rk || !ck || !violations) return NPAS_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(violations, 0, 4, st) != cudaSuccess) return NPAS_ERR_CUDA;
    const BbLayout L = bb_layout(*d);
    bb_mask_from_dense_kernel<<<L.nBlk, 64, 0, st>>>(*d, m, rk, ck, violations, L.nBi);
    count_launch();
    int32_t v = 0;
    if (cudaMemcpyAsync(&v, violations, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    return v ? NPAS_ERR_MASK_STRUCTURE : NPAS_OK;
}

}  // extern "C"
