// Two block-based GEMMs behind one another in one kernel: Y1 = f1(X W1' + b1 + R), Y2 = f2(Y1 W2' + b2), both results written.
// (The last layer of a bottleneck with its shortcut, and the first one of the next.)
//
// By itself the second layer reads Y1, four times as wide as everything else in the block, back from memory: 103 MB of the
// 360 that the two move for 64 images of 56x56.  Here a CTA owns 128 rows and takes Y1 in slabs of 64 columns: a slab's
// residual lands in a slot of shared memory, the epilogue of the first product adds to it and rounds in place, and the same
// slot is what the TMA stores as Y1 and what the tensor core reads as the A operand of the second product, which
// accumulates in tensor memory over the slabs.  Nothing else differs from the two kernels one after the other: the masked
// dense images of both blobs as W1 and W2, fp32 sums in the same order of columns, one rounding per result.
//
// Roles: warp 0 X tiles and weights (a stage: 64 rows of W1 and 64 columns of W2; where all stages of a tile fit they
// are loaded once and stay), warp 1 MMAs (the first product of a slab is issued ahead of the second product of the slab
// before it, whose epilogue runs meanwhile), two groups of eight epilogue warps that take slabs in turn (a slab is a chain of
// waits and conversions of 0.4 us, twice what its MMAs take), one warp for the residual, one for the stores.  Slots are taken in
// the order of the slabs of Y1 and Y2 of a tile.  (Asking L2 for residual slabs ahead of their slots made it slower: 47 -> 60 us.)
//
// What bounds it: for 64 images of 56x56 mostly bytes (262 MB at least, 40 us at the copy rate; 49.3 in calls by themselves, the two
// launches 58.5), the rest being the chain of waits of a slab; for few images the chain of both products.
#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

using namespace tc;

namespace {

constexpr int kEpiWarps = 16, kGroupWarps = 8;
constexpr int kFirstEpiWarp = 2;
constexpr int kResWarp = kFirstEpiWarp + kEpiWarps;         // requests the residual slabs, hands out slots
constexpr int kStoreWarp = kResWarp + 1;                    // stores the finished slabs
constexpr int kThreads = (kStoreWarp + 1) * 32;
constexpr int kRows = 128;
constexpr int kMaxStages = 8;
constexpr int kMaxSlots = 8;
constexpr uint32_t kSlabBytes = kRows * 128;              // 128 rows x 64 bf16, 128-byte swizzled
constexpr uint32_t kSmemLimit = 232448;
constexpr uint32_t kDescHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);
constexpr uint32_t kDescLboOne = 1u << 16;

struct LinTwoParams {
    int M, K1, N1, N2, nK1, nC, n_tiles, S, NS, XB;       // nC: slabs of Y1; S: weight stages; NS: slots; XB: X tiles in shared memory
    int relu1, relu2, early, resident;                    // early: the blobs may be read before the wait (Launch::blob_ready)
    uint32_t stage_bytes, off_w, off_slots, off_bias, off_bar, smem_bytes, tmem_cols;
};

struct LinTwoBars {
    uint64_t x_full[2], x_empty[2];
    uint64_t w_full[kMaxStages], w_empty[kMaxStages];
    uint64_t acc1_full[2], acc1_empty[2], acc2_full, acc2_empty;
    uint64_t slot_ready[kMaxSlots];                       // may be written by the epilogue (a residual slab has landed in it)
    uint64_t slot_done[kMaxSlots];                        // every warp of the slab's group has finished its part
    uint64_t slot_empty[kMaxSlots];                       // its store, and the second product, have read it
    uint32_t tmem_base;
    uint32_t abort_flag;
};

__device__ __forceinline__ uint64_t desc64(uint32_t lo) { return ((uint64_t)kDescHiSw128 << 32) | lo; }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kEpiWarps * 32) : "memory"); }
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *m, const void *src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(src)), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }

// a position in a ring, and the parity of its lap
struct Ring {
    uint32_t i = 0, ph = 0, n;
    __device__ explicit Ring(int size) : n((uint32_t)size) {}
    __device__ void step() { if (++i == n) { i = 0; ph ^= 1u; } }
};

__global__ void __launch_bounds__(kThreads, 1)
linear_bb_two_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w1, const __grid_constant__ CUtensorMap tmap_w2,
                     const __grid_constant__ CUtensorMap tmap_r, const __grid_constant__ CUtensorMap tmap_y1, const __grid_constant__ CUtensorMap tmap_y2,
                     const LinTwoParams p, const float *bias1, const float *bias2, const void *res, uint32_t *ws)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float *bias_s = reinterpret_cast<float *>(smem + p.off_bias);      // [N1 + N2]
    LinTwoBars *bars = reinterpret_cast<LinTwoBars *>(smem + p.off_bar);
    volatile uint32_t *abort_flag = &bars->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t x_tile = (uint32_t)p.nK1 * kSlabBytes;
    const int nS2 = p.N2 / 64;

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&bars->x_full[b], 1); mbar_init(&bars->x_empty[b], 1);
            mbar_init(&bars->acc1_full[b], 1); mbar_init(&bars->acc1_empty[b], kGroupWarps);
        }
        mbar_init(&bars->acc2_full, 1);
        mbar_init(&bars->acc2_empty, kEpiWarps);
        for (int s = 0; s < p.S; ++s) { mbar_init(&bars->w_full[s], 1); mbar_init(&bars->w_empty[s], 1); }
        for (int s = 0; s < p.NS; ++s) {
            mbar_init(&bars->slot_ready[s], 1); mbar_init(&bars->slot_done[s], kGroupWarps); mbar_init(&bars->slot_empty[s], 2);
        }
        bars->abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&tmap_x);
        prefetch_tensormap(&tmap_w1);
        prefetch_tensormap(&tmap_w2);
        prefetch_tensormap(&tmap_y1);
        prefetch_tensormap(&tmap_y2);
        if (res) prefetch_tensormap(&tmap_r);
    }
    if (warp == 1) tmem_alloc(&bars->tmem_base, p.tmem_cols);
    pdl_trigger();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();

    auto load_weights = [&](uint32_t stage, int c) {
        uint8_t *st = smem + p.off_w + (size_t)stage * p.stage_bytes;
        mbar_arrive_expect_tx(&bars->w_full[stage], p.stage_bytes);
        for (int k = 0; k < p.nK1; ++k) tma_load_2d(st + (size_t)k * 8192u, &tmap_w1, &bars->w_full[stage], k * 64, c * 64);
        tma_load_2d(st + (size_t)p.nK1 * 8192u, &tmap_w2, &bars->w_full[stage], c * 64, 0);
    };
    // the weights of the first ring of stages; in a chain of layers before the wait for the kernel before this one
    const int first = min(p.S, p.nC);
    if (tid == 0 && p.early)
        for (int c = 0; c < first; ++c) load_weights((uint32_t)c, c);
    pdl_wait();
    bias1 = behind_wait(bias1); bias2 = behind_wait(bias2);
    if (warp >= kFirstEpiWarp && warp < kResWarp) {
        for (int i = tid - kFirstEpiWarp * 32; i < p.N1 + p.N2; i += kEpiWarps * 32) {
            const float *b = i < p.N1 ? bias1 : bias2;
            bias_s[i] = b ? __ldg(b + (i < p.N1 ? i : i - p.N1)) : 0.f;
        }
        epi_sync();
    }
    const uint32_t tmem_base = bars->tmem_base, acc2 = tmem_base + 128u;

    if (warp == 0) {
        // ---- X tiles and weights ----------------------------------------------------------------------------------
        if (lane == 0) {
            Ring w(p.S), x(p.XB);
            bool ok = true;
            uint32_t stages = 0;                                  // requested so far
            int it = 0;
            for (int tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x, ++it) {
                if (it >= p.XB && !mbar_wait(&bars->x_empty[x.i], x.ph ^ 1u, abort_flag, ws, 0xA100)) break;
                mbar_arrive_expect_tx(&bars->x_full[x.i], x_tile);
                for (int k = 0; k < p.nK1; ++k)                   // (rows past M read as zeros)
                    tma_load_2d(smem + (size_t)x.i * x_tile + (size_t)k * kSlabBytes, &tmap_x, &bars->x_full[x.i], k * 64, tile * kRows);
                x.step();
                for (int c = 0; c < p.nC && !(p.resident && it); ++c, ++stages) {
                    if (stages >= (uint32_t)p.S && !mbar_wait(&bars->w_empty[w.i], w.ph ^ 1u, abort_flag, ws, 0xA110)) { ok = false; break; }
                    if (!p.early || stages >= (uint32_t)first) load_weights(w.i, c);
                    w.step();
                }
            }
        }
    } else if (warp == 1) {
        // ---- MMAs: product one of slab g, then product two of slab g - 1 --------------------------------------------
        if (elect_one()) {
            const uint32_t id1 = idesc_bf16_f32(128, 64), id2 = idesc_bf16_f32(128, (uint32_t)p.N2);
            const uint32_t x16 = (smem_u32(smem) >> 4) | kDescLboOne, w16 = (smem_u32(smem + p.off_w) >> 4) | kDescLboOne,
                           s16 = (smem_u32(smem + p.off_slots) >> 4) | kDescLboOne, w2_off = (uint32_t)p.nK1 * 512u;
            Ring w1(p.S), w2(p.S), x(p.XB), slot(p.NS);
            uint32_t g = 0, tiles2 = 0;                           // slabs of Y1 so far; tiles whose second product has begun
            int c2 = 0, skip = 0;                                 // the slab product two is due for, in its tile
            bool ok = true, due = false;
            auto second = [&]() {
                // (past the slabs of Y2, which have slots of their own; waited for like the others, or the parity of a slot's lap
                // would be that of the lap before the last one)
                for (int i = 0; i < skip; ++i, slot.step())
                    if (!mbar_wait(&bars->slot_done[slot.i], slot.ph, abort_flag, ws, 0xA200)) return false;
                skip = 0;
                if (c2 == 0 && tiles2++ > 0 && !mbar_wait(&bars->acc2_empty, tiles2 & 1u, abort_flag, ws, 0xA205)) return false;
                if (!mbar_wait(&bars->slot_done[slot.i], slot.ph, abort_flag, ws, 0xA210)) return false;
                tc_fence_after_sync();
                const uint32_t a_lo = s16 + slot.i * (kSlabBytes >> 4), b_lo = w16 + w2.i * (p.stage_bytes >> 4) + w2_off;
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j) mma_bf16_ss(acc2, desc64(a_lo + 2 * j), desc64(b_lo + 2 * j), id2, (c2 > 0 || j > 0) ? 1u : 0u);
                if (!p.resident) mma_commit(&bars->w_empty[w2.i]);
                mma_commit(&bars->slot_empty[slot.i]);
                w2.step();
                slot.step();
                if (++c2 == p.nC) {
                    mma_commit(&bars->acc2_full);
                    c2 = 0;
                    skip = nS2;
                }
                return true;
            };
            for (int tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x) {
                if (!mbar_wait(&bars->x_full[x.i], x.ph, abort_flag, ws, 0xA220)) break;
                for (int c = 0; c < p.nC; ++c, ++g) {
                    // (stages that stay are complete for good: the parity of their first and only phase)
                    if (!mbar_wait(&bars->w_full[w1.i], p.resident ? 0u : w1.ph, abort_flag, ws, 0xA230)) { ok = false; break; }
                    if (g >= 2 && !mbar_wait(&bars->acc1_empty[g & 1u], ((g >> 1) & 1u) ^ 1u, abort_flag, ws, 0xA240)) { ok = false; break; }
                    tc_fence_after_sync();
                    uint32_t a_lo = x16 + x.i * (x_tile >> 4), b_lo = w16 + w1.i * (p.stage_bytes >> 4);
                    for (int k = 0; k < p.nK1; ++k, a_lo += kSlabBytes >> 4, b_lo += 512u)
#pragma unroll
                        for (uint32_t j = 0; j < 4; ++j)
                            mma_bf16_ss(tmem_base + (g & 1u) * 64u, desc64(a_lo + 2 * j), desc64(b_lo + 2 * j), id1, (k > 0 || j > 0) ? 1u : 0u);
                    mma_commit(&bars->acc1_full[g & 1u]);
                    if (c == p.nC - 1) mma_commit(&bars->x_empty[x.i]);
                    w1.step();
                    if (due && !second()) { ok = false; break; }
                    due = true;
                }
                x.step();
            }
            if (ok && due) second();
        }
    } else if (warp == kResWarp) {
        // ---- slots: free again, and the residual slab requested into them -------------------------------------------
        if (lane == 0) {
            Ring slot(p.NS);
            uint32_t n = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x)
                for (int c = 0; c < p.nC + nS2; ++c, ++n) {
                    if (n >= (uint32_t)p.NS && !mbar_wait(&bars->slot_empty[slot.i], slot.ph ^ 1u, abort_flag, ws, 0xA500)) { ok = false; break; }
                    if (res && c < p.nC) {
                        mbar_arrive_expect_tx(&bars->slot_ready[slot.i], kSlabBytes);
                        tma_load_2d(smem + p.off_slots + (size_t)slot.i * kSlabBytes, &tmap_r, &bars->slot_ready[slot.i], c * 64, tile * kRows);
                    } else {
                        mbar_arrive(&bars->slot_ready[slot.i]);
                    }
                    slot.step();
                }
        }
    } else if (warp == kStoreWarp) {
        // ---- stores: when the one before has read its slot, that slot is free as far as stores go --------------------
        if (lane == 0) {
            Ring slot(p.NS);
            uint32_t prev = 0;
            bool ok = true, first_store = true, prev_last = false;      // prev_last: no second product reads the slot before
            for (int tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x)
                for (int c = 0; c < p.nC + nS2; ++c) {
                    if (!mbar_wait(&bars->slot_done[slot.i], slot.ph, abort_flag, ws, 0xA600)) { ok = false; break; }
                    const uint8_t *sp = smem + p.off_slots + (size_t)slot.i * kSlabBytes;
                    if (c < p.nC) tma_store_2d(&tmap_y1, sp, c * 64, tile * kRows);
                    else tma_store_2d(&tmap_y2, sp, (c - p.nC) * 64, tile * kRows);
                    bulk_commit();
                    if (!first_store) {
                        bulk_wait_read<1>();
                        mbar_arrive(&bars->slot_empty[prev]);
                        if (prev_last) mbar_arrive(&bars->slot_empty[prev]);
                    }
                    first_store = false; prev = slot.i; prev_last = c >= p.nC;
                    slot.step();
                }
            bulk_wait_read<0>();                                  // the slots stay valid until the last store has read them
        }
    } else {
        // ---- epilogues: warp -> group, TMEM lane quarter (warp % 4) and one half of a slab's columns ----------------------
        const int e = warp - kFirstEpiWarp, group = e >> 3, quarter = warp & 3, half = (e >> 2) & 1, m = quarter * 32 + lane;
        const uint32_t lanes = ((uint32_t)(quarter * 32) << 16) + (uint32_t)half * 32u;
        Ring slot(p.NS);
        uint32_t g = 0, it = 0;
        bool ok = true;
        // 32 sums of this thread's row, + bias (+ residual), one rounding, then ReLU on the packed pairs, into the slot
        auto finish = [&](const uint32_t (&r)[32], const float *bs, bool add, int relu) {
            uint8_t *sp = smem + p.off_slots + (size_t)slot.i * kSlabBytes + (uint32_t)m * 128u;
            if (!mbar_wait(&bars->slot_ready[slot.i], slot.ph, abort_flag, ws, 0xA410)) return false;
            const float4 *b4 = reinterpret_cast<const float4 *>(bs);
#pragma unroll
            for (int q = 0; q < 4; ++q) {                         // a 16-byte piece of the row (pieces XOR-ed with the row number)
                uint4 *piece = reinterpret_cast<uint4 *>(sp + (uint32_t)(((4 * half + q) ^ (m & 7)) * 16));
                const float4 u = b4[2 * q], w = b4[2 * q + 1];
                float v[8] = {__uint_as_float(r[8 * q]) + u.x, __uint_as_float(r[8 * q + 1]) + u.y, __uint_as_float(r[8 * q + 2]) + u.z,
                              __uint_as_float(r[8 * q + 3]) + u.w, __uint_as_float(r[8 * q + 4]) + w.x, __uint_as_float(r[8 * q + 5]) + w.y,
                              __uint_as_float(r[8 * q + 6]) + w.z, __uint_as_float(r[8 * q + 7]) + w.w};
                if (add) {
                    const uint4 a = *piece;
                    const uint32_t wv[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        v[2 * i] += __uint_as_float(wv[i] << 16);
                        v[2 * i + 1] += __uint_as_float(wv[i] & 0xFFFF0000u);
                    }
                }
                uint32_t o[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    o[i] = cvt_bf16x2(v[2 * i], v[2 * i + 1]);
                    if (relu) o[i] = relu_bf16x2(o[i]);
                }
                *piece = make_uint4(o[0], o[1], o[2], o[3]);
            }
            fence_proxy_async_smem();                             // the TMA store and the tensor core read what this thread wrote
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->slot_done[slot.i]);
            return true;
        };
        // the other group's slab: no lap of a slot is left out, or the parity waited for would be that of the lap before the last one
        auto pass = [&]() { return mbar_wait(&bars->slot_ready[slot.i], slot.ph, abort_flag, ws, 0xA415); };
        for (int tile = blockIdx.x; tile < p.n_tiles && ok; tile += gridDim.x, ++it) {
            uint32_t r[32];
            for (int c = 0; c < p.nC; ++c, ++g, slot.step()) {
                if ((int)(g & 1u) != group) {                     // (accumulator and group alternate together)
                    if (!pass()) { ok = false; break; }
                    continue;
                }
                if (!mbar_wait(&bars->acc1_full[group], (g >> 1) & 1u, abort_flag, ws, 0xA400)) { ok = false; break; }
                tc_fence_after_sync();
                tmem_ld_x32(tmem_base + (uint32_t)group * 64u + lanes, r);
                tmem_ld_wait();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc1_empty[group]);
                if (!finish(r, bias_s + c * 64 + half * 32, res != nullptr, p.relu1)) { ok = false; break; }
            }
            if (!ok || !mbar_wait(&bars->acc2_full, it & 1u, abort_flag, ws, 0xA420)) { ok = false; break; }
            tc_fence_after_sync();
            for (int s = 0; s < nS2; ++s, slot.step()) {
                if ((s & 1) != group) {
                    if (!pass()) { ok = false; break; }
                    continue;
                }
                tmem_ld_x32(acc2 + (uint32_t)s * 64u + lanes, r);
                tmem_ld_wait();
                tc_fence_before_sync();
                if (!finish(r, bias_s + p.N1 + s * 64 + half * 32, false, p.relu2)) { ok = false; break; }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->acc2_empty);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        // a role gave up: leave time for copies still in flight to land before the CTA retires
        const long long t0 = clock64();
        while (clock64() - t0 < 400000ll) { }
    }
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, p.tmem_cols);
    }
}

bool plan(const npas_linear_desc &a, const npas_linear_desc &b, LinTwoParams &p)
{
    if (a.M != b.M || a.O != b.I || a.x_dtype != NPAS_BF16 || a.y_dtype != NPAS_BF16 || b.x_dtype != NPAS_BF16 || b.y_dtype != NPAS_BF16) return false;
    if (b.has_residual || a.path || a.variant || b.path || b.variant) return false;
    if (a.I % 64 || a.O % 64 || b.O % 64 || b.O > 256) return false;
    p = {};
    p.M = a.M; p.K1 = a.I; p.N1 = a.O; p.N2 = b.O;
    p.nK1 = a.I / 64; p.nC = a.O / 64;
    p.n_tiles = (a.M + kRows - 1) / kRows;
    p.relu1 = a.relu; p.relu2 = b.relu;
    p.stage_bytes = (uint32_t)p.nK1 * 8192u + (uint32_t)p.N2 * 128u;
    const uint32_t x_tile = (uint32_t)p.nK1 * kSlabBytes, fixed = (uint32_t)(p.N1 + p.N2) * 4u + 128u + (uint32_t)sizeof(LinTwoBars) + 1024u;
    // an X tile, two weight stages and three slots at least; what is left goes to weights that then stay, to a second X tile where
    // tiles are short, to slots, then to stages
    p.XB = 1; p.S = p.nC < 2 ? p.nC : 2; p.NS = 3;
    auto bytes = [&]() { return fixed + p.XB * x_tile + p.S * p.stage_bytes + p.NS * kSlabBytes; };
    if (bytes() > kSmemLimit) return false;
    auto grow = [&](int &v, int most) {
        if (v >= most) return false;
        ++v;
        if (bytes() <= kSmemLimit) return true;
        --v;
        return false;
    };
    p.NS = 5;
    if (p.nC > 2 && p.nC <= kMaxStages) {
        p.S = p.nC;
        if (bytes() > kSmemLimit) p.S = 2;
    }
    if (bytes() > kSmemLimit) p.NS = 3;
    if (p.nC <= 4) grow(p.XB, 2);
    while (grow(p.NS, kMaxSlots)) { }
    while (p.S < p.nC && grow(p.S, kMaxStages)) { }
    p.resident = p.S == p.nC;
    p.off_w = (uint32_t)p.XB * x_tile;
    p.off_slots = p.off_w + (uint32_t)p.S * p.stage_bytes;
    p.off_bias = p.off_slots + (uint32_t)p.NS * kSlabBytes;
    p.off_bar = round_up(p.off_bias + (uint32_t)(p.N1 + p.N2) * 4u, 128);
    p.smem_bytes = p.off_bar + (uint32_t)sizeof(LinTwoBars) + 1024u;
    if (p.smem_bytes > kSmemLimit) return false;
    p.tmem_cols = 128 + p.N2 <= 256 ? 256 : 512;
    return true;
}

bool encode_2d(CUtensorMap *map, const void *base, uint64_t inner, uint64_t outer, uint32_t box_outer)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {inner * 2};
    const cuuint32_t box[2] = {64, box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Two layers in one launch where both layers' weights stay in shared memory beside two X tiles and five slots, whatever the
// rows (64 -> 256 -> 64, us, against the two launches: 784 rows 6.7 and 7.8, 12544 7.6 and 9.1, 200704 49.3 and 58.5).  With weights
// that come through a ring, or too few slots for the residual's latency, it is the slower way (50176x128 -> 512 -> 128 44 and
// 34, 50176x128 -> 256 -> 64 21.2 and 20.0): every CTA reads all weights again for each of its tiles.
bool linear_two_preferred(const npas_linear_desc &a, const npas_linear_desc &b)
{
    LinTwoParams p;
    return plan(a, b, p) && p.resident && p.XB == 2 && p.NS >= 5;
}

npas_status linear_two_launch(const npas_linear_desc &a, const npas_bb_desc &bba, const npas_linear_desc &b, const npas_bb_desc &bbb, const void *x,
                              const void *blob1, const float *bias1, const void *res, void *y1, const void *blob2, const float *bias2, void *y2,
                              uint32_t *ws, cudaStream_t st, Launch how)
{
    LinTwoParams p;
    if (!plan(a, b, p) || bba.w_packed != NPAS_BF16 || bbb.w_packed != NPAS_BF16) return NPAS_ERR_UNSUPPORTED;
    const BbLayout L1 = bb_layout(bba), L2 = bb_layout(bbb);
    CUtensorMap tmx, tw1, tw2, tmr, ty1, ty2;
    if (!encode_2d(&tmx, x, (uint64_t)p.K1, (uint64_t)p.M, kRows) ||
        !encode_2d(&tw1, static_cast<const uint8_t *>(blob1) + L1.off_dense, (uint64_t)p.K1, (uint64_t)p.N1, 64) ||
        !encode_2d(&tw2, static_cast<const uint8_t *>(blob2) + L2.off_dense, (uint64_t)p.N1, (uint64_t)p.N2, (uint32_t)p.N2) ||
        !encode_2d(&ty1, y1, (uint64_t)p.N1, (uint64_t)p.M, kRows) || !encode_2d(&ty2, y2, (uint64_t)p.N2, (uint64_t)p.M, kRows))
        return NPAS_ERR_CUDA;
    tmr = ty1;
    if (res && !encode_2d(&tmr, res, (uint64_t)p.N1, (uint64_t)p.M, kRows)) return NPAS_ERR_CUDA;
    if (allow_dynamic_smem(reinterpret_cast<const void *>(linear_bb_two_kernel), (int)kSmemLimit) != NPAS_OK) return NPAS_ERR_CUDA;
    const int sms = sm_count();
    p.early = how.blob_ready;
    const cudaError_t e = launch_pdl(how, linear_bb_two_kernel, dim3(p.n_tiles < sms ? p.n_tiles : sms), dim3(kThreads), p.smem_bytes, st, tmx, tw1, tw2, tmr,
                                     ty1, ty2, p, bias1, bias2, res, ws);
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // namespace npas
