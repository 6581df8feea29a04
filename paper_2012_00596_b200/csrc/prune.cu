// One-shot magnitude pruning of a layer under the two schemes (paper Sec. 5.2): turns dense
// weights into the block masks the packers take.  The score of a prunable group (a tap of a block;
// a row or a column of a block) is the sum of the squares of its weights, accumulated in fp64 in a
// fixed order (filters / rows outer, channels / columns inner; a square of a float is exact in
// fp64, so fused or separate multiply-add give the same bits); a block keeps its `keep`
// highest-scoring groups, ties go to the lower index.  Offline step: one CTA per block for the per-block counts; for the
// layer-wide budget a thread per group scores and a cluster selects.
#include "common.cuh"
#include "select_range.h"
#include "tc_common.cuh"

namespace npas {

template <typename T> __device__ inline double prune_load(const T *p);
template <> __device__ inline double prune_load<float>(const float *p) { return (double)*p; }
template <> __device__ inline double prune_load<uint16_t>(const uint16_t *p) { return (double)bf16_bits_to_f32(*p); }

// V consecutive weights (V = 1, 4, or 8 bf16), as they lie in memory
template <typename T, int V> struct PruneVec { uint32_t u[(V * sizeof(T) + 3) / 4]; };
template <typename T, int V> __device__ __forceinline__ PruneVec<T, V> prune_load_vec(const T *p)
{
    PruneVec<T, V> r;
    if constexpr (V * sizeof(T) == 16) { const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p)); r.u[0] = q.x; r.u[1] = q.y; r.u[2] = q.z; r.u[3] = q.w; }
    else if constexpr (V * sizeof(T) == 8) { const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p)); r.u[0] = q.x; r.u[1] = q.y; }
    else if constexpr (sizeof(T) == 4) r.u[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
    else r.u[0] = __ldg(p);
    return r;
}
template <typename T, int V> __device__ __forceinline__ double prune_at(const PruneVec<T, V> &r, int q)
{
    if constexpr (sizeof(T) == 4) return (double)__uint_as_float(r.u[q]);
    else return (double)__uint_as_float(q & 1 ? r.u[q / 2] & 0xFFFF0000u : r.u[q / 2] << 16);
}

// the `keep` largest of n <= 64 scores as a bitset; ties to the lower index
__device__ inline uint64_t top_k_bits(const double *score, int n, int keep)
{
    uint64_t bits = 0;
    for (int k = 0; k < keep; ++k) {
        int best = -1;
        for (int t = 0; t < n; ++t)
            if (!((bits >> t) & 1ull) && (best < 0 || score[t] > score[best])) best = t;
        bits |= 1ull << best;
    }
    return bits;
}

template <typename T>
__global__ void prune_bp_kernel(npas_bp_desc d, const T *__restrict__ w, int keep, uint64_t *tap_mask)
{
    __shared__ double score[64];
    const int RS = d.R * d.S, nCB = d.C / d.Nb, b = blockIdx.x, fb = b / nCB, cb = b - fb * nCB;
    const int t = threadIdx.x;
    if (t < RS) {
        double s = 0.0;
        for (int f = 0; f < d.Mb; ++f)
            for (int c = 0; c < d.Nb; ++c) {
                const double v = prune_load(w + ((size_t)(fb * d.Mb + f) * RS + t) * d.C + cb * d.Nb + c);
                s = fma(v, v, s);
            }
        score[t] = s;
    }
    __syncthreads();
    if (t == 0) tap_mask[b] = top_k_bits(score, RS, keep);
}

// One CTA per block: the block is staged once (coalesced), 64 threads score the rows and 64 the columns, each in the
// stated order, and every thread finds the rank of its own score; the kept ones are the set bits of two ballots.  (One
// thread picking the largest score `keep` times took 80 us on 2048x512 with 32x32 of 64x64 kept.)
template <typename T>
__global__ void __launch_bounds__(128)
prune_bb_kernel(npas_bb_desc d, const T *__restrict__ w, int keep_rows, int keep_cols,
                uint64_t *row_keep, uint64_t *col_keep)
{
    __shared__ float blk_s[64][65];
    __shared__ unsigned long long key_s[2][64];
    __shared__ unsigned int half_s[4];
    const int nBi = d.I / d.Bi, b = blockIdx.x, bo = b / nBi, bi = b - bo * nBi, t = threadIdx.x;
    const bool c1 = (t & 31) < d.Bi, c2 = (t & 31) + 32 < d.Bi;
    tc::pdl_wait();
    w = tc::behind_wait(w);
    const T *blk = w + (size_t)bo * d.Bo * d.I + (size_t)bi * d.Bi;
    float v[16][2];                                              // (the whole block on its way at once)
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int r = (t >> 5) + 4 * j;
        const T *p = blk + (size_t)r * d.I + (t & 31);
        v[j][0] = r < d.Bo && c1 ? (float)prune_load(p) : 0.f;
        v[j][1] = r < d.Bo && c2 ? (float)prune_load(p + 32) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) blk_s[(t >> 5) + 4 * j][(t & 31) + 32 * h] = v[j][h];
    __syncthreads();
    const int side = t >> 6, i = t & 63, n = side ? d.Bi : d.Bo, len = side ? d.Bo : d.Bi, keep = side ? keep_cols : keep_rows;
    unsigned long long key = 0;
    if (i < n) {
        double s = 0.0;
        const float *p = side ? &blk_s[0][i] : &blk_s[i][0];
        const int step = side ? 65 : 1;
#pragma unroll 16
        for (int j = 0; j < len; ++j) { const double v = (double)p[j * step]; s = fma(v, v, s); }
        key = (unsigned long long)__double_as_longlong(s);         // sums of squares order like their bit patterns
    }
    key_s[side][i] = key;
    __syncthreads();
    int rank = 0;
#pragma unroll 16
    for (int j = 0; j < n; ++j) rank += key_s[side][j] > key || (key_s[side][j] == key && j < i);
    const unsigned int kept = __ballot_sync(0xFFFFFFFFu, i < n && rank < keep);
    if ((t & 31) == 0) half_s[t >> 5] = kept;
    __syncthreads();
    if (i == 0) (side ? col_keep : row_keep)[b] = (uint64_t)half_s[2 * side] | ((uint64_t)half_s[2 * side + 1] << 32);
}

// ---- layer-wide budget -------------------------------------------------------------------------
// Scores of all (block, tap) groups, in group order (block major, tap minor), as fp64.  A thread per group, channel
// blocks fastest: neighbouring threads read neighbouring runs of Nb channels of the same filter and tap, V of them at a
// time.  The sums are ordered, so what counts is that loads do not wait for them: thirty-two vectors are on their way, and the
// next sixteen are requested before sixteen are added.  512x3x3x512 in 16x8 blocks fp32 (9.4 MB, 144 CTAs of four warps,
// nothing in L2): 6.6 us, 7.7 with sixteen on their way and eight at a time, 15 with one run after the other.
template <typename T, int V>
__global__ void __launch_bounds__(128)
prune_bp_scores_kernel(npas_bp_desc d, const T *__restrict__ w, double *scores)
{
    constexpr int kBatch = 16;
    tc::pdl_trigger();
    tc::pdl_wait();
    w = tc::behind_wait(w);
    const int RS = d.R * d.S, nCB = d.C / d.Nb;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, total = (long long)(d.K / d.Mb) * RS * nCB;
    if (i >= total) return;
    const int cb = (int)(i % nCB), rest = (int)(i / nCB), t = rest % RS, fb = rest / RS;
    const T *p = w + ((size_t)fb * d.Mb * RS + t) * d.C + (size_t)cb * d.Nb;      // the next vector to request
    const size_t step = (size_t)RS * d.C - d.Nb;                                   // from the end of a run to the next filter's
    const int vecs = d.Mb * (d.Nb / V), per_run = d.Nb / V;
    int asked = 0, in_run = 0;
    auto request = [&](PruneVec<T, V> (&v)[kBatch]) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
            if (asked < vecs) {
                v[j] = prune_load_vec<T, V>(p);
                ++asked;
                p += V;
                if (++in_run == per_run) { in_run = 0; p += step; }
            }
    };
    double s = 0.0;
    auto add = [&](const PruneVec<T, V> (&v)[kBatch], int first) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
            if (first + j < vecs) {
#pragma unroll
                for (int q = 0; q < V; ++q) { const double x = prune_at<T, V>(v[j], q); s = fma(x, x, s); }
            }
    };
    PruneVec<T, V> a[kBatch], b[kBatch];
    request(a);
    for (int done = 0; done < vecs; done += 2 * kBatch) {
        request(b);
        add(a, done);
        request(a);
        add(b, done + kBatch);
    }
    scores[((size_t)fb * nCB + cb) * RS + t] = s;
}

// Keeps the n_keep largest of G scores, ties to the lower index, and writes the tap sets.  One cluster; every CTA holds
// the keys of a range of whole blocks (in shared memory when they fit).  A sum of squares is never negative, so the order
// of the fp64 values is that of their bit patterns as unsigned integers.
//
// What bounds it is the number of steps that the whole cluster waits for (a cluster barrier and a round trip to the other
// CTAs' shared memory, about 1.2 us together) and of round trips to shared memory behind one another.  So one pass counts the
// keys in 1024 bins between the smallest and the largest of 256 sampled keys (every CTA samples the same ones; the outer bins
// take what lies beyond, so any sample is right and a bad one only costs another pass), every CTA adds the CTAs' counts and
// walks the bins downwards to the one in which the remaining budget falls; once that holds few enough keys, every CTA sends
// its own ones to all others, and after one more barrier each ranks its own among all of them, by score and index.  18432
// scores end after one pass with about 60 keys to rank (256 bins left 430, whose ranking took as long as all the rest); a bin that
// holds more than kSelRank keys is divided again, and only when it is a single value that so many keys share are they taken in
// index order.  18432 groups: 8.4 us; 11.0 with the bits in which keys differ found first
// and eight of them decided per pass, until a digit held exactly the budget (five or six cluster barriers, here two).
constexpr int kSelThreads = 256;
constexpr uint32_t kSelSmemKeys = 24576;                        // 192 KB of keys per CTA
constexpr uint32_t kSelRank = 512;                              // keys that are ranked directly
static_assert(kSelBins == 4 * kSelThreads, "four neighbouring bins per thread");
constexpr int kSelBatch = 10;                                   // keys of a thread whose loads are in flight together

struct SelShared {
    alignas(16) unsigned int hist[2][kSelBins];
    unsigned long long warp_lo[kSelThreads / 32], warp_hi[kSelThreads / 32];
    unsigned long long rank_key[kSelRank];
    unsigned int rank_at[kSelRank];
    unsigned int warp_sums[kSelThreads / 32];
    unsigned int pick_bin, pick_above, pick_have, pick_before, mine;
};

__device__ __forceinline__ unsigned int sel_rank() { unsigned int r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void sel_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void sel_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void sel_cluster_sync() { sel_cluster_arrive(); sel_cluster_wait(); }
__device__ __forceinline__ unsigned int sel_peer(const void *p, unsigned int rank)
{
    unsigned int q;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(q) : "r"((unsigned int)__cvta_generic_to_shared(p)), "r"(rank));
    return q;
}
__device__ __forceinline__ uint4 sel_remote(const void *p, unsigned int rank)
{
    uint4 v;
    asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(sel_peer(p, rank)) : "memory");
    return v;
}

__global__ void __launch_bounds__(kSelThreads)
prune_select_kernel(const unsigned long long *__restrict__ keys, long long n_keep, int RS, unsigned long long *tap_mask,
                    long long n_blocks, int n_ctas, int in_smem)
{
    extern __shared__ unsigned long long key_smem[];
    __shared__ SelShared sh;
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const unsigned int rank = sel_rank();
    const long long per = (n_blocks + n_ctas - 1) / n_ctas, b_lo = min(n_blocks, rank * per), b_hi = min(n_blocks, b_lo + per);
    const long long n = (b_hi - b_lo) * RS, total = n_blocks * RS;
    const unsigned int first = (unsigned int)(b_lo * RS);
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    for (int i = 0; i < 2; ++i) *reinterpret_cast<uint4 *>(&sh.hist[i][4 * t]) = zero4;
    if (t == 0) sh.mine = 0;
    tc::pdl_wait();                    // (started while the scores are being computed)
    keys = tc::behind_wait(keys);
    const unsigned long long *src = keys + b_lo * RS;
    // f(key, index) for this CTA's keys, a batch of loads at a time
    auto each = [&](auto f) {
        for (long long i0 = t; i0 < n; i0 += kSelThreads * kSelBatch) {
            unsigned long long k[kSelBatch];
#pragma unroll
            for (int j = 0; j < kSelBatch; ++j) k[j] = i0 + j * kSelThreads < n ? src[i0 + j * kSelThreads] : 0;
#pragma unroll
            for (int j = 0; j < kSelBatch; ++j)
                if (i0 + j * kSelThreads < n) f(k[j], i0 + j * kSelThreads);
        }
    };
    const unsigned long long sample = keys[t * total / kSelThreads];
    if (in_smem) {
        each([&](unsigned long long k, long long i) { key_smem[i] = k; });
        src = key_smem;
    }
    unsigned long long base = sample, top = sample;
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        base = min(base, __shfl_xor_sync(0xFFFFFFFFu, base, d));
        top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, d));
    }
    if (lane == 0) { sh.warp_lo[wid] = base; sh.warp_hi[wid] = top; }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSelThreads / 32; ++i) { base = min(base, sh.warp_lo[i]); top = max(top, sh.warp_hi[i]); }
    int shift = sel_first_shift(base, top);

    // the budget left, `need`, falls among the `have` keys in [lo, hi], of which CTAs of lower rank hold `before`
    // (how many passes that takes at most is a property of the ranges alone, select_range.h; were a budget to fall among no keys, which
    // takes scores that change under the kernel, the search would end there)
    uint64_t lo = 0, hi = ~0ull;
    unsigned int need = (unsigned int)n_keep, have = (unsigned int)total, before = first;
    for (int pass = 0; pass < kSelPasses && need != have && have > kSelRank && lo != hi; ++pass) {
        unsigned int *hist = sh.hist[pass & 1];
        if (pass == 0)
            each([&](unsigned long long k, long long) { atomicAdd(&hist[sel_first_bin(k, base, shift)], 1u); });
        else {
            shift = sel_shift(hi - lo);
            each([&](unsigned long long k, long long) { if (k >= lo && k <= hi) atomicAdd(&hist[sel_bin(k, lo, shift)], 1u); });
        }
        sel_cluster_sync();
        {
            // (a thread per four bins) counts of all CTAs, then how many keys lie in these bins or higher ones (warp scans from the top, then over the warps)
            uint4 c = zero4, lower = zero4;
            const int bin0 = kSelBins - 4 - 4 * t;
#pragma unroll
            for (unsigned int r = 0; r < 8; ++r)
                if (r < (unsigned int)n_ctas) {
                    const uint4 v = sel_remote(&hist[bin0], r);
                    if (r == rank) lower = c;
                    c.x += v.x; c.y += v.y; c.z += v.z; c.w += v.w;
                }
            const unsigned int sum = c.x + c.y + c.z + c.w;
            unsigned int up = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, up, d); if (lane >= d) up += v; }
            if (lane == 31) sh.warp_sums[wid] = up;
            if (t == 0) sh.pick_have = 0;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSelThreads / 32; ++i) up += i < wid ? sh.warp_sums[i] : 0u;
            const unsigned int cs[4] = {c.x, c.y, c.z, c.w}, ls[4] = {lower.x, lower.y, lower.z, lower.w};
            unsigned int above = up - sum;                         // keys in higher bins than the one looked at
#pragma unroll
            for (int j = 3; j >= 0; --j) {
                if (above < need && above + cs[j] >= need) { sh.pick_bin = (unsigned int)(bin0 + j); sh.pick_above = above; sh.pick_have = cs[j]; sh.pick_before = ls[j]; }
                above += cs[j];
            }
            *reinterpret_cast<uint4 *>(&sh.hist[(pass + 1) & 1][4 * t]) = zero4;      // (every CTA has read the counts of the pass before)
        }
        __syncthreads();
        have = sh.pick_have;
        if (have == 0) { need = 0; break; }               // (every CTA has the same counts)
        need -= sh.pick_above;
        before = sh.pick_before;
        if (pass == 0) sel_first_range(sh.pick_bin, base, shift, lo, hi);
        else sel_range(sh.pick_bin, shift, lo, hi);
        __syncthreads();
    }
    const bool all = need == have, ranked = !all && have <= kSelRank;
    if (ranked) {
        // this CTA's keys of the range, to every CTA (listed first: a store per thread and CTA then, not one after another)
        each([&](unsigned long long k, long long i) {
            if (k < lo || k > hi) return;
            const unsigned int at = before + atomicAdd(&sh.mine, 1u);
            sh.rank_key[at] = k; sh.rank_at[at] = first + (unsigned int)i;
        });
        __syncthreads();
        for (unsigned int e = t; e < sh.mine * 8; e += kSelThreads) {
            const unsigned int at = before + e / 8, r = e & 7;
            if (r >= (unsigned int)n_ctas || r == rank) continue;
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(sel_peer(&sh.rank_key[at], r)), "l"(sh.rank_key[at]) : "memory");
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(sel_peer(&sh.rank_at[at], r)), "r"(sh.rank_at[at]) : "memory");
        }
    }
    sel_cluster_arrive();              // (the sets without the range, meanwhile)
    const long long nb = b_hi - b_lo;
    if (all || ranked) {
        for (long long b = t; b < nb; b += kSelThreads) {
            unsigned long long m = 0;
            for (int i0 = 0; i0 < RS; i0 += 9) {
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    const unsigned long long k = i0 + j < RS ? src[b * RS + i0 + j] : 0;
                    m |= (unsigned long long)(i0 + j < RS && (k > hi || (all && k >= lo))) << ((i0 + j) & 63);
                }
            }
            tap_mask[b_lo + b] = m;
        }
    }
    sel_cluster_wait();                // (from here on no CTA reads or writes another one's memory, but for equal keys)
    if (ranked) {
        // a warp per key of this CTA: how many of all the range's keys come before it
        __syncthreads();               // (the sets are stored, which the cluster barrier, arrived at before, does not say)
        for (unsigned int c = before + wid; c < before + sh.mine; c += kSelThreads / 32) {
            const unsigned long long k = sh.rank_key[c];
            const unsigned int at = sh.rank_at[c];
            unsigned int ahead = 0;
            for (unsigned int j0 = lane; j0 < have; j0 += 128) {
#pragma unroll
                for (unsigned int j = j0; j < j0 + 128; j += 32) {
                    const unsigned long long o = j < have ? sh.rank_key[j] : 0ull;
                    const unsigned int o_at = j < have ? sh.rank_at[j] : ~0u;          // (nothing comes behind every key)
                    ahead += (unsigned int)(o > k) | ((unsigned int)(o == k) & (unsigned int)(o_at < at));
                }
            }
            ahead = __reduce_add_sync(0xFFFFFFFFu, ahead);
            if (lane == 0 && ahead < need) atomicOr(tap_mask + at / (unsigned int)RS, 1ull << at % (unsigned int)RS);
        }
    } else if (!all) {
        // equal keys: keys above them, and the first `need` of them in index order
        const long long chunk = (nb + kSelThreads - 1) / kSelThreads, t_lo = min(nb, t * chunk), t_hi = min(nb, t_lo + chunk);
        unsigned int up = 0;
        for (long long i = t_lo * RS; i < t_hi * RS; ++i) up += src[i] == lo;
        const unsigned int mine = up;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, up, d); if (lane >= d) up += v; }
        if (lane == 31) sh.warp_sums[wid] = up;
        __syncthreads();
        for (int i = 0; i < wid; ++i) up += sh.warp_sums[i];
        unsigned int ahead = before + up - mine;
        for (long long b = t_lo; b < t_hi; ++b) {
            unsigned long long m = 0;
            for (int i = 0; i < RS; ++i) {
                const unsigned long long k = src[b * RS + i];
                m |= (unsigned long long)(k > lo || (k == lo && ahead < need)) << i;
                ahead += k == lo;
            }
            tap_mask[b_lo + b] = m;
        }
    }
}

extern "C" {

npas_status npas_prune_bp_magnitude(const npas_bp_desc *d, const void *w, int32_t keep_taps, uint64_t *tap_mask,
                                    void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!w || !tap_mask) return NPAS_ERR_NULL;
    if (keep_taps < 0 || keep_taps > d->R * d->S) return NPAS_ERR_SHAPE;
    if (!aligned16(w) || (reinterpret_cast<uintptr_t>(tap_mask) & 7)) return NPAS_ERR_ALIGNMENT;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nBlk = (d->K / d->Mb) * (d->C / d->Nb);
    if (d->w_in == NPAS_F32) prune_bp_kernel<float><<<nBlk, 64, 0, st>>>(*d, static_cast<const float *>(w), keep_taps, tap_mask);
    else prune_bp_kernel<uint16_t><<<nBlk, 64, 0, st>>>(*d, static_cast<const uint16_t *>(w), keep_taps, tap_mask);
    count_launch();
    return launch_status();
}

npas_status npas_prune_bp_global_workspace(const npas_bp_desc *d, size_t *ws_bytes)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!ws_bytes) return NPAS_ERR_NULL;
    *ws_bytes = round_up((uint32_t)((d->K / d->Mb) * (d->C / d->Nb) * d->R * d->S) * 8u, 256);
    return NPAS_OK;
}

npas_status npas_prune_bp_magnitude_global(const npas_bp_desc *d, const void *w, int64_t n_keep, uint64_t *tap_mask,
                                           void *ws, size_t ws_bytes, void *stream)
{
    npas_status s = check_bp_desc(d);
    if (s != NPAS_OK) return s;
    if (!w || !tap_mask || !ws) return NPAS_ERR_NULL;
    const long long nBlk = (long long)(d->K / d->Mb) * (d->C / d->Nb), G = nBlk * d->R * d->S;
    if (n_keep < 0 || n_keep > G) return NPAS_ERR_SHAPE;
    if (!aligned16(w) || !aligned16(ws) || (reinterpret_cast<uintptr_t>(tap_mask) & 7)) return NPAS_ERR_ALIGNMENT;
    size_t need = 0;
    npas_prune_bp_global_workspace(d, &need);
    if (ws_bytes < need) return NPAS_ERR_BUFFER_TOO_SMALL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double *scores = static_cast<double *>(ws);
    unsigned long long *masks = reinterpret_cast<unsigned long long *>(tap_mask);
    if (n_keep == 0) return cudaMemsetAsync(masks, 0, (size_t)nBlk * 8, st) == cudaSuccess ? NPAS_OK : NPAS_ERR_CUDA;
    unsigned threads = 128;                                      // (few groups: small CTAs, on more SMs)
    while (threads > 32 && G <= (long long)threads * sm_count() / 2) threads /= 2;
    const unsigned grid = (unsigned)((G + threads - 1) / threads);
    const float *wf = static_cast<const float *>(w);
    const uint16_t *wh = static_cast<const uint16_t *>(w);
    auto go = [&](auto kernel, auto *wp) { return tc::launch_pdl({}, kernel, dim3(grid), dim3(threads), 0, st, *d, wp, scores); };
    cudaError_t e;
    if (d->w_in == NPAS_F32) e = d->Nb % 4 == 0 ? go(prune_bp_scores_kernel<float, 4>, wf) : go(prune_bp_scores_kernel<float, 1>, wf);
    else e = d->Nb % 8 == 0 ? go(prune_bp_scores_kernel<uint16_t, 8>, wh) : d->Nb % 4 == 0 ? go(prune_bp_scores_kernel<uint16_t, 4>, wh) : go(prune_bp_scores_kernel<uint16_t, 1>, wh);
    if (e != cudaSuccess) return NPAS_ERR_CUDA;
    // as many CTAs (a power of two, at most eight) as give each about two thousand keys
    const int RS = d->R * d->S;
    int ctas = 1;
    while (ctas < 8 && G > 2048ll * ctas) ctas *= 2;
    const long long most = (nBlk + ctas - 1) / ctas * RS;
    const int in_smem = most <= kSelSmemKeys;
    const size_t smem = in_smem ? (size_t)most * 8 : 0;
    if (allow_dynamic_smem(reinterpret_cast<const void *>(prune_select_kernel), (int)(kSelSmemKeys * 8)) != NPAS_OK) return NPAS_ERR_CUDA;
    if (tc::launch_pdl_cluster({}, prune_select_kernel, dim3(ctas), dim3(kSelThreads), ctas, smem, st, reinterpret_cast<const unsigned long long *>(scores),
                               (long long)n_keep, RS, masks, nBlk, ctas, in_smem) != cudaSuccess)
        return NPAS_ERR_CUDA;
    count_launch(2);
    return launch_status();
}

npas_status npas_prune_bb_magnitude(const npas_bb_desc *d, const void *w, int32_t keep_rows, int32_t keep_cols,
                                    uint64_t *row_keep, uint64_t *col_keep, void *stream)
{
    npas_status s = check_bb_desc(d);
    if (s != NPAS_OK) return s;
    if (!w || !row_keep || !col_keep) return NPAS_ERR_NULL;
    if (keep_rows < 0 || keep_rows > d->Bo || keep_cols < 0 || keep_cols > d->Bi) return NPAS_ERR_SHAPE;
    if (!aligned16(w) || (reinterpret_cast<uintptr_t>(row_keep) & 7) || (reinterpret_cast<uintptr_t>(col_keep) & 7))
        return NPAS_ERR_ALIGNMENT;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nBlk = (d->O / d->Bo) * (d->I / d->Bi);
    const cudaError_t e = d->w_in == NPAS_F32
        ? tc::launch_pdl({}, prune_bb_kernel<float>, dim3(nBlk), dim3(128), 0, st, *d, static_cast<const float *>(w), keep_rows, keep_cols, row_keep, col_keep)
        : tc::launch_pdl({}, prune_bb_kernel<uint16_t>, dim3(nBlk), dim3(128), 0, st, *d, static_cast<const uint16_t *>(w), keep_rows, keep_cols, row_keep, col_keep);
    if (e != cudaSuccess) return NPAS_ERR_CUDA;
    count_launch();
    return launch_status();
}

}  // extern "C"

}  // namespace npas
