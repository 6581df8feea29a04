// One-shot magnitude pruning of a layer under the two schemes (paper Sec. 5.2): turns dense
// weights into the block masks the packers take.  The score of a prunable group (a tap of a block;
// a row or a column of a block) is the sum of the squares of its weights, accumulated in fp64 in a
// fixed order (filters / rows outer, channels / columns inner; a square of a float is exact in
// fp64, so fused or separate multiply-add give the same bits); a block keeps its `keep`
// highest-scoring groups, ties go to the lower index.  Offline step: one CTA per block for the per-block counts; for the
// layer-wide budget a thread per group scores and a cluster selects.
#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

template <typename T> __device__ inline double prune_load(const T *p);
template <> __device__ inline double prune_load<float>(const float *p) { return (double)*p; }
template <> __device__ inline double prune_load<uint16_t>(const uint16_t *p) { return (double)bf16_bits_to_f32(*p); }

// V consecutive weights (V = 1, 4, or 8 bf16) as floats
template <int V> __device__ __forceinline__ void prune_load_vec(const float *p, float (&v)[V])
{
    if constexpr (V == 4) { const float4 u = __ldg(reinterpret_cast<const float4 *>(p)); v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w; }
    else v[0] = __ldg(p);
}
template <int V> __device__ __forceinline__ void prune_load_vec(const uint16_t *p, float (&v)[V])
{
    if constexpr (V == 1) v[0] = bf16_bits_to_f32(__ldg(p));
    else {
        uint32_t u[V / 2];
        if constexpr (V == 8) { const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p)); u[0] = q.x; u[1] = q.y; u[2] = q.z; u[3] = q.w; }
        else { const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p)); u[0] = q.x; u[1] = q.y; }
#pragma unroll
        for (int j = 0; j < V / 2; ++j) { v[2 * j] = __uint_as_float(u[j] << 16); v[2 * j + 1] = __uint_as_float(u[j] & 0xFFFF0000u); }
    }
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
    const T *blk = w + (size_t)bo * d.Bo * d.I + (size_t)bi * d.Bi;
    const bool c1 = (t & 31) < d.Bi, c2 = (t & 31) + 32 < d.Bi;
#pragma unroll 8
    for (int r = t >> 5; r < d.Bo; r += 4) {
        const T *p = blk + (size_t)r * d.I + (t & 31);
        const float a = c1 ? (float)prune_load(p) : 0.f, b2 = c2 ? (float)prune_load(p + 32) : 0.f;
        blk_s[r][t & 31] = a; blk_s[r][(t & 31) + 32] = b2;
    }
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
// time.  The sums are ordered, so what counts is that loads do not wait for them: eight vectors at a time are requested,
// the next eight before the present ones are added (512x3x3x512 in 16x8 blocks: 15 us with one run after the other).
template <typename T, int V>
__global__ void __launch_bounds__(128)
prune_bp_scores_kernel(npas_bp_desc d, const T *__restrict__ w, double *scores)
{
    constexpr int kBatch = 8;
    tc::pdl_trigger();
    const int RS = d.R * d.S, nCB = d.C / d.Nb;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, total = (long long)(d.K / d.Mb) * RS * nCB;
    if (i >= total) return;
    const int cb = (int)(i % nCB), rest = (int)(i / nCB), t = rest % RS, fb = rest / RS;
    const T *p = w + ((size_t)fb * d.Mb * RS + t) * d.C + (size_t)cb * d.Nb;      // the next vector to request
    const size_t step = (size_t)RS * d.C - d.Nb;                                   // from the end of a run to the next filter's
    const int vecs = d.Mb * (d.Nb / V), per_run = d.Nb / V;
    int asked = 0, in_run = 0;
    auto request = [&](float (&v)[kBatch][V]) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            if (asked < vecs) {
                prune_load_vec<V>(p, v[j]);
                ++asked;
                p += V;
                if (++in_run == per_run) { in_run = 0; p += step; }
            } else {
#pragma unroll
                for (int q = 0; q < V; ++q) v[j][q] = 0.f;                          // (adding +0 to a sum of squares changes nothing)
            }
        }
    };
    double s = 0.0;
    auto add = [&](const float (&v)[kBatch][V]) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j)
#pragma unroll
            for (int q = 0; q < V; ++q) s = fma((double)v[j][q], (double)v[j][q], s);
    };
    float a[kBatch][V], b[kBatch][V];
    request(a);
    for (int done = 0; done < vecs; done += 2 * kBatch) {
        request(b);
        add(a);
        request(a);
        add(b);
    }
    scores[((size_t)fb * nCB + cb) * RS + t] = s;
}

// Keeps the n_keep largest of G scores, ties to the lower index, and writes the tap sets.  One cluster; every CTA holds
// the keys of a range of whole blocks (in shared memory when they fit).  A sum of squares is never negative, so the order
// of the fp64 values is that of their bit patterns as unsigned integers: the threshold is found by a radix select over
// the bits in which keys differ at all, eight at a time from the top.  Per pass every CTA counts its candidates per digit,
// and after one cluster barrier every CTA adds the CTAs' counts (through distributed shared memory) and walks the digits
// downwards to the one in which the remaining budget falls.  The search ends when that digit holds exactly the budget,
// after three or four passes for scores that differ; only when all bits are used up do equal keys remain to be taken in
// index order.  (One CTA over all 64 bits, with every key of a pass hitting the same few counters, took 77 us for 18432
// groups.)
constexpr int kSelThreads = 256;
constexpr uint32_t kSelSmemKeys = 24576;                        // 192 KB of keys per CTA

struct SelShared {
    unsigned int hist[2][256];
    unsigned long long all_and, all_or, warp_and[kSelThreads / 32], warp_or[kSelThreads / 32];
    unsigned int warp_sums[kSelThreads / 32];
    unsigned int eq_total;
    unsigned int pick[2];
};

__device__ __forceinline__ unsigned int sel_rank() { unsigned int r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void sel_cluster_sync() { asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ unsigned int sel_remote(const void *p, unsigned int rank)
{
    unsigned int a = (unsigned int)__cvta_generic_to_shared(p), v;
    asm volatile("{\n\t.reg .u32 q;\n\tmapa.shared::cluster.u32 q, %1, %2;\n\tld.shared::cluster.u32 %0, [q];\n\t}" : "=r"(v) : "r"(a), "r"(rank) : "memory");
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
    const unsigned long long *src = keys + b_lo * RS;
    const long long n = (b_hi - b_lo) * RS;
    sh.hist[0][t] = 0; sh.hist[1][t] = 0;
    tc::pdl_wait();                    // (started while the scores are being computed)
    {
        unsigned long long a = ~0ull, o = 0ull;
#pragma unroll 4
        for (long long i = t; i < n; i += kSelThreads) {
            const unsigned long long k = src[i];
            if (in_smem) key_smem[i] = k;
            a &= k; o |= k;
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) { a &= __shfl_xor_sync(0xFFFFFFFFu, a, d); o |= __shfl_xor_sync(0xFFFFFFFFu, o, d); }
        if (lane == 0) { sh.warp_and[wid] = a; sh.warp_or[wid] = o; }
        __syncthreads();
        if (wid == 0) {
            a = sh.warp_and[lane & (kSelThreads / 32 - 1)]; o = sh.warp_or[lane & (kSelThreads / 32 - 1)];
#pragma unroll
            for (int d = kSelThreads / 64; d; d >>= 1) { a &= __shfl_xor_sync(0xFFFFFFFFu, a, d); o |= __shfl_xor_sync(0xFFFFFFFFu, o, d); }
            if (lane == 0) { sh.all_and = a; sh.all_or = o; }
        }
    }
    if (in_smem) src = key_smem;
    sel_cluster_sync();
    // (a lane per CTA, then across the warp: one round trip)
    unsigned long long all_and = ~0ull, all_or = 0ull;
    if (lane < n_ctas) {
        const unsigned int *pa = reinterpret_cast<const unsigned int *>(&sh.all_and), *po = reinterpret_cast<const unsigned int *>(&sh.all_or);
        all_and = (unsigned long long)sel_remote(pa, lane) | ((unsigned long long)sel_remote(pa + 1, lane) << 32);
        all_or = (unsigned long long)sel_remote(po, lane) | ((unsigned long long)sel_remote(po + 1, lane) << 32);
    }
#pragma unroll
    for (int d = 4; d; d >>= 1) { all_and &= __shfl_xor_sync(0xFFFFFFFFu, all_and, d); all_or |= __shfl_xor_sync(0xFFFFFFFFu, all_or, d); }
    all_and = __shfl_sync(0xFFFFFFFFu, all_and, 0); all_or = __shfl_sync(0xFFFFFFFFu, all_or, 0);
    const unsigned long long differ = all_and ^ all_or;
    int bits = differ ? 64 - __clzll((long long)differ) : 0;     // bits still to be decided
    unsigned long long prefix = bits == 64 ? 0ull : all_and >> bits << bits, mask = bits == 64 ? 0ull : ~0ull << bits;
    unsigned int need = (unsigned int)n_keep, have = 0xFFFFFFFFu;      // to take among the keys with this prefix; how many there are
    if (bits == 0) have = (unsigned int)(n_blocks * RS);
    for (int pass = 0; bits > 0 && need != have; ++pass) {
        const int w = min(8, bits), shift = bits - w;
        unsigned int *hist = sh.hist[pass & 1];
#pragma unroll 4
        for (long long i = t; i < n; i += kSelThreads) {
            const unsigned long long k = src[i];
            if ((k & mask) == prefix) atomicAdd(&hist[(unsigned int)(k >> shift) & 255u & ((1u << w) - 1u)], 1u);
        }
        sel_cluster_sync();
        {
            // (a thread per digit) counts of all CTAs, then how many keys have this digit or a larger one (warp scans from the top, then over the warps)
            unsigned int c = 0;
            const int digit = 255 - t;
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (r < n_ctas) c += sel_remote(&hist[digit], r);
            unsigned int up = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, up, d); if (lane >= d) up += v; }
            if (lane == 31) sh.warp_sums[wid] = up;
            __syncthreads();
            for (int i = 0; i < wid; ++i) up += sh.warp_sums[i];
            if (up >= need && up - c < need) { sh.pick[0] = (unsigned int)digit; sh.pick[1] = up - c; sh.eq_total = c; }
        }
        __syncthreads();
        need -= sh.pick[1];
        have = sh.eq_total;
        prefix |= (unsigned long long)sh.pick[0] << shift;
        bits = shift;
        mask = bits == 64 ? 0ull : ~0ull << bits;
        sh.hist[(pass + 1) & 1][t] = 0;            // (every CTA has read the counts of the pass before)
        __syncthreads();
    }
    // keys above the prefix are kept; of those with the prefix all, or (equal keys) the first `need` in index order
    const bool ranked = need != have;
    const long long nb = b_hi - b_lo, chunk = (nb + kSelThreads - 1) / kSelThreads;
    const long long t_lo = min(nb, t * chunk), t_hi = min(nb, t_lo + chunk);
    unsigned int before = 0;
    if (ranked) {
        unsigned int mine = 0;
        for (long long i = t_lo * RS; i < t_hi * RS; ++i) mine += (src[i] & mask) == prefix;
        unsigned int up = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const unsigned int v = __shfl_up_sync(0xFFFFFFFFu, up, d); if (lane >= d) up += v; }
        if (lane == 31) sh.warp_sums[wid] = up;
        __syncthreads();
        for (int i = 0; i < wid; ++i) up += sh.warp_sums[i];
        if (t == kSelThreads - 1) sh.eq_total = up;
        sel_cluster_sync();
        for (unsigned int r = 0; r < rank; ++r) before += sel_remote(&sh.eq_total, r);
        before += up - mine;
    }
    if (!ranked) {
        for (long long b = t; b < nb; b += kSelThreads) {
            unsigned long long m = 0;
            for (int i = 0; i < RS; ++i) m |= (unsigned long long)((src[b * RS + i] & mask) >= prefix) << i;
            tap_mask[b_lo + b] = m;
        }
    } else {
        for (long long b = t_lo; b < t_hi; ++b) {
            unsigned long long m = 0;
            for (int i = 0; i < RS; ++i) {
                const unsigned long long k = src[b * RS + i] & mask;
                const bool eq = k == prefix;
                m |= (unsigned long long)(k > prefix || (eq && before < need)) << i;
                before += eq;
            }
            tap_mask[b_lo + b] = m;
        }
    }
    sel_cluster_sync();                // no CTA leaves while another may read its shared memory
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
    const unsigned grid = (unsigned)((G + 127) / 128);
    const float *wf = static_cast<const float *>(w);
    const uint16_t *wh = static_cast<const uint16_t *>(w);
    if (d->w_in == NPAS_F32) {
        if (d->Nb % 4 == 0) prune_bp_scores_kernel<float, 4><<<grid, 128, 0, st>>>(*d, wf, scores);
        else prune_bp_scores_kernel<float, 1><<<grid, 128, 0, st>>>(*d, wf, scores);
    } else {
        if (d->Nb % 8 == 0) prune_bp_scores_kernel<uint16_t, 8><<<grid, 128, 0, st>>>(*d, wh, scores);
        else if (d->Nb % 4 == 0) prune_bp_scores_kernel<uint16_t, 4><<<grid, 128, 0, st>>>(*d, wh, scores);
        else prune_bp_scores_kernel<uint16_t, 1><<<grid, 128, 0, st>>>(*d, wh, scores);
    }
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
    if (d->w_in == NPAS_F32)
        prune_bb_kernel<float><<<nBlk, 128, 0, st>>>(*d, static_cast<const float *>(w), keep_rows, keep_cols, row_keep, col_keep);
    else
        prune_bb_kernel<uint16_t><<<nBlk, 128, 0, st>>>(*d, static_cast<const uint16_t *>(w), keep_rows, keep_cols, row_keep, col_keep);
    count_launch();
    return launch_status();
}

}  // extern "C"

}  // namespace npas
