// Block-based pruned GEMM in float64: the float32 path (products and sums in float64, one rounding at the store) and the
// fall-back for geometries the tcgen05 kernels do not take (bf16 inputs).  Only kept rows and columns are multiplied.
//
// A CTA owns 8 to 32 rows of X and one row of weight blocks.  Its rows of X (up to 512 columns at a time) are requested
// together, so that the memory latency is paid once and not once per block.  Groups of up to four warps take the column blocks
// in turn; a warp multiplies eight kept rows of the block by the rows of X with m8n8k4 float64 matrix instructions:
// the packed weights come straight from the blob into the A fragments (every weight is used by one warp only), the kept
// columns of X are picked out of the staged rows and widened on their way into the B fragments.  The next block's header, lists
// and first weights are on their way while a block is multiplied.  The result is added to
// the group's accumulators, which lie in shared memory because every block keeps other rows; the groups' sums are added
// at the end in a fixed order.
//
// Why matrix instructions: they run at the rate of the FMA instructions (64 FMAs per cycle and SM measured for both), but
// an 8x8x4 tile takes 64 operand words where FMAs fed from shared memory need one or two 16-byte loads per four FMAs; with
// FMAs the shared-memory path set the pace.  392x512 -> 512, 64x64 blocks keeping 32x32: 543 us with one row per thread
// walking the lists, 28.6 with 2x4 register tiles, 16.3 with four groups of them; with matrix instructions 9.5, and 7.9 on 136
// CTAs of 24 rows with the next block's loads on their way.
#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

namespace {

constexpr int kBM = 32;                     // rows of X per CTA
constexpr int kMaxWarps = 16;               // per CTA; a group has a warp per eight rows of a block, four at most
constexpr int kMaxGroups = 15;              // (one named barrier each)
constexpr int kAccPitch = 34;               // elements between the rows of the accumulators
constexpr int kPhaseCols = 512;             // columns of X staged at a time
constexpr int kSteps = 8;                   // matrix steps (of four columns) whose operands are in flight together

// Loads from global memory: as they stand (the pointer is a const __restrict__ argument), or NC: as __ldg, where the pointer
// comes from behind_wait and a plain load could not move across a store to shared memory.  (The kernel of blocks of up to 32
// rows is 2 to 20 % slower with the second form, the other one with the first.)
template <bool NC, typename T> __device__ __forceinline__ T lin_get(const T *p)
{
    if constexpr (NC) return __ldg(p);
    else return *p;
}
template <bool NC> __device__ __forceinline__ float lin_load(const float *p) { return lin_get<NC>(p); }
template <bool NC> __device__ __forceinline__ float lin_load(const uint16_t *p) { return bf16_bits_to_f32(lin_get<NC>(p)); }
template <typename T> __device__ inline void lin_store(T *p, float v);
template <> __device__ inline void lin_store<float>(float *p, float v) { *p = v; }
template <> __device__ inline void lin_store<uint16_t>(uint16_t *p, float v) { *p = f32_bits_to_bf16(__float_as_uint(v)); }

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// a warp copies `width` elements of a row of X, widened; `pairs`: the row and every piece of it start on even elements
template <bool NC> __device__ __forceinline__ void stage_row(float *dst, const float *src, int width, bool, int lane)
{
#pragma unroll 4
    for (int c = lane; c < width; c += 32) dst[c] = lin_get<NC>(src + c);
}
template <bool NC> __device__ __forceinline__ void stage_row(float *dst, const uint16_t *src, int width, bool pairs, int lane)
{
    if (pairs) {
#pragma unroll 4
        for (int c = 2 * lane; c < width; c += 64) {
            const uint32_t v = lin_get<NC>(reinterpret_cast<const uint32_t *>(src + c));
            *reinterpret_cast<float2 *>(dst + c) = make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
        }
    } else {
#pragma unroll 4
        for (int c = lane; c < width; c += 32) dst[c] = lin_load<NC>(src + c);
    }
}

__device__ __forceinline__ void group_sync(int g, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(threads) : "memory"); }

// D[8 x 8] += A[8 x 4] * B[4 x 8]; lane l holds A(l / 4, l % 4), B(l % 4, l / 4), D(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// Where the sum of row r of a block and row m of X lies in a group's accumulators: neighbours change places in every other eight rows, or a
// half warp that reads sixteen rows of one m would meet every bank twice.
__device__ __forceinline__ int acc_at(int r, int m) { return r * kAccPitch + (m ^ (r >> 3 & 1)); }

struct LinSimtSmem { uint32_t groups, group_threads, phase_cols, off_grp, grp_bytes, bytes; };

// Shared memory: the staged rows of X, then the accumulators of every group.
inline LinSimtSmem smem_plan(const npas_bb_desc &bb, int rows)
{
    LinSimtSmem s;
    const uint32_t Bi = bb.Bi, nBi = bb.I / Bi;
    s.phase_cols = bb.I < kPhaseCols ? (uint32_t)bb.I : kPhaseCols / Bi * Bi;
    s.off_grp = round_up(rows * (round_up(s.phase_cols, 8) + 4u) * 4u, 16);
    s.grp_bytes = (uint32_t)bb.Bo * kAccPitch * 8u;
    s.group_threads = bb.Bo > 24 ? 128u : (uint32_t)(bb.Bo + 7) / 8 * 32u;
    s.groups = kMaxWarps * 32 / s.group_threads;
    const uint32_t room = (232448u - 512u - s.off_grp) / s.grp_bytes;      // (beside the staged biases)
    if (s.groups > kMaxGroups) s.groups = kMaxGroups;
    if (s.groups > room) s.groups = room;
    if (s.groups > nBi) s.groups = nBi;
    s.bytes = s.off_grp + s.groups * s.grp_bytes;
    return s;
}

}  // namespace

// Rows of X per CTA, 8 MT of them: as many as fill the chip.  What a CTA spends whatever its rows (the chain of header, lists and
// weights, the sums of the groups) is about as long as four tiles of eight rows take on the matrix pipe, so the best MT is
// the one with the least rounds of CTAs times (4 + MT): 392x512 -> 512 runs on 136 CTAs of 24 rows (104 of 32 rows before).
static int simt_tiles(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    const long long sms = sm_count(), nBo = bb.O / bb.Bo;
    int best = 4;
    long long least = 0;
    for (int mt = 4; mt >= 1; --mt) {
        const long long rounds = ((d.M + 8 * mt - 1) / (8 * mt) * nBo + sms - 1) / sms, cost = rounds * (4 + mt);
        if (mt == 4 || cost < least) { best = mt; least = cost; }
    }
    return best;
}

// (registers for a second CTA wherever the groups leave threads for it)
template <typename TX, typename TY, int MT>
__global__ void __maxnreg__(104)
linear_bb_simt_kernel(npas_linear_desc d, int Bo, int Bi, BbLayout L, LinSimtSmem S, const TX *__restrict__ x,
                      const uint8_t *__restrict__ blob, const float *__restrict__ bias, const TY *__restrict__ res,
                      TY *__restrict__ y)
{
    constexpr int kRows = 8 * MT;
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ double bias_s[64];
    const int t = threadIdx.x, nt = blockDim.x, gt = (int)S.group_threads, g = t / gt, tg = t - g * gt, lane = t & 31;
    float *xraw = reinterpret_cast<float *>(sm);                                               // [kRows][pitch]
    double *acc = reinterpret_cast<double *>(sm + S.off_grp + (size_t)g * S.grp_bytes);       // [Bo][kAccPitch]

    int bo = blockIdx.y, m0 = blockIdx.x * kRows;
    const int rows_here = min(kRows, d.M - m0), nBi = (int)L.nBi, G = (int)S.groups;
    const bool x16 = sizeof(TX) == 4 && (d.I & 3) == 0 && (Bi & 3) == 0;
    const bool x2 = (d.I & 1) == 0 && (Bi & 1) == 0;
    const int per_phase = (int)S.phase_cols / Bi, k = lane & 3, q = lane >> 2, r_first = (tg >> 5) * 8;

    tc::pdl_trigger();
    if (g < G)                                                                                 // (the threads behind the groups help with X and Y)
        for (int e = tg; e < Bo * kAccPitch; e += gt) acc[e] = 0;
    tc::pdl_wait();
    const int z = tc::zero_behind_wait();                              // (every address below follows from these two; opaque pointers: up to 3 % slower)
    bo += z; m0 += z;
    const uint32_t *voff = reinterpret_cast<const uint32_t *>(blob + L.off_voff);
    const TX *vals = reinterpret_cast<const TX *>(blob + L.off_values);

    // A block's header, and this warp's first eight kept rows by 32 kept columns of it.  (A row or column number outside the
    // block counts for nothing.)
    struct Header { uint32_t blk, off, cnt; };
    struct Part { float w[kSteps]; int col[kSteps], row; };
    for (int b0 = 0; b0 < nBi; b0 += per_phase) {
        const int nb = min(per_phase, nBi - b0), width = nb * Bi, pitch = (int)round_up((uint32_t)width, 8) + 4;
        auto header = [&](int b) {
            Header h = {0, 0, 0};
            if (b >= nb || g >= G) return h;
            h.blk = (uint32_t)bo * L.nBi + b0 + b;
            h.off = __ldg(voff + h.blk);
            h.cnt = __ldg(reinterpret_cast<const uint16_t *>(blob + L.off_cnt + 2 * h.blk));
            return h;
        };
        auto part = [&](const Header &h, int r0, int c0) {
            Part p;
            const int nr = min((int)(h.cnt & 0xFFu), Bo), nc = min((int)(h.cnt >> 8), Bi), r = r0 + q;
            const TX *w = vals + h.off + (size_t)r * nc;
            const uint8_t *cl = blob + L.off_cols + (size_t)h.blk * Bi;
            p.row = r < nr ? __ldg(blob + L.off_rows + (size_t)h.blk * Bo + r) : Bo;
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
                const int c = c0 + 4 * i + k;
                p.w[i] = r < nr && c < nc ? lin_load<true>(w + c) : 0.f;
                p.col[i] = c < nc ? __ldg(cl + c) : Bi;
            }
            return p;
        };
        Header now = header(g), next = header(g + G);                  // (on their way while the rows of X are requested)
        if (b0) __syncthreads();                                       // the phase before has been read
        for (int r = t >> 5; r < rows_here; r += nt >> 5) {            // a warp per row
            const TX *src = x + (size_t)(m0 + r) * d.I + (size_t)b0 * Bi;
            float *dst = xraw + r * pitch;
            if (x16) for (int c = lane * 4; c < width; c += 128) cp_async16(dst + c, src + c);
            else stage_row<true>(dst, src, width, x2, lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (t < Bo) bias_s[t] = bias ? (double)__ldg(bias + bo * Bo + t) : 0.;
        Part first = part(now, r_first, 0);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        for (int b = g < G ? g : nb; b < nb; b += G) {
            const Header h = now;
            Part p = first;
            if (b + G < nb) {                                          // the next block's, while this one is multiplied
                now = next;
                first = part(now, r_first, 0);
                next = header(b + 2 * G);
            }
            const int nr = min((int)(h.cnt & 0xFFu), Bo), nc = min((int)(h.cnt >> 8), Bi), col0 = b * Bi;
            for (int r0 = r_first; r0 < nr; r0 += gt / 4) {            // eight kept rows per warp
                double a[MT][2] = {};
                int row = Bo;
                for (int c0 = 0; c0 < nc; c0 += 4 * kSteps) {
                    if (r0 != r_first || c0) p = part(h, r0, c0);
                    row = p.row;
#pragma unroll
                    for (int i = 0; i < kSteps; ++i) {
                        if (c0 + 4 * i >= nc) break;
                        const bool in = p.col[i] < Bi;
                        const float *xp = xraw + q * pitch + col0 + p.col[i];
#pragma unroll
                        for (int m = 0; m < MT; ++m) mma_f64(a[m], (double)p.w[i], in ? (double)xp[m * 8 * pitch] : 0.);
                    }
                }
                if (row < Bo) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        double2 *s = reinterpret_cast<double2 *>(acc + row * kAccPitch + m * 8 + 2 * k);
                        double2 v = *s;
                        v.x += row & 8 ? a[m][1] : a[m][0]; v.y += row & 8 ? a[m][0] : a[m][1];      // (acc_at)
                        *s = v;
                    }
                }
            }
            group_sync(g, gt);         // the next block adds to other rows from other warps
        }
    }
    __syncthreads();
    // The groups' sums in order, bias, residual, ReLU, one rounding.
    const double *acc0 = reinterpret_cast<const double *>(sm + S.off_grp);
    const size_t acc_step = S.grp_bytes / 8;
    if (res) {
        // A warp takes eight outputs of four rows at a time: whole 32-byte sectors.  Four of them, so that the residual's loads do
        // not wait for one another's stores.
        const int across = (Bo + 7) / 8, warps = nt >> 5, step_r = warps % across, step_m = warps / across;
        int ru = (t >> 5) % across, mu = (t >> 5) / across;
        for (const int m4 = (rows_here + 3) / 4; mu < m4;) {
            int r[4], m[4];
            float rv[4];
            double v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                r[j] = ru * 8 + (lane & 7); m[j] = mu * 4 + (lane >> 3);
                if (r[j] >= Bo || m[j] >= rows_here) m[j] = -1;
                ru += step_r; mu += step_m;
                if (ru >= across) { ru -= across; ++mu; }
                rv[j] = m[j] >= 0 ? lin_load<true>(res + (size_t)(m0 + m[j]) * d.O + bo * Bo + r[j]) : 0.f;
                v[j] = m[j] >= 0 ? acc0[acc_at(r[j], m[j])] : 0.;
            }
            for (int i = 1; i < G; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] += m[j] >= 0 ? acc0[i * acc_step + acc_at(r[j], m[j])] : 0.;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (m[j] < 0) continue;
                v[j] += bias_s[r[j]];
                v[j] += (double)rv[j];
                if (d.relu) v[j] = v[j] > 0 ? v[j] : 0;
                lin_store(y + (size_t)(m0 + m[j]) * d.O + bo * Bo + r[j], (float)v[j]);
            }
        }
    } else {
        // Consecutive threads along the row of Y.  (The form above without its loads: 1722x64 -> 512 7.5 us, here 5.7; 3136x64 -> 512 13.2 and
        // 10.4; 392x512 -> 512 8.1 and 7.9.)
        const int step_r = nt % Bo, step_m = nt / Bo;
        int r = t % Bo;
#pragma unroll 4
        for (int m = t / Bo; m < rows_here;) {
            double v = acc0[acc_at(r, m)];
            for (int i = 1; i < G; ++i) v += acc0[i * acc_step + acc_at(r, m)];
            v += bias_s[r];
            if (d.relu) v = v > 0 ? v : 0;
            lin_store(y + (size_t)(m0 + m) * d.O + bo * Bo + r, (float)v);
            r += step_r; m += step_m;
            if (r >= Bo) { r -= Bo; ++m; }
        }
    }
}

// ---- blocks of up to 32 rows --------------------------------------------------------------------------------------------------
// Many blocks, each a header, lists and a few weights: a chain of loads for a handful of matrix instructions, whose latency is
// what bounds it.  So here a block belongs to one warp, which has the next block's lists and first weights (and the header of the
// one after) on their way, accumulates in a tile of its own and meets the others only between phases of 256 columns; with
// three CTAs per SM and `gb` rows of blocks on the same staged rows of X.  The warps' sums are added in order at the end.
struct LinRowsPlan { uint32_t warps, gb, phase_cols, pitch, off_acc, bytes; };
constexpr int kRowsWarps = 8;
constexpr int kRowsOutputs = 16;            // outputs per CTA where a row of blocks has fewer
constexpr int kRowsCols = 256;              // columns of X staged at a time

static LinRowsPlan rows_plan(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    LinRowsPlan p;
    const uint32_t nBo = bb.O / bb.Bo, nBi = bb.I / bb.Bi, mt = (uint32_t)(d.M + kBM - 1) / kBM;
    p.gb = bb.Bo < kRowsOutputs ? kRowsOutputs / bb.Bo : 1u;
    while (p.gb > 1 && (uint64_t)mt * ((nBo + p.gb - 1) / p.gb) < 4ull * sm_count()) --p.gb;
    p.phase_cols = bb.I < kRowsCols ? (uint32_t)bb.I : kRowsCols / bb.Bi * bb.Bi;
    p.pitch = round_up(p.phase_cols, 8) + 4;
    p.warps = p.gb * nBi < kRowsWarps ? p.gb * nBi : kRowsWarps;
    p.off_acc = round_up(kBM * p.pitch * 4u, 16);
    p.bytes = p.off_acc + p.warps * p.gb * bb.Bo * kAccPitch * 8u;
    return p;
}

// Against the kernel above, whose CTA gives a block to several warps and takes as few rows as fill the chip: here where that one
// would need a second round of CTAs and a row of blocks has work for all warps (392x512 -> 512 in 32x32 blocks keeping 8x16 17.2 us
// there, 8.4 here; 160x512 -> 512 in 16x64 keeping 8x32 10.2 and 9.4; 3136x508 -> 508 in 4x4 keeping 2x2 1030 and 497), two CTAs per
// SM and half of the warps, or four per SM in any case (705x128 -> 960, two blocks of 20x64 in a row, 17 and 9).  On smaller grids the
// kernel above is the better one (100x512 -> 512 in 16x64 5.9 and 8.9, 392x64 -> 512 in 32x32 5.1 and 9.3).
static bool rows_preferred(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    const long long ctas = (long long)((d.M + kBM - 1) / kBM) * (bb.O / bb.Bo), sms = sm_count();
    const int nBi = bb.I / bb.Bi;
    return bb.Bo <= 32 && (ctas >= 4 * sms || (ctas >= 2 * sms && nBi >= 4) || (ctas > sms && nBi >= 8));
}

// HELP: warps behind the plan's, which have no blocks and only move X and Y.
template <typename TX, typename TY, bool HELP>
__global__ void __launch_bounds__(kRowsWarps * 32, 3)
linear_bb_rows_kernel(npas_linear_desc d, int Bo, int Bi, BbLayout L, LinRowsPlan S, const TX *__restrict__ x,
                      const uint8_t *__restrict__ blob, const float *__restrict__ bias, const TY *__restrict__ res,
                      TY *__restrict__ y)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const int t = threadIdx.x, nt = blockDim.x, warp = t >> 5, lane = t & 31, k = lane & 3, q = lane >> 2, W = (int)S.warps, pitch = (int)S.pitch;
    const int bo0 = blockIdx.y * (int)S.gb, gb = min((int)S.gb, (int)L.nBo - bo0), outs = gb * Bo;
    float *xs = reinterpret_cast<float *>(sm);                                                          // [kBM][pitch]
    double *acc0 = reinterpret_cast<double *>(sm + S.off_acc), *acc = acc0 + (size_t)warp * outs * kAccPitch;   // [W][outs][kAccPitch]
    const int m0 = blockIdx.x * kBM, rows_here = min(kBM, d.M - m0), nBi = (int)L.nBi, per_phase = (int)S.phase_cols / Bi;
    const bool x16 = sizeof(TX) == 4 && (d.I & 3) == 0 && (Bi & 3) == 0, x2 = (d.I & 1) == 0 && (Bi & 1) == 0;

    tc::pdl_trigger();
    if (!HELP || warp < W)
        for (int e = lane; e < outs * kAccPitch; e += 32) acc[e] = 0;
    tc::pdl_wait();
    for (int b0 = tc::zero_behind_wait(); b0 < nBi; b0 += per_phase) {
        const int nb = min(per_phase, nBi - b0), width = nb * Bi;
        if (b0) __syncthreads();                                       // the phase before has been read
        for (int r = warp; r < rows_here; r += HELP ? nt >> 5 : W) {      // a warp per row
            const TX *src = x + (size_t)(m0 + r) * d.I + (size_t)b0 * Bi;
            float *dst = xs + r * pitch;
            if (x16) for (int c = lane * 4; c < width; c += 128) cp_async16(dst + c, src + c);
            else stage_row<false>(dst, src, width, x2, lane);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        // the phase's blocks, a warp every W-th: row of blocks `hr`, block b0 + `hb` of it
        struct Block { uint32_t blk, off, cnt; int at, base, row, c0, c1; float w[4]; };
        int hr = !HELP || warp < W ? 0 : gb, hb = warp;
        while (hb >= nb) { hb -= nb; ++hr; }
        auto header = [&](Block &n) {
            n.off = n.cnt = 0; n.blk = ~0u;
            if (hr >= gb) return;
            n.blk = (uint32_t)(bo0 + hr) * L.nBi + (uint32_t)(b0 + hb);
            n.at = hr * Bo * kAccPitch; n.base = hb * Bi;
            n.off = reinterpret_cast<const uint32_t *>(blob + L.off_voff)[n.blk];
            n.cnt = *reinterpret_cast<const uint16_t *>(blob + L.off_cnt + 2 * n.blk);
            hb += W;
            while (hb >= nb) { hb -= nb; ++hr; }
        };
        auto kept = [&](const Block &n, int &nr, int &nc) { nr = min((int)(n.cnt & 0xFFu), Bo); nc = min((int)(n.cnt >> 8), Bi); };
        // rows r0 .. r0 + 7, columns c0 .. c0 + 15 of the block's weights
        auto weights = [&](const Block &n, int nr, int nc, int r0, int c0, float (&w)[4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = c0 + 4 * i + k;
                w[i] = r0 + q < nr && c < nc ? lin_load<false>(reinterpret_cast<const TX *>(blob + L.off_values) + n.off + (r0 + q) * nc + c) : 0.f;
            }
        };
        auto lists = [&](Block &n) {
            if (n.blk == ~0u) return;
            int nr, nc;
            kept(n, nr, nc);
            const uint8_t *rl = blob + L.off_rows + (size_t)n.blk * Bo, *cl = blob + L.off_cols + (size_t)n.blk * Bi;
            n.row = lane < nr ? rl[lane] : Bo;                         // (a row or column number outside the block counts for nothing)
            n.c0 = lane < nc ? cl[lane] : Bi;
            n.c1 = lane + 32 < nc ? cl[lane + 32] : Bi;
            weights(n, nr, nc, 0, 0, n.w);
        };
        Block now, next;
        header(now);
        lists(now);
        header(next);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        while (now.blk != ~0u) {
            const Block b = now;
            now = next;
            lists(now);
            header(next);
            int nr, nc;
            kept(b, nr, nc);
            for (int r0 = 0; r0 < nr; r0 += 8) {
                const int row = __shfl_sync(0xFFFFFFFFu, b.row, (r0 + q) & 31);
                double a[kBM / 8][2] = {};
                for (int c0 = 0; c0 < nc; c0 += 16) {
                    float w[4];
                    if (r0 | c0) weights(b, nr, nc, r0, c0, w);
                    else {
#pragma unroll
                        for (int i = 0; i < 4; ++i) w[i] = b.w[i];
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (c0 + 4 * i >= nc) break;
                        const int col = __shfl_sync(0xFFFFFFFFu, c0 < 32 ? b.c0 : b.c1, (c0 + 4 * i + k) & 31);
                        const float *xp = xs + q * pitch + b.base + col;
#pragma unroll
                        for (int m = 0; m < kBM / 8; ++m) mma_f64(a[m], (double)w[i], col < Bi ? (double)xp[m * 8 * pitch] : 0.);
                    }
                }
                if (r0 + q < nr && row < Bo) {
#pragma unroll
                    for (int m = 0; m < kBM / 8; ++m) {
                        double2 *p = reinterpret_cast<double2 *>(acc + b.at + row * kAccPitch + m * 8 + 2 * k);
                        double2 v = *p;
                        v.x += a[m][0]; v.y += a[m][1];
                        *p = v;
                    }
                }
                __syncwarp();                                          // (two rows of the list may be one, in a damaged blob)
            }
        }
    }
    __syncthreads();
    // the warps' sums in order, bias, residual, ReLU, one rounding; consecutive threads along the row of Y
    for (int e = t + tc::zero_behind_wait(); e < outs * rows_here; e += nt) {
        const int m = e / outs, r = e - m * outs;
        const size_t o = (size_t)(m0 + m) * d.O + (size_t)bo0 * Bo + r;
        double v = acc0[r * kAccPitch + m];
        for (int w = 1; w < W; ++w) v += acc0[((size_t)w * outs + r) * kAccPitch + m];
        if (bias) v += (double)bias[bo0 * Bo + r];
        if (res) v += (double)lin_load<false>(res + o);
        if (d.relu) v = v > 0 ? v : 0;
        lin_store(y + o, (float)v);
    }
}

template <typename TX, typename TY>
static npas_status launch(const npas_linear_desc &d, const npas_bb_desc &bb, const BbLayout &L, dim3 grid, const void *x,
                          const void *blob, const float *bias, const void *res, void *y, cudaStream_t st, Launch how)
{
    if (rows_preferred(d, bb)) {
        const LinRowsPlan p = rows_plan(d, bb);
        // up to four warps where an SM has room for them beside all its CTAs, the ones without blocks to move X and Y (200x64 -> 1000 in
        // 8x64 blocks, one warp, three CTAs per SM: 10 us, with four 5.9; 2000x64 -> 512 in 32x32, seven per SM: 13.4 and 17.7)
        const uint32_t gy = (L.nBo + p.gb - 1) / p.gb, per_sm = (grid.x * gy + (uint32_t)sm_count() - 1) / (uint32_t)sm_count();
        uint32_t warps = per_sm <= 6 ? 4 : 24 / per_sm;
        if (warps < p.warps) warps = p.warps;
        auto k = warps > p.warps ? linear_bb_rows_kernel<TX, TY, true> : linear_bb_rows_kernel<TX, TY, false>;
        if (allow_dynamic_smem(reinterpret_cast<const void *>(k), (int)p.bytes) != NPAS_OK) return NPAS_ERR_CUDA;
        const cudaError_t e = tc::launch_pdl(how, k, dim3(grid.x, gy), dim3(warps * 32), p.bytes, st, d, (int)bb.Bo, (int)bb.Bi, L, p,
                                             static_cast<const TX *>(x), static_cast<const uint8_t *>(blob), bias, static_cast<const TY *>(res), static_cast<TY *>(y));
        count_launch();
        return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
    }
    const int tiles = simt_tiles(d, bb);
    const LinSimtSmem S = smem_plan(bb, 8 * tiles);
    // threads beyond the groups' where an SM has few CTAs: rows of X and outputs are moved by all of them (392x64 -> 512, one block
    // of 64x64 in a row, 6.9 us with the group's 128 threads, 4.6 with 512)
    const dim3 ctas((d.M + 8 * tiles - 1) / (8 * tiles), L.nBo);
    const uint32_t per_sm = (ctas.x * ctas.y + (uint32_t)sm_count() - 1) / (uint32_t)sm_count(), wanted = per_sm == 1 ? 512u : per_sm == 2 ? 256u : 128u;
    const uint32_t threads = S.group_threads * S.groups > wanted ? S.group_threads * S.groups : wanted;
    auto go = [&](auto k) {
        if (allow_dynamic_smem(reinterpret_cast<const void *>(k), (int)S.bytes) != NPAS_OK) return NPAS_ERR_CUDA;
        const cudaError_t e = tc::launch_pdl(how, k, ctas, dim3(threads), S.bytes, st, d, (int)bb.Bo,
                                             (int)bb.Bi, L, S, static_cast<const TX *>(x), static_cast<const uint8_t *>(blob), bias, static_cast<const TY *>(res),
                                             static_cast<TY *>(y));
        count_launch();
        return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
    };
    return tiles == 4 ? go(linear_bb_simt_kernel<TX, TY, 4>) : tiles == 3 ? go(linear_bb_simt_kernel<TX, TY, 3>)
         : tiles == 2 ? go(linear_bb_simt_kernel<TX, TY, 2>) : go(linear_bb_simt_kernel<TX, TY, 1>);
}

npas_status linear_simt_launch(const npas_linear_desc &d, const npas_bb_desc &bb, const void *x,
                               const void *blob, const float *bias, const void *res, void *y, cudaStream_t st, Launch how)
{
    const BbLayout L = bb_layout(bb);
    const dim3 grid((d.M + kBM - 1) / kBM, L.nBo);
    if (grid.y > 65535) return NPAS_ERR_UNSUPPORTED;
    if (d.x_dtype == NPAS_F32 && d.y_dtype == NPAS_F32) return launch<float, float>(d, bb, L, grid, x, blob, bias, res, y, st, how);
    if (d.x_dtype == NPAS_BF16 && d.y_dtype == NPAS_BF16) return launch<uint16_t, uint16_t>(d, bb, L, grid, x, blob, bias, res, y, st, how);
    if (d.x_dtype == NPAS_BF16 && d.y_dtype == NPAS_F32) return launch<uint16_t, float>(d, bb, L, grid, x, blob, bias, res, y, st, how);
    return NPAS_ERR_DTYPE;
}

}  // namespace npas
