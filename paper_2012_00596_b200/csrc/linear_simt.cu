// Block-based pruned GEMM in float64: the float32 path (products and sums in float64, one rounding at the store) and the
// fall-back for geometries the tcgen05 kernels do not take (bf16 inputs).  Only kept rows and columns are multiplied.
//
// A CTA owns 32 rows of X and one row of weight blocks.  Its rows of X (up to 512 columns at a time) are requested
// together, so that the memory latency is paid once and not once per block.  Groups of up to four warps take the column blocks
// in turn; a warp multiplies eight kept rows of the block by the 32 rows of X with m8n8k4 float64 matrix instructions:
// the packed weights come straight from the blob into the A fragments (every weight is used by one warp only), the kept
// columns of X are picked out of the staged rows and widened on their way into the B fragments.  The result is added to
// the group's accumulators, which lie in shared memory because every block keeps other rows; the groups' sums are added
// at the end in a fixed order.
//
// Why matrix instructions: they run at the rate of the FMA instructions (64 FMAs per cycle and SM measured for both), but
// an 8x8x4 tile takes 64 operand words where FMAs fed from shared memory need one or two 16-byte loads per four FMAs; with
// FMAs the shared-memory path set the pace.  392x512 -> 512, 64x64 blocks keeping 32x32: 543 us with one row per thread
// walking the lists, 28.6 with 2x4 register tiles, 16.3 with four groups of them.
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

template <typename T> __device__ inline float lin_load(const T *p);
template <> __device__ inline float lin_load<float>(const float *p) { return *p; }
template <> __device__ inline float lin_load<uint16_t>(const uint16_t *p) { return bf16_bits_to_f32(*p); }
template <typename T> __device__ inline void lin_store(T *p, float v);
template <> __device__ inline void lin_store<float>(float *p, float v) { *p = v; }
template <> __device__ inline void lin_store<uint16_t>(uint16_t *p, float v) { *p = f32_bits_to_bf16(__float_as_uint(v)); }

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void group_sync(int g, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(threads) : "memory"); }

// D[8 x 8] += A[8 x 4] * B[4 x 8]; lane l holds A(l / 4, l % 4), B(l % 4, l / 4), D(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

struct LinSimtSmem { uint32_t groups, group_threads, phase_cols, off_grp, grp_bytes, bytes; };

// Shared memory: the staged rows of X, then the accumulators of every group.
inline LinSimtSmem smem_plan(const npas_bb_desc &bb)
{
    LinSimtSmem s;
    const uint32_t Bi = bb.Bi, nBi = bb.I / Bi;
    s.phase_cols = bb.I < kPhaseCols ? (uint32_t)bb.I : kPhaseCols / Bi * Bi;
    s.off_grp = round_up(kBM * (round_up(s.phase_cols, 8) + 4u) * 4u, 16);
    s.grp_bytes = (uint32_t)bb.Bo * kAccPitch * 8u;
    s.group_threads = bb.Bo > 24 ? 128u : (uint32_t)(bb.Bo + 7) / 8 * 32u;
    s.groups = kMaxWarps * 32 / s.group_threads;
    const uint32_t room = (232448u - s.off_grp) / s.grp_bytes;
    if (s.groups > kMaxGroups) s.groups = kMaxGroups;
    if (s.groups > room) s.groups = room;
    if (s.groups > nBi) s.groups = nBi;
    s.bytes = s.off_grp + s.groups * s.grp_bytes;
    return s;
}

}  // namespace

template <typename TX, typename TY>
__global__ void __launch_bounds__(kMaxWarps * 32)
linear_bb_simt_kernel(npas_linear_desc d, int Bo, int Bi, BbLayout L, LinSimtSmem S, const TX *__restrict__ x,
                      const uint8_t *__restrict__ blob, const float *__restrict__ bias, const TY *__restrict__ res,
                      TY *__restrict__ y)
{
    extern __shared__ __align__(16) uint8_t sm[];
    const int t = threadIdx.x, nt = blockDim.x, gt = (int)S.group_threads, g = t / gt, tg = t - g * gt, lane = t & 31;
    float *xraw = reinterpret_cast<float *>(sm);                                               // [kBM][pitch]
    double *acc = reinterpret_cast<double *>(sm + S.off_grp + (size_t)g * S.grp_bytes);       // [Bo][kAccPitch]

    const int bo = blockIdx.y, m0 = blockIdx.x * kBM, rows_here = min(kBM, d.M - m0), nBi = (int)L.nBi;
    const uint32_t *voff = reinterpret_cast<const uint32_t *>(blob + L.off_voff);
    const TX *vals = reinterpret_cast<const TX *>(blob + L.off_values);
    const bool x16 = sizeof(TX) == 4 && (d.I & 3) == 0 && (Bi & 3) == 0;
    const int per_phase = (int)S.phase_cols / Bi;

    tc::pdl_trigger();
    tc::pdl_wait();
    for (int e = tg; e < Bo * kAccPitch; e += gt) acc[e] = 0;
    for (int b0 = 0; b0 < nBi; b0 += per_phase) {
        const int nb = min(per_phase, nBi - b0), width = nb * Bi, pitch = (int)round_up((uint32_t)width, 8) + 4;
        if (b0) __syncthreads();                                       // the phase before has been read
        for (int r = t >> 5; r < rows_here; r += nt >> 5) {            // a warp per row
            const TX *src = x + (size_t)(m0 + r) * d.I + (size_t)b0 * Bi;
            float *dst = xraw + r * pitch;
            if (x16) for (int c = (t & 31) * 4; c < width; c += 128) cp_async16(dst + c, src + c);
            else for (int c = t & 31; c < width; c += 32) dst[c] = lin_load(src + c);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        bool waited = false;
        uint32_t off_next = 0, cnt_next = 0;                           // a block's header is fetched one block ahead
        auto fetch = [&](int b) {
            if (b >= nb) return;
            const uint32_t blk = (uint32_t)bo * L.nBi + b0 + b;
            off_next = voff[blk];
            cnt_next = *reinterpret_cast<const uint16_t *>(blob + L.off_cnt + 2 * blk);
        };
        fetch(g);
        for (int b = g; b < nb || !waited; b += S.groups) {
            const uint32_t blk = (uint32_t)bo * L.nBi + b0 + (b < nb ? b : 0);
            const int nr = b < nb ? min((int)(cnt_next & 0xFFu), Bo) : 0, nc = b < nb ? min((int)(cnt_next >> 8), Bi) : 0;
            const TX *w = vals + off_next;
            const uint8_t *rl = blob + L.off_rows + (size_t)blk * Bo, *cl = blob + L.off_cols + (size_t)blk * Bi;
            fetch(b + (int)S.groups);
            const int k = lane & 3, q = lane >> 2, col0 = b * Bi;
            for (int r0 = (tg >> 5) * 8; r0 < nr || !waited; r0 += gt / 4) {      // eight kept rows per warp
                const int r = r0 + q;
                double d[kBM / 8][2] = {};
                const int row = r < nr ? rl[r] : 0;                 // (a row or column number outside the block counts for nothing)
                for (int c0 = 0; c0 < nc || !waited; c0 += 4 * kSteps) {
                    float wv[kSteps];
                    int col[kSteps];
#pragma unroll
                    for (int i = 0; i < kSteps; ++i) {
                        const int c = c0 + 4 * i + k;
                        wv[i] = (r < nr && c < nc) ? lin_load(w + r * nc + c) : 0.f;
                        col[i] = c < nc ? (int)cl[c] : -1;
                        if (col[i] >= Bi) col[i] = -1;
                    }
                    if (!waited) {                                     // the rows of X of this phase (every thread comes here once)
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        __syncthreads();
                        waited = true;
                    }
#pragma unroll
                    for (int i = 0; i < kSteps; ++i) {
                        if (c0 + 4 * i >= nc) break;
                        const double a = (double)wv[i];
                        const float *xp = xraw + q * pitch + col0 + col[i];
#pragma unroll
                        for (int m = 0; m < kBM / 8; ++m) mma_f64(d[m], a, col[i] >= 0 ? (double)xp[m * 8 * pitch] : 0.);
                    }
                }
                if (r < nr && row < Bo) {
#pragma unroll
                    for (int m = 0; m < kBM / 8; ++m) {
                        double2 *p = reinterpret_cast<double2 *>(acc + row * kAccPitch + m * 8 + 2 * k);
                        double2 v = *p;
                        v.x += d[m][0]; v.y += d[m][1];
                        *p = v;
                    }
                }
            }
            group_sync(g, gt);         // the next block adds to other rows from other warps
        }
    }
    __syncthreads();
    // bias, residual, ReLU, one rounding; consecutive threads along the row of Y
    const double *acc0 = reinterpret_cast<const double *>(sm + S.off_grp);
    const size_t acc_step = S.grp_bytes / 8;
    const int wide = Bo > 32 ? 64 : Bo > 16 ? 32 : Bo > 8 ? 16 : 8, r = t & (wide - 1);
    if (r >= Bo) return;
    const double bv = bias ? (double)bias[bo * Bo + r] : 0.;
    const int step = nt / wide;
#pragma unroll 4
    for (int m = t / wide; m < rows_here; m += step) {
        const size_t o = (size_t)(m0 + m) * d.O + bo * Bo + r;
        double v = acc0[r * kAccPitch + m];
        for (uint32_t i = 1; i < S.groups; ++i) v += acc0[i * acc_step + r * kAccPitch + m];
        v += bv;
        if (res) v += (double)lin_load(res + o);
        if (d.relu) v = v > 0 ? v : 0;
        lin_store(y + o, (float)v);
    }
}

template <typename TX, typename TY>
static npas_status launch(const npas_linear_desc &d, const npas_bb_desc &bb, const BbLayout &L, dim3 grid, const void *x,
                          const void *blob, const float *bias, const void *res, void *y, cudaStream_t st, Launch how)
{
    const LinSimtSmem S = smem_plan(bb);
    auto k = linear_bb_simt_kernel<TX, TY>;
    if (allow_dynamic_smem(reinterpret_cast<const void *>(k), (int)S.bytes) != NPAS_OK) return NPAS_ERR_CUDA;
    const cudaError_t e = tc::launch_pdl(how, k, grid, dim3(S.group_threads * S.groups), S.bytes, st, d, (int)bb.Bo, (int)bb.Bi, L, S, static_cast<const TX *>(x),
                                         static_cast<const uint8_t *>(blob), bias, static_cast<const TY *>(res), static_cast<TY *>(y));
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
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
