// Block-punched convolution in float64 over the kept (channel block, tap) pairs.  This is the kernel for the float32 path
// (TF32 tensor-core products are too coarse for a 1e-5 tolerance; products of two float32 are exact in float64, so the only
// rounding is the final store) and for bf16 geometries outside the tcgen05 kernels' envelopes (odd block and channel
// counts, wide images).
//
// A CTA's eight warps are KW shares of the pairs by 8 / KW tiles of 32 consecutive output pixels, for 8 or 16 filters of
// one filter block: a warp multiplies the packed weights of its pairs (the A fragments of m8n8k4 float64 matrix
// instructions, read straight from the blob) with the channels under the tap at its 32 pixels (B fragments, read through L1
// and widened), and partial sums are added in warp order through shared memory.  What a step of four channels reads is
// described in shared memory once per CTA: offsets in X and in the values, the tap, the channels.
//
// What bounds it: small layers the chain of loads over a warp's pairs (16x16x32 -> 32: 15.5 us as one thread's chain on eight
// CTAs, 4.6 with KW = 8), large ones the instructions around the loads of X: with sixteen filters per load and one share
// per tile 8x56x200x128 -> 128 (three of nine taps) takes 444 us in float32 and 490 in bf16 (1171 and 1150 with eight filters
// and shares of eight steps, 1305 and 1029 on FMAs; the float64 pipe alone would take 236).
#include <type_traits>

#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

namespace {

constexpr int kPixels = 32;          // output pixels per warp
constexpr int kWarps = 8;
constexpr int kSteps = 4;            // matrix steps whose operands are in flight together
constexpr int kMaxSteps = 768;       // matrix steps (four channels of a pair) described at a time

template <typename T> __device__ inline float load_as_f32(const T *p);
template <> __device__ inline float load_as_f32<float>(const float *p) { return __ldg(p); }
template <> __device__ inline float load_as_f32<uint16_t>(const uint16_t *p) { return bf16_bits_to_f32(__ldg(p)); }

// Where a filter block's pairs begin or end.  Both forms read through the pointer the kernel was given, at an offset known behind the
// wait only, and differ in nothing but where the compiler then places the kernel's loads: float32 layers are 2 to 4 % slower with __ldg
// (32x56x56x20 -> 32 60.4 us against 57.9, 16x28x28x64 -> 64 with a residual 41.4 against 37.6), bf16 ones 0 to 6 % without
// (16x14x14x36 -> 36 13.0 against 12.3).
template <typename TX> __device__ __forceinline__ uint32_t pair_bound(const uint32_t *p)
{
    if constexpr (sizeof(TX) == 2) return __ldg(p);
    else return *p;
}

template <typename T> __device__ inline void store_from_f32(T *p, float v);
template <> __device__ inline void store_from_f32<float>(float *p, float v) { *p = v; }
template <> __device__ inline void store_from_f32<uint16_t>(uint16_t *p, float v) { *p = f32_bits_to_bf16(__float_as_uint(v)); }

// D[8 x 8] += A[8 x 4] * B[4 x 8]; lane l holds A(l / 4, l % 4), B(l % 4, l / 4), D(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

}  // namespace

// NB: channels per block when that is 4 or 8 (divisions become shifts), else 0; FG: filters per CTA, in eights
template <typename TX, typename TY, int NB, int FG>
__global__ void __launch_bounds__(kWarps * 32)
conv_bp_simt_kernel(npas_conv_desc d, int Mb, int Nb_, int P, int Q, int KW, const TX *__restrict__ x,
                    const uint8_t *__restrict__ blob, const float *__restrict__ bias,
                    const TY *__restrict__ res, TY *__restrict__ y)
{
    constexpr int kFilters = 8 * FG;
    const int Nb = NB ? NB : Nb_;
    // element offset of the tap and the step's first channel in X; r | s << 16; offset in the values; channels of the step
    __shared__ uint4 step_s[kMaxSteps];
    __shared__ __align__(16) double part_s[kWarps][kFilters][kPixels + 2];

    tc::pdl_trigger();
    tc::pdl_wait();
    const int z = tc::zero_behind_wait();                                    // in the header's address, the bias', and every pixel number
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob) + z;      // (lists and values lie at offsets that it holds)
    const uint32_t nCB = d.C / Nb, G = NB ? NB : (Nb % 8 == 0) ? 8 : Nb;
    const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_BLK]);
    const uint32_t *pairs = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
    const TX *vals = reinterpret_cast<const TX *>(blob + hdr[BP_OFF_VALUES]);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = lane & 3, q8 = lane >> 2;
    const int kw = warp & (KW - 1), pt = warp / KW, fb = blockIdx.y, f0 = blockIdx.z * kFilters, nf = min(kFilters, Mb - f0);
    const long long npix = (long long)d.N * P * Q, pix0 = (long long)blockIdx.x * (kPixels * (kWarps / KW)) + z;

    // this lane's four pixels (one of every group of eight): top-left input position and where it lies
    int h0[kPixels / 8], w0[kPixels / 8];
    const TX *base[kPixels / 8];
#pragma unroll
    for (int m = 0; m < kPixels / 8; ++m) {
        const long long pix = pix0 + pt * kPixels + m * 8 + q8;
        h0[m] = -(1 << 29); w0[m] = 0; base[m] = x;                      // past the end: never inside the image
        if (pix < npix) {
            const int n = (int)(pix / (P * Q)), rem = (int)(pix - (long long)n * (P * Q)), p = rem / Q;
            h0[m] = p * d.stride - d.pad; w0[m] = (rem - p * Q) * d.stride - d.pad;
            base[m] = x + (((long long)n * d.H + h0[m]) * d.W + w0[m]) * d.C + k;
        }
    }
    double acc[FG][kPixels / 8][2] = {};
    const uint32_t j_begin = pair_bound<TX>(blk_off + (size_t)fb * nCB), j_end = pair_bound<TX>(blk_off + (size_t)(fb + 1) * nCB);
    const uint32_t spp = (Nb + 3) / 4;                                   // matrix steps per pair
    const uint32_t s_all = (j_end - j_begin) * spp;
    const TX *wp = vals + ((size_t)j_begin * Nb * Mb + (f0 + q8) * G + k);
    for (uint32_t b0 = 0; b0 < s_all; b0 += kMaxSteps) {
        const int steps = (int)min((uint32_t)kMaxSteps, s_all - b0);
        if (b0) __syncthreads();
        for (int e = tid; e < steps; e += kWarps * 32) {
            const uint32_t j = (b0 + e) / spp, c0 = (b0 + e - j * spp) * 4, pw = pairs[j_begin + j], tap = pw >> 16, cb = pw & 0xFFFFu;
            const uint32_t r = tap / d.S, sx = tap - r * d.S, wo = (j * (Nb / G) + c0 / G) * Mb * G + c0 % G;
            // (a pair outside the layer counts for nothing: its tap lies beside every image)
            step_s[e] = r < (uint32_t)d.R && cb < nCB ? make_uint4((r * d.W + sx) * d.C + cb * Nb + c0, r | (sx << 16), wo, Nb - c0)
                                                      : make_uint4(0u, 0xFFFFFFFFu, wo, Nb - c0);
        }
        __syncthreads();
        // this warp's share of the steps (contiguous, so that its sums have one order)
        const int per = (steps + KW - 1) / KW, s_end = min(steps, (kw + 1) * per);
        for (int s0 = kw * per; s0 < s_end; s0 += kSteps) {
            float a[kSteps][FG], b[kSteps][kPixels / 8];
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
                const uint4 st = step_s[min(s0 + i, s_end - 1)];
                const bool on = s0 + i < s_end && k < (int)st.w;
                const int r = st.y & 0xFFFF, sx = st.y >> 16;
#pragma unroll
                for (int g = 0; g < FG; ++g) a[i][g] = (on && q8 + 8 * g < nf) ? load_as_f32(wp + st.z + 8 * g * G) : 0.f;
#pragma unroll
                for (int m = 0; m < kPixels / 8; ++m) {
                    const bool in = on && (unsigned)(h0[m] + r) < (unsigned)d.H && (unsigned)(w0[m] + sx) < (unsigned)d.W;
                    b[i][m] = in ? load_as_f32(base[m] + st.x) : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < kSteps; ++i)
#pragma unroll
                for (int m = 0; m < kPixels / 8; ++m) {
                    const double bv = (double)b[i][m];
#pragma unroll
                    for (int g = 0; g < FG; ++g) mma_f64(acc[g][m], (double)a[i][g], bv);
                }
        }
    }
#pragma unroll
    for (int g = 0; g < FG; ++g)
#pragma unroll
        for (int m = 0; m < kPixels / 8; ++m)
            *reinterpret_cast<double2 *>(&part_s[warp][g * 8 + q8][m * 8 + 2 * k]) = make_double2(acc[g][m][0], acc[g][m][1]);
    __syncthreads();
    // the shares in order, then bias, residual, ReLU, one rounding at the store
    const int f = tid & (kFilters - 1);
    if (f >= nf) return;
    const double bv = bias ? (double)bias[fb * Mb + f0 + f + z] : 0.;
    for (int e = tid / kFilters; e < kPixels * (kWarps / KW); e += kWarps * 32 / kFilters) {
        const long long pix = pix0 + e;
        if (pix >= npix) return;
        const int m = e & (kPixels - 1), t0 = e / kPixels * KW;
        double v = part_s[t0][f][m];
        for (int w = 1; w < KW; ++w) v += part_s[t0 + w][f][m];
        const size_t o = (size_t)pix * d.K + fb * Mb + f0 + f;
        v += bv;
        if (res) v += (double)load_as_f32(res + o);
        if (d.relu) v = v > 0 ? v : 0;
        store_from_f32(y + o, (float)v);
    }
}

template <typename TX, typename TY>
static npas_status launch(const npas_conv_desc &d, const npas_bp_desc &bp, int P, int Q, const void *x, const void *blob,
                          const float *bias, const void *res, void *y, cudaStream_t st, Launch how)
{
    const long long npix = (long long)d.N * P * Q;
    auto groups = [&](int filters) { return (long long)(bp.K / bp.Mb) * ((bp.Mb + filters - 1) / filters); };
    // sixteen filters per CTA share a pixel's loads and set-up, where that leaves four CTAs per SM (16x112x112x3 -> 64, nine taps:
    // 117 us, with eight 167; 56x56x20 -> 32 of four images, too few CTAs, stays with eight)
    const bool wide = bp.Mb > 8 && (npix + kPixels * kWarps - 1) / (kPixels * kWarps) * groups(16) >= 4ll * sm_count();
    const int filters = wide ? 16 : 8;
    const long long fgroups = groups(filters);
    const int taps = bp.max_taps > 0 && bp.max_taps < d.R * d.S ? bp.max_taps : d.R * d.S;
    const long long steps = (long long)(d.C / bp.Nb) * taps * ((bp.Nb + 3) / 4);
    // Shares of the pairs: one while there are enough CTAs without (five for four SMs), two to eight where there are not, and up to
    // four CTAs per SM as long as a warp keeps 64 steps.  Set-up and the sum over the shares are paid per 32 pixels and share:
    // shares of eight steps whatever the grid took 254 us for 32x28x28x68 -> 68 (4x4 blocks, three taps), one share takes 136;
    // 28x28x36 -> 60 of two images 13.4 with two, 9.8 with four and 14 with eight; 2x14x14x64 -> 64, where only shares fill the
    // chip, 21 with one and 6.8 with eight.
    auto ctas = [&](int kw) { return (npix * kw + kPixels * kWarps - 1) / (kPixels * kWarps) * fgroups; };
    int KW = 1;
    while (KW < kWarps && (ctas(KW) * 4 < 5ll * sm_count() || (steps >= 64 * KW && ctas(KW) < 4ll * sm_count()))) KW *= 2;
    const long long tile = kPixels * (kWarps / KW);
    const dim3 grid((unsigned)((npix + tile - 1) / tile), bp.K / bp.Mb, (bp.Mb + filters - 1) / filters);
    if (grid.y > 65535 || grid.z > 65535) return NPAS_ERR_UNSUPPORTED;
    auto go = [&](auto kernel) {
        return tc::launch_pdl(how, kernel, grid, dim3(kWarps * 32), 0, st, d, (int)bp.Mb, (int)bp.Nb, P, Q, KW, static_cast<const TX *>(x),
                              static_cast<const uint8_t *>(blob), bias, static_cast<const TY *>(res), static_cast<TY *>(y));
    };
    auto width = [&](auto nb) {
        constexpr int NB = decltype(nb)::value;
        return wide ? go(conv_bp_simt_kernel<TX, TY, NB, 2>) : go(conv_bp_simt_kernel<TX, TY, NB, 1>);
    };
    using std::integral_constant;
    auto blocks = [&]() {
        // (float32 only: bf16 layers, whose loads are half as wide, are 5 to 15 % faster without)
        if constexpr (sizeof(TX) == 4) {
            if (bp.Nb == 4) return width(integral_constant<int, 4>{});
            if (bp.Nb == 8) return width(integral_constant<int, 8>{});
        }
        return width(integral_constant<int, 0>{});
    };
    const cudaError_t e = blocks();
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

npas_status conv_simt_launch(const npas_conv_desc &d, const npas_bp_desc &bp, const void *x,
                             const void *blob, const float *bias, const void *res, void *y,
                             cudaStream_t st, Launch how)
{
    const int P = (d.H + 2 * d.pad - d.R) / d.stride + 1, Q = (d.W + 2 * d.pad - d.S) / d.stride + 1;
    if (d.x_dtype == NPAS_F32 && d.y_dtype == NPAS_F32) return launch<float, float>(d, bp, P, Q, x, blob, bias, res, y, st, how);
    if (d.x_dtype == NPAS_BF16 && d.y_dtype == NPAS_BF16) return launch<uint16_t, uint16_t>(d, bp, P, Q, x, blob, bias, res, y, st, how);
    if (d.x_dtype == NPAS_BF16 && d.y_dtype == NPAS_F32) return launch<uint16_t, float>(d, bp, P, Q, x, blob, bias, res, y, st, how);
    return NPAS_ERR_DTYPE;
}

}  // namespace npas
