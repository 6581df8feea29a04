// Block-punched convolution in float64 over the kept (channel block, tap) pairs.  This is the kernel for the float32 path
// (TF32 tensor-core products are too coarse for a 1e-5 tolerance; products of two float32 are exact in float64, so the only
// rounding is the final store) and for bf16 geometries outside the tcgen05 kernels' envelopes (odd block and channel
// counts, wide images).
//
// A CTA's eight warps are KW shares of the pairs by 8 / KW tiles of 32 consecutive output pixels, for up to 8 filters of
// one filter block: a warp multiplies the packed weights of its pairs (the A fragments of m8n8k4 float64 matrix
// instructions, read straight from the blob: with four channels per group they are its value order) with the channels
// under the tap at its 32 pixels (B fragments, read through L1 and widened), and partial sums are added in warp order
// through shared memory.  Splitting the pairs is what small layers need (their time was one thread's chain of global
// loads over all pairs: 16x16x32 -> 32 took 15.5 us on eight CTAs, 5.0 with KW = 8); with enough pixels for every SM a
// warp keeps at least eight matrix steps, because tile set-up and the final pass cost about as much.
#include "common.cuh"
#include "tc_common.cuh"

namespace npas {

namespace {

constexpr int kPixels = 32;          // output pixels per warp
constexpr int kFilters = 8;          // filters per CTA
constexpr int kWarps = 8;
constexpr int kSteps = 4;            // matrix steps whose operands are in flight together
constexpr int kMaxPairs = 1024;      // pair words staged at a time

template <typename T> __device__ inline float load_as_f32(const T *p);
template <> __device__ inline float load_as_f32<float>(const float *p) { return __ldg(p); }
template <> __device__ inline float load_as_f32<uint16_t>(const uint16_t *p) { return bf16_bits_to_f32(__ldg(p)); }

template <typename T> __device__ inline void store_from_f32(T *p, float v);
template <> __device__ inline void store_from_f32<float>(float *p, float v) { *p = v; }
template <> __device__ inline void store_from_f32<uint16_t>(uint16_t *p, float v) { *p = f32_bits_to_bf16(__float_as_uint(v)); }

// D[8 x 8] += A[8 x 4] * B[4 x 8]; lane l holds A(l / 4, l % 4), B(l % 4, l / 4), D(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void mma_f64(double (&d)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

}  // namespace

// NB: channels per block when that is 4 or 8 (the packed values are then whole matrix steps), else 0
template <typename TX, typename TY, int NB>
__global__ void __launch_bounds__(kWarps * 32)
conv_bp_simt_kernel(npas_conv_desc d, int Mb, int Nb_, int P, int Q, int KW, const TX *__restrict__ x,
                    const uint8_t *__restrict__ blob, const float *__restrict__ bias,
                    const TY *__restrict__ res, TY *__restrict__ y)
{
    __shared__ uint2 pair_s[kMaxPairs];                                   // element offset of the tap and channel block; r | s << 16
    __shared__ __align__(16) double part_s[kWarps][kFilters][kPixels + 2];

    tc::pdl_trigger();
    tc::pdl_wait();
    const int Nb = NB ? NB : Nb_;
    const uint32_t *hdr = reinterpret_cast<const uint32_t *>(blob);
    const uint32_t nCB = d.C / Nb, G = NB ? NB : (Nb % 8 == 0) ? 8 : Nb;
    const uint32_t *blk_off = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_BLK]);
    const uint32_t *pairs = reinterpret_cast<const uint32_t *>(blob + hdr[BP_OFF_PAIRS]);
    const TX *vals = reinterpret_cast<const TX *>(blob + hdr[BP_OFF_VALUES]);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = lane & 3, q8 = lane >> 2;
    const int kw = warp & (KW - 1), pt = warp / KW, fb = blockIdx.y, f0 = blockIdx.z * kFilters, nf = min(kFilters, Mb - f0);
    const long long npix = (long long)d.N * P * Q, pix0 = (long long)blockIdx.x * (kPixels * (kWarps / KW));

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
    double acc[kPixels / 8][2] = {};
    const uint32_t j_begin = blk_off[(size_t)fb * nCB], j_end = blk_off[(size_t)(fb + 1) * nCB];
    const int spp = (Nb + 3) / 4;                                        // matrix steps per pair
    for (uint32_t j0 = j_begin; j0 < j_end; j0 += kMaxPairs) {
        const int nj = (int)min((uint32_t)kMaxPairs, j_end - j0);
        if (j0 != j_begin) __syncthreads();
        for (int e = tid; e < nj; e += kWarps * 32) {
            const uint32_t pw = pairs[j0 + e], tap = pw >> 16, cb = pw & 0xFFFFu, r = tap / d.S, sx = tap - r * d.S;
            // (a pair outside the layer counts for nothing: its tap lies beside every image)
            pair_s[e] = r < (uint32_t)d.R && cb < nCB ? make_uint2((r * d.W + sx) * d.C + cb * Nb, r | (sx << 16)) : make_uint2(0u, 0xFFFFFFFFu);
        }
        __syncthreads();
        // this warp's share of the steps (contiguous, so that its sums have one order)
        const int steps = nj * spp, per = (steps + KW - 1) / KW, s_end = min(steps, (kw + 1) * per);
        const TX *wp = vals + ((size_t)j0 * (Nb / G) * Mb + f0 + q8) * G;
        for (int s0 = kw * per; s0 < s_end; s0 += kSteps) {
            float a[kSteps], b[kSteps][kPixels / 8];
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
                const int s = min(s0 + i, s_end - 1), pj = s / spp, c = (s - pj * spp) * 4 + k;
                const bool on = s0 + i < s_end && (NB || c < Nb);
                const uint2 pw = pair_s[pj];
                const int r = pw.y & 0xFFFF, sx = pw.y >> 16, c0 = c - k;
                const TX *wv = NB ? wp + (size_t)pj * Mb * NB + c : wp + ((size_t)pj * (Nb / G) + c / G) * Mb * G + c % G;
                a[i] = (on && q8 < nf) ? load_as_f32(wv) : 0.f;
#pragma unroll
                for (int m = 0; m < kPixels / 8; ++m) {
                    const bool in = on && (unsigned)(h0[m] + r) < (unsigned)d.H && (unsigned)(w0[m] + sx) < (unsigned)d.W;
                    b[i][m] = in ? load_as_f32(base[m] + (pw.x + c0)) : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < kSteps; ++i)
#pragma unroll
                for (int m = 0; m < kPixels / 8; ++m) mma_f64(acc[m], (double)a[i], (double)b[i][m]);
        }
    }
#pragma unroll
    for (int m = 0; m < kPixels / 8; ++m)
        *reinterpret_cast<double2 *>(&part_s[warp][q8][m * 8 + 2 * k]) = make_double2(acc[m][0], acc[m][1]);
    __syncthreads();
    // the shares in order, then bias, residual, ReLU, one rounding at the store
    const int f = tid & (kFilters - 1);
    if (f >= nf) return;
    const double bv = bias ? (double)bias[fb * Mb + f0 + f] : 0.;
    for (int e = tid >> 3; e < kPixels * (kWarps / KW); e += kPixels) {
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
    const long long npix = (long long)d.N * P * Q, fgroups = (long long)(bp.K / bp.Mb) * ((bp.Mb + kFilters - 1) / kFilters);
    // shares of the pairs: as many as leave a warp eight steps, more while there are not two CTAs per SM
    const int taps = bp.max_taps > 0 && bp.max_taps < d.R * d.S ? bp.max_taps : d.R * d.S;
    const long long steps = (long long)(d.C / bp.Nb) * taps * ((bp.Nb + 3) / 4);
    int KW = 1;
    while (KW < kWarps && (steps > 8 * KW || (npix * KW / (kPixels * kWarps) + 1) * fgroups < 2 * sm_count())) KW *= 2;
    const long long tile = kPixels * (kWarps / KW);
    const dim3 grid((unsigned)((npix + tile - 1) / tile), bp.K / bp.Mb, (bp.Mb + kFilters - 1) / kFilters);
    if (grid.y > 65535 || grid.z > 65535) return NPAS_ERR_UNSUPPORTED;
    auto go = [&](auto kernel) {
        return tc::launch_pdl(how, kernel, grid, dim3(kWarps * 32), 0, st, d, (int)bp.Mb, (int)bp.Nb, P, Q, KW, static_cast<const TX *>(x),
                              static_cast<const uint8_t *>(blob), bias, static_cast<const TY *>(res), static_cast<TY *>(y));
    };
    const cudaError_t e = bp.Nb == 4 ? go(conv_bp_simt_kernel<TX, TY, 4>) : bp.Nb == 8 ? go(conv_bp_simt_kernel<TX, TY, 8>) : go(conv_bp_simt_kernel<TX, TY, 0>);
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
