// C-ABI entry points that validate arguments and pick a kernel; see npas.h for the contract.
#include <vector>

#include "common.cuh"
#include "internal_api.h"
#include "tc_common.cuh"

namespace npas {

std::atomic<uint64_t> &launch_counter()
{
    static std::atomic<uint64_t> c{0};
    return c;
}

// Y[n,p,q,:] = X[n, p*stride, q*stride, :]: a block per output row and kSubUnits 16-byte units of it, a thread's copies in flight together.
// A programmatic dependent like the layers around it.  What bounds it: bytes (64x56x56x256: 51 MB, 8 us at the copy rate).  A thread per unit, with
// three 64-bit divisions for 16 bytes, behind a plain launch took 11: network of 64 images with its three of them 935 -> 925 us.
constexpr int kSubThreads = 256, kSubPer = 4, kSubUnits = kSubThreads * kSubPer;

__global__ void __launch_bounds__(kSubThreads) subsample_kernel(int H, int W, int P, int Q, int stride, int row16, const uint4 *x, uint4 *y)
{
    tc::pdl_trigger();
    const unsigned n = blockIdx.x / (unsigned)P, p = blockIdx.x - n * (unsigned)P;
    const int units = Q * row16;
    tc::pdl_wait();
    x = tc::behind_wait(x);
    const uint4 *src = x + ((size_t)n * H + (size_t)p * stride) * W * row16;
    uint4 *dst = y + (size_t)blockIdx.x * units, v[kSubPer];
    for (int u0 = (int)blockIdx.y * kSubUnits + (int)threadIdx.x; u0 < units; u0 += (int)gridDim.y * kSubUnits) {
#pragma unroll
        for (int i = 0; i < kSubPer; ++i) {
            const int u = u0 + i * kSubThreads, q = u / row16;
            if (u < units) v[i] = __ldg(src + (size_t)q * stride * row16 + (u - q * row16));
        }
#pragma unroll
        for (int i = 0; i < kSubPer; ++i)
            if (u0 + i * kSubThreads < units) dst[u0 + i * kSubThreads] = v[i];
    }
}

__global__ void maxpool_kernel(int N, int H, int W, int C, int R, int stride, int pad, int P, int Q,
                               const uint16_t *__restrict__ x, uint16_t *__restrict__ y)
{
    // one thread per (pixel, group of 8 channels): 16-byte loads and stores
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c8n = C / 8;
    const long long total = (long long)N * P * Q * c8n;
    if (idx >= total) return;
    const int c8 = (int)(idx % c8n);
    long long pix = idx / c8n;
    const int q = (int)(pix % Q); pix /= Q;
    const int p = (int)(pix % P);
    const int n = (int)(pix / P);
    float best[8];
    bool seen = false;
    for (int r = 0; r < R; ++r)
        for (int s = 0; s < R; ++s) {
            const int h = p * stride + r - pad, v = q * stride + s - pad;
            if (h < 0 || h >= H || v < 0 || v >= W) continue;
            const uint4 u = *reinterpret_cast<const uint4 *>(x + (((size_t)n * H + h) * W + v) * C + c8 * 8);
            const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xFFFF0000u);
                best[2 * i] = seen ? fmaxf(best[2 * i], lo) : lo;
                best[2 * i + 1] = seen ? fmaxf(best[2 * i + 1], hi) : hi;
            }
            seen = true;
        }
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t lo = seen ? __float_as_uint(best[2 * i]) >> 16 : 0u;
        const uint32_t hi = seen ? __float_as_uint(best[2 * i + 1]) & 0xFFFF0000u : 0u;
        o[i] = lo | hi;
    }
    *reinterpret_cast<uint4 *>(y + (((size_t)n * P + p) * Q + q) * C + c8 * 8) = make_uint4(o[0], o[1], o[2], o[3]);
}

}  // namespace npas

using namespace npas;

extern "C" {

const char *npas_status_string(npas_status s)
{
    switch (s) {
        case NPAS_OK: return "ok";
        case NPAS_ERR_NULL: return "null pointer argument";
        case NPAS_ERR_SHAPE: return "shape or block size not accepted";
        case NPAS_ERR_DTYPE: return "dtype combination not accepted";
        case NPAS_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case NPAS_ERR_MASK_STRUCTURE: return "mask is not of the pruning scheme's block structure";
        case NPAS_ERR_BLOB: return "packed blob header does not match the descriptor";
        case NPAS_ERR_BUFFER_TOO_SMALL: return "buffer too small";
        case NPAS_ERR_UNSUPPORTED: return "geometry not supported by the requested kernel";
        case NPAS_ERR_CUDA: return "CUDA runtime error";
        case NPAS_ERR_TIMEOUT: return "a bounded device-side wait expired";
    }
    return "unknown status";
}

uint32_t npas_abi_version(void) { return kAbiVersion; }
uint64_t npas_launch_count(void) { return launch_counter().load(); }

npas_status npas_conv2d_bp_workspace(const npas_conv_desc *d, const npas_bp_desc *bp, size_t *ws_bytes)
{
    if (!d || !ws_bytes) return NPAS_ERR_NULL;
    npas_status s = check_bp_desc(bp);
    if (s != NPAS_OK) return s;
    *ws_bytes = NPAS_WORKSPACE_BYTES;      // status words only: no kernel of this build needs more
    return NPAS_OK;
}

npas_status npas_linear_bb_workspace(const npas_linear_desc *d, const npas_bb_desc *bb, size_t *ws_bytes)
{
    if (!d || !ws_bytes) return NPAS_ERR_NULL;
    npas_status s = check_bb_desc(bb);
    if (s != NPAS_OK) return s;
    *ws_bytes = NPAS_WORKSPACE_BYTES;
    return NPAS_OK;
}

// Kernel ids (the values `path` takes to force one): 1 float64, 3 tcgen05 with both operands in
// shared memory, 5 three-channel first layer, 6 dense operand image, 7 the same on CTA pairs, 8 kept
// pairs only.  Returns 0 when the requested path does not take the geometry.
// Path 6 has two forms: the persistent kernel, and for few output tiles the one that splits channels and taps over a
// cluster (asked for by `variant`, or chosen when no kernel was asked for; where the pair kernel has half a wave of its
// stride-1 items, that one stays the choice).
// Path 7 likewise: the form for channels and filters off multiples of 64 and 128 is asked for by a bit of `variant`, or chosen.
struct ConvChoice { int kernel; bool split, wide; };

static ConvChoice conv_choose(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    // automatic: the first-layer kernel; kept pairs only where that was measured faster (few taps kept,
    // blocks of 16 channels or more); else the dense-image kernels; else shared-memory operands; else float64
    if (conv_stem_supported(d, bp)) return {5, false, false};
    if (conv_kr_preferred(d, bp)) return {8, false, false};
    if (conv_d2_wide_preferred(d, bp)) return {7, false, true};
    if (!(d.stride == 1 && conv_d2_preferred(d, bp)) && conv_sk_preferred(d, bp)) return {6, true, false};
    if (conv_d2_preferred(d, bp)) return {7, false, false};
    if (conv_dn_supported(d, bp)) return {6, false, false};
    if (conv_tc_supported(d, bp)) return {3, false, false};
    return {d.path == 2 ? 0 : 1, false, false};
}

// (kept per thread like the plans: several of them are compared)
static ConvChoice conv_choice(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    ConvChoice c{};
    cached_plan(d, bp, 0, c, [&](ConvChoice &q) { q = conv_choose(d, bp); return true; });
    return c;
}

static bool conv_split(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    if (d.path == 6) return d.variant != 0;
    return (d.path == 0 || d.path == 2) && conv_choice(d, bp).split;
}

static int conv_kernel_for(const npas_conv_desc &d, const npas_bp_desc &bp)
{
    switch (d.path) {
        case 1: return 1;
        case 3: return conv_tc_supported(d, bp) ? 3 : 0;
        case 5: return conv_stem_supported(d, bp) ? 5 : 0;
        case 6: return (d.variant ? conv_sk_supported(d, bp) : conv_dn_supported(d, bp)) ? 6 : 0;
        case 7: return conv_d2_supported(d, bp) ? 7 : 0;
        case 8: return conv_kr_supported(d, bp) ? 8 : 0;
        case 0: case 2: break;
        default: return 0;
    }
    return conv_choice(d, bp).kernel;
}

// Path 5 has two forms: the persistent kernel, and for few output tiles the one that splits the input over a cluster
// (asked for by the upper half of `variant`, or chosen when no kernel was asked for).
static bool linear_split_k(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    if (d.variant >> 16) return linear_sk_supported(d, bb);
    return (d.path == 0 || d.path == 2) && linear_sk_preferred(d, bb);
}

// 1 float64, 3 gathered X (kept columns only), 5 masked dense image by TMA, 6 the same on CTA pairs.
static int linear_kernel_for(const npas_linear_desc &d, const npas_bb_desc &bb)
{
    switch (d.path) {
        case 1: return 1;
        case 3: return linear_tc_supported(d, bb) ? 3 : 0;
        case 5: return (d.variant >> 16 ? linear_sk_supported(d, bb) : linear_dn_supported(d, bb)) ? 5 : 0;
        case 6: return linear_d2_supported(d, bb) ? 6 : 0;
        case 0: case 2: break;
        default: return 0;
    }
    // automatic: both operands by TMA (on CTAs or CTA pairs, whichever the model of both puts lower), then the gather
    // kernel, then float64
    if (linear_sk_preferred(d, bb)) return 5;
    // (256 or more inputs and less than a sixteenth of the chip in 128 x 128 tiles stay on pairs: there the two are within the
    // model's error of each other)
    const bool tiny = d.I >= 256 && (long long)((d.M + 127) / 128) * ((d.O + 127) / 128) * 16 < sm_count();
    if (linear_d2_supported(d, bb) && (tiny || linear_d2_cost(d, bb) < linear_dn_cost(d, bb))) return 6;
    if (linear_dn_supported(d, bb)) return 5;
    if (linear_tc_supported(d, bb)) return 3;
    return d.path == 2 ? 0 : 1;
}

static npas_status check_conv_args(const npas_conv_desc *d, const npas_bp_desc *bp)
{
    if (!d) return NPAS_ERR_NULL;
    npas_status s = check_bp_desc(bp);
    if (s != NPAS_OK) return s;
    if (d->N <= 0 || d->H <= 0 || d->W <= 0 || d->stride <= 0 || d->pad < 0) return NPAS_ERR_SHAPE;
    if (d->C != bp->C || d->K != bp->K || d->R != bp->R || d->S != bp->S) return NPAS_ERR_SHAPE;
    if (d->H + 2 * d->pad < d->R || d->W + 2 * d->pad < d->S) return NPAS_ERR_SHAPE;
    if (d->x_dtype != bp->w_packed) return NPAS_ERR_DTYPE;
    if (d->y_dtype != NPAS_F32 && d->y_dtype != NPAS_BF16) return NPAS_ERR_DTYPE;
    if (d->x_dtype == NPAS_F32 && d->y_dtype != NPAS_F32) return NPAS_ERR_DTYPE;
    return NPAS_OK;
}

static npas_status check_linear_args(const npas_linear_desc *d, const npas_bb_desc *bb)
{
    if (!d) return NPAS_ERR_NULL;
    npas_status s = check_bb_desc(bb);
    if (s != NPAS_OK) return s;
    if (d->M <= 0 || d->I != bb->I || d->O != bb->O) return NPAS_ERR_SHAPE;
    if (d->x_dtype != bb->w_packed) return NPAS_ERR_DTYPE;
    if (d->y_dtype != NPAS_F32 && d->y_dtype != NPAS_BF16) return NPAS_ERR_DTYPE;
    if (d->x_dtype == NPAS_F32 && d->y_dtype != NPAS_F32) return NPAS_ERR_DTYPE;
    return NPAS_OK;
}

npas_status npas_conv2d_bp_kernel(const npas_conv_desc *d, const npas_bp_desc *bp, int32_t *kernel_id)
{
    if (!kernel_id) return NPAS_ERR_NULL;
    npas_status s = check_conv_args(d, bp);
    if (s != NPAS_OK) return s;
    *kernel_id = conv_kernel_for(*d, *bp);
    return *kernel_id ? NPAS_OK : NPAS_ERR_UNSUPPORTED;
}

npas_status npas_linear_bb_kernel(const npas_linear_desc *d, const npas_bb_desc *bb, int32_t *kernel_id)
{
    if (!kernel_id) return NPAS_ERR_NULL;
    npas_status s = check_linear_args(d, bb);
    if (s != NPAS_OK) return s;
    *kernel_id = linear_kernel_for(*d, *bb);
    return *kernel_id ? NPAS_OK : NPAS_ERR_UNSUPPORTED;
}

// where a call of a chain stands in it -> how its kernels are launched
static Launch launch_of(int32_t chain)
{
    Launch how;
    how.plain = chain == NPAS_CHAIN_FIRST;
    how.blob_ready = chain != NPAS_CHAIN_NONE;
    return how;
}

npas_status npas_conv2d_bp(const npas_conv_desc *d, const npas_bp_desc *bp, const void *x,
                           const void *blob, const float *bias, const void *res, void *y, void *ws,
                           size_t ws_bytes, void *stream)
{
    return npas_internal_conv2d_bp(d, bp, x, blob, bias, res, y, ws, ws_bytes, NPAS_CHAIN_NONE, stream);
}

npas_status npas_internal_conv2d_bp(const npas_conv_desc *d, const npas_bp_desc *bp, const void *x,
                                    const void *blob, const float *bias, const void *res, void *y, void *ws,
                                    size_t ws_bytes, int32_t chain, void *stream)
{
    npas_status s = check_conv_args(d, bp);
    if (s != NPAS_OK) return s;
    if (!x || !blob || !y || !ws) return NPAS_ERR_NULL;
    if (d->has_bias && !bias) return NPAS_ERR_NULL;
    if (d->has_residual && !res) return NPAS_ERR_NULL;
    if (!aligned16(x) || !aligned16(blob) || !aligned16(y) || !aligned16(ws) || (bias && !aligned16(bias)) ||
        (res && !aligned16(res)))
        return NPAS_ERR_ALIGNMENT;
    if (ws_bytes < NPAS_WORKSPACE_BYTES) return NPAS_ERR_BUFFER_TOO_SMALL;
    if (x == y) return NPAS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float *b = d->has_bias ? bias : nullptr;
    const void *r = d->has_residual ? res : nullptr;
    uint32_t *w = static_cast<uint32_t *>(ws);
    const Launch how = launch_of(chain);
    switch (conv_kernel_for(*d, *bp)) {
        case 1: return conv_simt_launch(*d, *bp, x, blob, b, r, y, st, how);
        case 3: return conv_tc_launch(*d, *bp, x, blob, b, r, y, w, st);
        case 5: return conv_stem_launch(*d, *bp, x, blob, b, y, w, st, false, how);
        case 6:
            if (conv_split(*d, *bp)) return conv_sk_launch(*d, *bp, x, blob, b, r, y, w, st, how);
            return conv_dn_launch(*d, *bp, x, blob, b, r, y, w, st, how);
        case 7: return conv_d2_launch(*d, *bp, x, blob, b, r, y, w, st, how,
                                      d->path == 7 ? (d->variant & conv_d2_wide_variant()) != 0 : conv_choice(*d, *bp).wide);
        case 8: return conv_kr_launch(*d, *bp, x, blob, b, r, y, w, st, how);
    }
    return NPAS_ERR_UNSUPPORTED;
}

npas_status npas_conv2d_bp_maxpool(const npas_conv_desc *d, const npas_bp_desc *bp, int32_t pool_r, int32_t pool_stride,
                                   int32_t pool_pad, const void *x, const void *blob, const float *bias, void *y_pooled,
                                   void *ws, size_t ws_bytes, void *stream)
{
    return npas_internal_conv2d_bp_maxpool(d, bp, pool_r, pool_stride, pool_pad, x, blob, bias, y_pooled, ws, ws_bytes,
                                           NPAS_CHAIN_NONE, stream);
}

npas_status npas_internal_conv2d_bp_maxpool(const npas_conv_desc *d, const npas_bp_desc *bp, int32_t pool_r, int32_t pool_stride,
                                            int32_t pool_pad, const void *x, const void *blob, const float *bias, void *y_pooled,
                                            void *ws, size_t ws_bytes, int32_t chain, void *stream)
{
    npas_status s = check_conv_args(d, bp);
    if (s != NPAS_OK) return s;
    if (!x || !blob || !y_pooled || !ws) return NPAS_ERR_NULL;
    if (d->has_bias && !bias) return NPAS_ERR_NULL;
    if (pool_r <= 0 || pool_stride <= 0 || pool_pad < 0 || pool_pad >= pool_r) return NPAS_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(blob) || !aligned16(y_pooled) || !aligned16(ws) || (bias && !aligned16(bias)))
        return NPAS_ERR_ALIGNMENT;
    if (ws_bytes < NPAS_WORKSPACE_BYTES) return NPAS_ERR_BUFFER_TOO_SMALL;
    if (x == y_pooled) return NPAS_ERR_UNSUPPORTED;
    // fused where a kernel has the pooled epilogue: the three-channel first layer with ReLU, bf16 output and
    // the 3x3 / stride-2 / pad-1 window; everything else is left to the two separate calls
    if (d->has_residual || pool_r != 3 || pool_stride != 2 || pool_pad != 1 || (d->path != 0 && d->path != 2 && d->path != 5) ||
        !conv_stem_pool_supported(*d, *bp))
        return NPAS_ERR_UNSUPPORTED;
    return conv_stem_launch(*d, *bp, x, blob, d->has_bias ? bias : nullptr, y_pooled, static_cast<uint32_t *>(ws),
                            static_cast<cudaStream_t>(stream), true, launch_of(chain));
}

npas_status npas_linear_bb(const npas_linear_desc *d, const npas_bb_desc *bb, const void *x,
                           const void *blob, const float *bias, const void *residual, void *y, void *ws,
                           size_t ws_bytes, void *stream)
{
    return npas_internal_linear_bb(d, bb, x, blob, bias, residual, y, ws, ws_bytes, NPAS_CHAIN_NONE, stream);
}

npas_status npas_internal_linear_bb(const npas_linear_desc *d, const npas_bb_desc *bb, const void *x,
                                    const void *blob, const float *bias, const void *residual, void *y, void *ws,
                                    size_t ws_bytes, int32_t chain, void *stream)
{
    npas_status s = check_linear_args(d, bb);
    if (s != NPAS_OK) return s;
    if (!x || !blob || !y || !ws) return NPAS_ERR_NULL;
    if (d->has_bias && !bias) return NPAS_ERR_NULL;
    if (d->has_residual && !residual) return NPAS_ERR_NULL;
    if (!aligned16(x) || !aligned16(blob) || !aligned16(y) || !aligned16(ws) || (bias && !aligned16(bias)))
        return NPAS_ERR_ALIGNMENT;
    if (ws_bytes < NPAS_WORKSPACE_BYTES) return NPAS_ERR_BUFFER_TOO_SMALL;
    if (x == y) return NPAS_ERR_UNSUPPORTED;
    const void *r = d->has_residual ? residual : nullptr;
    if (r && (!aligned16(r) || r == y)) return r == y ? NPAS_ERR_UNSUPPORTED : NPAS_ERR_ALIGNMENT;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float *b = d->has_bias ? bias : nullptr;
    uint32_t *w = static_cast<uint32_t *>(ws);
    const Launch how = launch_of(chain);
    switch (linear_kernel_for(*d, *bb)) {
        case 1: return linear_simt_launch(*d, *bb, x, blob, b, r, y, st, how);
        case 3: return linear_tc_launch(*d, *bb, x, blob, b, r, y, w, st);
        case 5:
            if (linear_split_k(*d, *bb)) return linear_sk_launch(*d, *bb, x, blob, b, r, y, w, st, how);
            return linear_dn_launch(*d, *bb, x, blob, b, r, y, w, st, how);
        case 6: return linear_d2_launch(*d, *bb, x, blob, b, r, y, w, st, how);
    }
    return NPAS_ERR_UNSUPPORTED;
}

int32_t npas_internal_linear_two_preferred(const npas_linear_desc *a, const npas_linear_desc *b) { return linear_two_preferred(*a, *b); }

npas_status npas_internal_linear_two(const npas_linear_desc *a, const npas_bb_desc *bba, const npas_linear_desc *b, const npas_bb_desc *bbb,
                                     const void *x, const void *blob1, const float *bias1, const void *residual, void *y1, const void *blob2,
                                     const float *bias2, void *y2, void *ws, size_t ws_bytes, int32_t chain, void *stream)
{
    npas_status s = check_linear_args(a, bba);
    if (s == NPAS_OK) s = check_linear_args(b, bbb);
    if (s != NPAS_OK) return s;
    if (!x || !blob1 || !y1 || !blob2 || !y2 || !ws || (a->has_bias && !bias1) || (b->has_bias && !bias2) || (a->has_residual && !residual)) return NPAS_ERR_NULL;
    for (const void *q : {x, blob1, static_cast<const void *>(y1), blob2, static_cast<const void *>(y2), static_cast<const void *>(ws), residual,
                          static_cast<const void *>(bias1), static_cast<const void *>(bias2)})
        if (q && !aligned16(q)) return NPAS_ERR_ALIGNMENT;
    if (ws_bytes < NPAS_WORKSPACE_BYTES) return NPAS_ERR_BUFFER_TOO_SMALL;
    return linear_two_launch(*a, *bba, *b, *bbb, x, blob1, a->has_bias ? bias1 : nullptr, a->has_residual ? residual : nullptr, y1, blob2,
                             b->has_bias ? bias2 : nullptr, y2, static_cast<uint32_t *>(ws), static_cast<cudaStream_t>(stream), launch_of(chain));
}

}  // extern "C"

// ---- auto-tuning: measure every kernel / tile shape that takes the layer, keep the fastest --------
namespace {

struct Timer {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    bool ok = false;
    Timer() { ok = cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess; }
    ~Timer() { if (e0) cudaEventDestroy(e0); if (e1) cudaEventDestroy(e1); }
};

// Times `reps` launches of one candidate after a warm-up launch; < 0 when it declined or failed.
template <typename F>
float time_candidate(F launch, int reps, void *ws, cudaStream_t st, Timer &t)
{
    if (launch() != NPAS_OK) return -1.f;
    int32_t detail = 0;
    if (npas_check_device_status(ws, st, &detail) != NPAS_OK) return -1.f;
    cudaEventRecord(t.e0, st);
    for (int i = 0; i < reps; ++i)
        if (launch() != NPAS_OK) return -1.f;
    cudaEventRecord(t.e1, st);
    if (cudaEventSynchronize(t.e1) != cudaSuccess) return -1.f;
    if (npas_check_device_status(ws, st, &detail) != NPAS_OK) return -1.f;
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, t.e0, t.e1) != cudaSuccess) return -1.f;
    return ms * 1000.f / reps;
}

struct Cand { int path, variant; };

// The fastest of `cands`; the first is the automatic choice, written out as a forced one.  `run(c)` launches a candidate or
// declines it.  What beats the automatic choice is timed against it twice more, in turn, and has to be 3 % faster: less is within
// the noise of a measurement and of what it differs from use in (one layer's buffers, in L2 all the time), and a plan must not be
// slower than no plan.
template <typename R>
npas_status tune(const std::vector<Cand> &cands, R run, int reps, void *ws, cudaStream_t st, int32_t *path_out, int32_t *variant_out, float *us_out)
{
    Timer t;
    if (!t.ok) return NPAS_ERR_CUDA;
    auto time = [&](const Cand &c) { return time_candidate([&] { return run(c); }, reps, ws, st, t); };
    int best = -1;
    float best_us = 0.f, first_us = -1.f;
    for (size_t i = 0; i < cands.size(); ++i) {
        if (cands[i].path == 1 && i > 0 && best >= 0) continue;          // the float64 kernels only when nothing else takes the layer
        if (i > 0 && cands[i].path == cands[0].path && cands[i].variant == cands[0].variant) continue;
        const float us = time(cands[i]);
        if (us < 0.f) continue;
        if (i == 0) first_us = us;
        if (best < 0 || us < best_us) { best = (int)i; best_us = us; }
    }
    if (best < 0) return NPAS_ERR_UNSUPPORTED;
    if (best > 0 && first_us >= 0.f) {
        for (int round = 0; round < 2; ++round) {
            const float f = time(cands[0]), b = time(cands[(size_t)best]);
            if (f >= 0.f && f < first_us) first_us = f;
            if (b >= 0.f && b < best_us) best_us = b;
        }
        if (best_us > 0.97f * first_us) { best = 0; best_us = first_us; }
    }
    *path_out = cands[(size_t)best].path;
    *variant_out = cands[(size_t)best].variant;
    if (us_out) *us_out = best_us;
    return NPAS_OK;
}

}  // namespace

extern "C" {

npas_status npas_tune_conv2d_bp(const npas_conv_desc *d, const npas_bp_desc *bp, const void *x, const void *blob,
                                const float *bias, const void *res, void *y, void *ws, size_t ws_bytes,
                                int32_t reps, int32_t *path_out, int32_t *variant_out, float *us_out, void *stream)
{
    if (!path_out || !variant_out) return NPAS_ERR_NULL;
    npas_status s = check_conv_args(d, bp);
    if (s != NPAS_OK) return s;
    if (reps < 1 || reps > 10000) return NPAS_ERR_SHAPE;
    npas_conv_desc q = *d;
    q.path = 0; q.variant = 0;
    const int kid = conv_kernel_for(q, *bp);
    std::vector<Cand> cands;
    cands.push_back({kid, kid == 6 && conv_split(q, *bp) ? conv_sk_variant(q, *bp) : kid == 7 && conv_d2_wide_preferred(q, *bp) ? conv_d2_wide_variant() : 0});
    // every item shape of the pair kernel: filters per item 64, 128 or 256, position tiles per CTA 1 or 2
    for (const Cand &c : {Cand{5, 0}, Cand{8, 0}, Cand{7, 64 | (1 << 16)}, Cand{7, 64 | (2 << 16)}, Cand{7, 128 | (1 << 16)}, Cand{7, 128 | (2 << 16)},
                          Cand{7, 256 | (1 << 16)}, Cand{7, 256 | (2 << 16)}, Cand{7, conv_d2_wide_variant()}, Cand{6, 0}, Cand{3, 0}})
        cands.push_back(c);
    int32_t split[64];
    const int n = conv_sk_shapes(q, *bp, split, 64);
    for (int i = 0; i < n; ++i) cands.push_back({6, split[i]});
    cands.push_back({1, 0});
    auto run = [&](const Cand &c) {
        npas_conv_desc e = *d;
        e.path = c.path; e.variant = c.variant;
        if (!conv_kernel_for(e, *bp)) return NPAS_ERR_UNSUPPORTED;
        return npas_conv2d_bp(&e, bp, x, blob, bias, res, y, ws, ws_bytes, stream);
    };
    return tune(cands, run, reps, ws, static_cast<cudaStream_t>(stream), path_out, variant_out, us_out);
}

npas_status npas_tune_linear_bb(const npas_linear_desc *d, const npas_bb_desc *bb, const void *x, const void *blob,
                                const float *bias, const void *res, void *y, void *ws, size_t ws_bytes,
                                int32_t reps, int32_t *path_out, int32_t *variant_out, float *us_out, void *stream)
{
    if (!path_out || !variant_out) return NPAS_ERR_NULL;
    npas_status s = check_linear_args(d, bb);
    if (s != NPAS_OK) return s;
    if (reps < 1 || reps > 10000) return NPAS_ERR_SHAPE;
    npas_linear_desc q = *d;
    q.path = 0; q.variant = 0;
    const int kid = linear_kernel_for(q, *bb);
    std::vector<Cand> cands;
    cands.push_back({kid, kid == 5 && linear_split_k(q, *bb) ? linear_sk_variant(q, *bb) : 0});
    // column tiles of the two persistent kernels; column tile and CTAs per tile of the split-input form
    for (int bn : {256, 192, 128}) cands.push_back({6, bn});
    for (int bn : {256, 192, 128, 64, 32, 16}) cands.push_back({5, bn});
    for (int bn : {16, 32, 64, 128})
        for (int ks : {1, 2, 4, 8}) cands.push_back({5, bn | (ks << 16)});
    cands.push_back({3, 0});
    cands.push_back({1, 0});
    auto run = [&](const Cand &c) {
        npas_linear_desc e = *d;
        e.path = c.path; e.variant = c.variant;
        if (!linear_kernel_for(e, *bb)) return NPAS_ERR_UNSUPPORTED;
        return npas_linear_bb(&e, bb, x, blob, bias, res, y, ws, ws_bytes, stream);
    };
    return tune(cands, run, reps, ws, static_cast<cudaStream_t>(stream), path_out, variant_out, us_out);
}

// One launch or two, each on the plan its descriptor names: the faster of three measurements of either, in turn.
npas_status npas_internal_tune_linear_two(const npas_linear_desc *a, const npas_bb_desc *bba, const npas_linear_desc *b, const npas_bb_desc *bbb,
                                          const void *x, const void *blob1, const float *bias1, const void *residual, void *y1, const void *blob2,
                                          const float *bias2, void *y2, void *ws, size_t ws_bytes, int32_t reps, int32_t *together_out, float *us_out, void *stream)
{
    if (!a || !b || !together_out || !us_out) return NPAS_ERR_NULL;
    if (reps < 1 || reps > 10000) return NPAS_ERR_SHAPE;
    npas_linear_desc a0 = *a, b0 = *b;
    a0.path = a0.variant = b0.path = b0.variant = 0;
    if (!linear_two_preferred(a0, b0)) return NPAS_ERR_UNSUPPORTED;
    Timer t;
    if (!t.ok) return NPAS_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto one = [&] {
        return npas_internal_linear_two(&a0, bba, &b0, bbb, x, blob1, bias1, residual, y1, blob2, bias2, y2, ws, ws_bytes, NPAS_CHAIN_NONE, stream);
    };
    auto two = [&] {
        const npas_status s = npas_linear_bb(a, bba, x, blob1, bias1, residual, y1, ws, ws_bytes, stream);
        return s != NPAS_OK ? s : npas_linear_bb(b, bbb, y1, blob2, bias2, nullptr, y2, ws, ws_bytes, stream);
    };
    float us[2] = {-1.f, -1.f};
    for (int round = 0; round < 3; ++round)
        for (int i = 0; i < 2; ++i) {
            const float u = i ? time_candidate(one, reps, ws, st, t) : time_candidate(two, reps, ws, st, t);
            if (u >= 0.f && (us[i] < 0.f || u < us[i])) us[i] = u;
        }
    if (us[0] < 0.f && us[1] < 0.f) return NPAS_ERR_CUDA;
    *together_out = us[0] < 0.f || (us[1] >= 0.f && us[1] < us[0]);
    *us_out = us[*together_out];
    return NPAS_OK;
}

npas_status npas_blob_check(const npas_bp_desc *bp, const npas_bb_desc *bb, const void *blob,
                            size_t blob_bytes, void *stream)
{
    if (!blob || (!bp && !bb) || (bp && bb)) return NPAS_ERR_NULL;
    if (blob_bytes < 128) return NPAS_ERR_BUFFER_TOO_SMALL;
    uint32_t h[32];
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(h, blob, 128, cudaMemcpyDeviceToHost, st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (bp) {
        npas_status s = check_bp_desc(bp);
        if (s != NPAS_OK) return s;
        if (h[BP_MAGIC] != kMagicBP || h[BP_VERSION] != kVersion) return NPAS_ERR_BLOB;
        const BpLayout L = bp_layout(*bp, h[BP_NPAIRS]);
        const uint32_t want[] = {(uint32_t)bp->w_packed, (uint32_t)bp->K, (uint32_t)bp->C, (uint32_t)bp->R,
                                 (uint32_t)bp->S, (uint32_t)bp->Mb, (uint32_t)bp->Nb, L.nFB, L.nCB, h[BP_NPAIRS],
                                 L.off_blk, L.off_pairs, L.off_values, L.total, L.G, L.off_image, L.off_tapu, L.GI,
                                 L.off_ktoff, L.off_kt, L.GS, L.nKt};
        for (int i = 0; i < 22; ++i)
            if (h[BP_DTYPE + i] != want[i]) return NPAS_ERR_BLOB;
        if (h[BP_NPAIRS] > L.nFB * L.nCB * (uint32_t)(bp->R * bp->S)) return NPAS_ERR_BLOB;
        return L.total <= blob_bytes ? NPAS_OK : NPAS_ERR_BUFFER_TOO_SMALL;
    }
    npas_status s = check_bb_desc(bb);
    if (s != NPAS_OK) return s;
    if (h[BB_MAGIC] != kMagicBB || h[BB_VERSION] != kVersionBB) return NPAS_ERR_BLOB;
    const BbLayout L = bb_layout(*bb);
    const uint32_t off_tiles = L.off_values + round_up(h[BB_NVALS] * L.es, 128);
    if (h[BB_KP] < 16 || h[BB_KP] % 16 || h[BB_KP] > 64 || h[BB_OFF_TILES] != off_tiles) return NPAS_ERR_BLOB;
    const uint32_t total = off_tiles + round_up(L.nBlk * h[BB_KP] * (uint32_t)bb->Bo * L.es, 128);
    const uint32_t want[] = {(uint32_t)bb->w_packed, (uint32_t)bb->O, (uint32_t)bb->I, (uint32_t)bb->Bo,
                             (uint32_t)bb->Bi, L.nBo, L.nBi, h[BB_NVALS], L.off_cnt, L.off_rows, L.off_cols,
                             L.off_voff, L.off_values, total};
    for (int i = 0; i < 14; ++i)
        if (h[BB_DTYPE + i] != want[i]) return NPAS_ERR_BLOB;
    if (h[BB_OFF_DENSE] != L.off_dense) return NPAS_ERR_BLOB;
    return total <= blob_bytes ? NPAS_OK : NPAS_ERR_BUFFER_TOO_SMALL;
}

npas_status npas_check_device_status(void *ws, void *stream, int32_t *detail)
{
    if (!ws) return NPAS_ERR_NULL;
    uint32_t w[2] = {0, 0};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(w, ws, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (detail) *detail = (int32_t)w[WS_DETAIL];
    if (w[WS_STATUS] == 0) return NPAS_OK;
    if (cudaMemsetAsync(ws, 0, 8, st) != cudaSuccess) return NPAS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return NPAS_ERR_CUDA;
    return w[WS_STATUS] == (uint32_t)NPAS_ERR_BLOB ? NPAS_ERR_BLOB : NPAS_ERR_TIMEOUT;
}

npas_status npas_maxpool2d(int32_t N, int32_t H, int32_t W, int32_t C, int32_t R, int32_t stride,
                           int32_t pad, const void *x, void *y, void *stream)
{
    if (!x || !y) return NPAS_ERR_NULL;
    if (N <= 0 || H <= 0 || W <= 0 || C <= 0 || C % 8 || R <= 0 || stride <= 0 || pad < 0 || pad >= R)
        return NPAS_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(y)) return NPAS_ERR_ALIGNMENT;
    const int P = (H + 2 * pad - R) / stride + 1, Q = (W + 2 * pad - R) / stride + 1;
    const long long total = (long long)N * P * Q * (C / 8);
    maxpool_kernel<<<(unsigned)((total + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        N, H, W, C, R, stride, pad, P, Q, static_cast<const uint16_t *>(x), static_cast<uint16_t *>(y));
    count_launch();
    return launch_status();
}

npas_status npas_subsample2d(int32_t N, int32_t H, int32_t W, int32_t C, int32_t stride,
                             int32_t elem_bytes, const void *x, void *y, void *stream)
{
    if (!x || !y) return NPAS_ERR_NULL;
    if (N <= 0 || H <= 0 || W <= 0 || C <= 0 || stride <= 0) return NPAS_ERR_SHAPE;
    if (elem_bytes != 2 && elem_bytes != 4) return NPAS_ERR_DTYPE;
    if (((long long)C * elem_bytes) % 16) return NPAS_ERR_SHAPE;
    if (!aligned16(x) || !aligned16(y)) return NPAS_ERR_ALIGNMENT;
    if (x == y) return NPAS_ERR_UNSUPPORTED;
    const int P = (H - 1) / stride + 1, Q = (W - 1) / stride + 1, row16 = C * elem_bytes / 16;
    const long long lines = (long long)N * P, units = (long long)Q * row16;
    if (lines > 0x7FFFFFFF || units > 0x3FFFFFFF) return NPAS_ERR_SHAPE;
    const long long parts = (units + kSubUnits - 1) / kSubUnits;
    const cudaError_t e = tc::launch_pdl(Launch{}, subsample_kernel, dim3((unsigned)lines, (unsigned)(parts < 65535 ? parts : 65535)), dim3(kSubThreads), 0,
                                         static_cast<cudaStream_t>(stream), H, W, P, Q, stride, row16, static_cast<const uint4 *>(x), static_cast<uint4 *>(y));
    count_launch();
    return e == cudaSuccess ? launch_status() : NPAS_ERR_CUDA;
}

}  // extern "C"
