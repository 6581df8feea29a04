// The compute calls of the Python binding, in native code: argument checks, descriptors, the output tensor, the
// current stream and the library call, without a Python-level step in between.
//
// A call through ctypes spent 14 us of host time (descriptor objects, pointer wrappers, stream lookup, and torch's
// own Python entry for the output tensor), more than most layers take on the GPU.  This file is an ordinary CPython
// extension that links against libnpas.so; binding.py keeps the public functions, with their arguments, defaults
// and errors, and hands their arguments over positionally.  A compute function returns the output tensor, or the
// npas_status as an int when the library refused the call (binding.py raises).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/cuda/EmptyTensor.h>
#include <ATen/ops/empty.h>
#include <ATen/ops/zeros.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/autograd/python_variable.h>

#include <atomic>
#include <cmath>
#include <mutex>
#include <vector>

#include "npas.h"
#include "internal_api.h"

namespace {

bool fail_assert(const char *what)
{
    PyErr_SetString(PyExc_AssertionError, what);
    return false;
}

// A tensor argument (None allowed where `optional`); the reference stays borrowed from the argument.
bool tensor_arg(PyObject *o, const at::Tensor *&t, bool optional, const char *name)
{
    t = nullptr;
    if (optional && o == Py_None) return true;
    if (!THPVariable_Check(o)) { PyErr_Format(PyExc_TypeError, "%s must be a torch.Tensor", name); return false; }
    t = &THPVariable_Unpack(o);
    return true;
}

bool int_arg(PyObject *o, int32_t &v)
{
    const long l = PyLong_AsLong(o);
    if (l == -1 && PyErr_Occurred()) return false;
    v = (int32_t)l;
    return true;
}

bool dtype_of(at::ScalarType t, int32_t &code)
{
    if (t == at::kFloat) { code = NPAS_F32; return true; }
    if (t == at::kBFloat16) { code = NPAS_BF16; return true; }
    PyErr_Format(PyExc_TypeError, "unsupported dtype %s", c10::toString(t));
    return false;
}

bool dtype_arg(PyObject *o, at::ScalarType otherwise, at::ScalarType &t)
{
    if (o == Py_None) { t = otherwise; return true; }
    if (!THPDtype_Check(o)) { PyErr_SetString(PyExc_TypeError, "out_dtype must be a torch.dtype"); return false; }
    t = reinterpret_cast<THPDtype *>(o)->scalar_type;
    return true;
}

// The descriptor structures are ctypes objects that the caller may have changed: read through the buffer protocol.
template <typename D>
bool desc_arg(PyObject *o, D &d)
{
    Py_buffer view;
    if (PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) return false;
    const bool ok = view.len == (Py_ssize_t)sizeof(D);
    if (ok) memcpy(&d, view.buf, sizeof(D));
    PyBuffer_Release(&view);
    if (!ok) PyErr_SetString(PyExc_TypeError, "descriptor of the wrong type");
    return ok;
}

void *ptr(const at::Tensor *t) { return t ? t->data_ptr() : nullptr; }

at::Tensor new_tensor(at::IntArrayRef size, at::ScalarType t, const at::Device &dev)
{
    return at::Tensor(at::detail::empty_cuda(size, t, dev, std::nullopt));
}

// Status words for calls that bring no workspace: nobody can read them afterwards, so all such calls on a device share
// one buffer, kept for the life of the process (a zeroed allocation per call cost a launch).  A call inside a stream
// capture that finds none yet gets one of its own.
bool shared_workspace(const at::Device &dev, at::Tensor &own, void *&p)
{
    constexpr int kMaxDevices = 64;
    static std::atomic<void *> kept[kMaxDevices];
    static std::mutex mu;
    const int i = dev.index();
    if (i >= 0 && i < kMaxDevices && (p = kept[i].load(std::memory_order_acquire)) != nullptr) return true;
    const auto opt = at::TensorOptions().dtype(at::kByte).device(dev);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(c10::cuda::getCurrentCUDAStream().stream(), &cap);
    if (cap != cudaStreamCaptureStatusNone || i < 0 || i >= kMaxDevices) {
        own = at::zeros({NPAS_WORKSPACE_BYTES}, opt);
        p = own.data_ptr();
        return true;
    }
    std::lock_guard<std::mutex> lock(mu);
    if ((p = kept[i].load(std::memory_order_acquire)) == nullptr) {
        auto *t = new at::Tensor(at::zeros({NPAS_WORKSPACE_BYTES}, opt));      // (never freed: it lives as long as the process)
        cudaStreamSynchronize(c10::cuda::getCurrentCUDAStream().stream());     // other streams may use it from here on
        p = t->data_ptr();
        kept[i].store(p, std::memory_order_release);
    }
    return true;
}

bool workspace_arg(const at::Tensor *ws, const at::Tensor &x, at::Tensor &own, void *&p, size_t &bytes)
{
    if (ws) { p = ws->data_ptr(); bytes = (size_t)ws->numel(); return true; }
    bytes = NPAS_WORKSPACE_BYTES;
    return shared_workspace(x.device(), own, p);
}

PyObject *result(npas_status s, PyObject *out_given, at::Tensor &&made)
{
    if (s != NPAS_OK) return PyLong_FromLong((long)s);
    if (out_given) { Py_INCREF(out_given); return out_given; }
    return THPVariable_Wrap(std::move(made));
}

template <typename F>
PyObject *guarded(F f)
{
    try {
        return f();
    } catch (const std::exception &e) {
        if (!PyErr_Occurred()) PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

// conv2d_bp(x, blob, desc, bias, residual, stride, pad, relu, out_dtype, out, ws, path, variant)
PyObject *conv2d_bp(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *x, *blob, *bias, *res, *out, *ws;
        npas_bp_desc bp;
        npas_conv_desc d = {};
        at::ScalarType ot;
        if (n != 13) { PyErr_SetString(PyExc_TypeError, "conv2d_bp takes 13 arguments"); return nullptr; }
        if (!tensor_arg(a[0], x, false, "x") || !tensor_arg(a[1], blob, false, "blob.data") || !desc_arg(a[2], bp) ||
            !tensor_arg(a[3], bias, true, "bias") || !tensor_arg(a[4], res, true, "residual") || !int_arg(a[5], d.stride) ||
            !int_arg(a[6], d.pad) || !tensor_arg(a[9], out, true, "out") || !tensor_arg(a[10], ws, true, "ws") ||
            !int_arg(a[11], d.path) || !int_arg(a[12], d.variant))
            return nullptr;
        const int relu = PyObject_IsTrue(a[7]);
        if (relu < 0) return nullptr;
        if (!(x->is_cuda() && x->is_contiguous() && x->dim() == 4)) { fail_assert("x must be a contiguous 4-D CUDA tensor"); return nullptr; }
        if (!dtype_arg(a[8], x->scalar_type(), ot)) return nullptr;
        if (d.stride == 0) { PyErr_SetString(PyExc_ZeroDivisionError, "stride is zero"); return nullptr; }
        d.N = (int32_t)x->size(0); d.H = (int32_t)x->size(1); d.W = (int32_t)x->size(2); d.C = (int32_t)x->size(3);
        d.K = bp.K; d.R = bp.R; d.S = bp.S;
        d.relu = relu; d.has_bias = bias != nullptr; d.has_residual = res != nullptr;
        auto positions = [&](int64_t in, int64_t taps) {      // floor division, as the shape of the output tensor
            const int64_t v = in + 2 * (int64_t)d.pad - taps, q = v / d.stride;
            return q - ((v % d.stride != 0) && ((v < 0) != (d.stride < 0)) ? 1 : 0) + 1;
        };
        at::Tensor made, own;
        if (!out) made = new_tensor({x->size(0), positions(x->size(1), bp.R), positions(x->size(2), bp.S), bp.K}, ot, x->device());
        if (!dtype_of(x->scalar_type(), d.x_dtype) || !dtype_of(out ? out->scalar_type() : ot, d.y_dtype)) return nullptr;
        void *w = nullptr, *y = out ? out->data_ptr() : made.data_ptr();
        size_t wb = 0;
        if (!workspace_arg(ws, *x, own, w, wb)) return nullptr;
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        npas_status s;
        Py_BEGIN_ALLOW_THREADS
        s = npas_conv2d_bp(&d, &bp, x->data_ptr(), blob->data_ptr(), static_cast<const float *>(ptr(bias)), ptr(res), y, w, wb, st);
        Py_END_ALLOW_THREADS
        return result(s, out ? a[9] : nullptr, std::move(made));
    });
}

// conv2d_bp_maxpool(x, blob, desc, bias, stride, pad, relu, pool_r, pool_stride, pool_pad, out, ws, path)
PyObject *conv2d_bp_maxpool(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *x, *blob, *bias, *out, *ws;
        npas_bp_desc bp;
        npas_conv_desc d = {};
        int32_t pr, ps, pp;
        if (n != 13) { PyErr_SetString(PyExc_TypeError, "conv2d_bp_maxpool takes 13 arguments"); return nullptr; }
        if (!tensor_arg(a[0], x, false, "x") || !tensor_arg(a[1], blob, false, "blob.data") || !desc_arg(a[2], bp) ||
            !tensor_arg(a[3], bias, true, "bias") || !int_arg(a[4], d.stride) || !int_arg(a[5], d.pad) || !int_arg(a[7], pr) ||
            !int_arg(a[8], ps) || !int_arg(a[9], pp) || !tensor_arg(a[10], out, true, "out") || !tensor_arg(a[11], ws, true, "ws") ||
            !int_arg(a[12], d.path))
            return nullptr;
        const int relu = PyObject_IsTrue(a[6]);
        if (relu < 0) return nullptr;
        if (!(x->is_cuda() && x->is_contiguous() && x->dim() == 4)) { fail_assert("x must be a contiguous 4-D CUDA tensor"); return nullptr; }
        if (d.stride == 0 || ps == 0) { PyErr_SetString(PyExc_ZeroDivisionError, "stride is zero"); return nullptr; }
        d.N = (int32_t)x->size(0); d.H = (int32_t)x->size(1); d.W = (int32_t)x->size(2); d.C = (int32_t)x->size(3);
        d.K = bp.K; d.R = bp.R; d.S = bp.S;
        d.relu = relu; d.has_bias = bias != nullptr;
        auto floor_div = [](int64_t v, int64_t q) { return v / q - ((v % q != 0) && ((v < 0) != (q < 0)) ? 1 : 0); };
        const int64_t P = floor_div(x->size(1) + 2 * d.pad - bp.R, d.stride) + 1, Q = floor_div(x->size(2) + 2 * d.pad - bp.S, d.stride) + 1;
        at::Tensor made, own;
        if (!out) made = new_tensor({x->size(0), floor_div(P + 2 * pp - pr, ps) + 1, floor_div(Q + 2 * pp - pr, ps) + 1, bp.K}, x->scalar_type(), x->device());
        if (!dtype_of(x->scalar_type(), d.x_dtype) || !dtype_of(out ? out->scalar_type() : x->scalar_type(), d.y_dtype)) return nullptr;
        void *w = nullptr, *y = out ? out->data_ptr() : made.data_ptr();
        size_t wb = 0;
        if (!workspace_arg(ws, *x, own, w, wb)) return nullptr;
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        npas_status s;
        Py_BEGIN_ALLOW_THREADS
        s = npas_conv2d_bp_maxpool(&d, &bp, pr, ps, pp, x->data_ptr(), blob->data_ptr(), static_cast<const float *>(ptr(bias)), y, w, wb, st);
        Py_END_ALLOW_THREADS
        return result(s, out ? a[10] : nullptr, std::move(made));
    });
}

// linear_bb(x, blob, desc, bias, residual, relu, out_dtype, out, ws, path, variant)
PyObject *linear_bb(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *x, *blob, *bias, *res, *out, *ws;
        npas_bb_desc bb;
        npas_linear_desc d = {};
        at::ScalarType ot;
        if (n != 11) { PyErr_SetString(PyExc_TypeError, "linear_bb takes 11 arguments"); return nullptr; }
        if (!tensor_arg(a[0], x, false, "x") || !tensor_arg(a[1], blob, false, "blob.data") || !desc_arg(a[2], bb) ||
            !tensor_arg(a[3], bias, true, "bias") || !tensor_arg(a[4], res, true, "residual") || !tensor_arg(a[7], out, true, "out") ||
            !tensor_arg(a[8], ws, true, "ws") || !int_arg(a[9], d.path) || !int_arg(a[10], d.variant))
            return nullptr;
        const int relu = PyObject_IsTrue(a[5]);
        if (relu < 0) return nullptr;
        if (!(x->is_cuda() && x->is_contiguous() && x->dim() == 2)) { fail_assert("x must be a contiguous 2-D CUDA tensor"); return nullptr; }
        if (!dtype_arg(a[6], x->scalar_type(), ot)) return nullptr;
        at::Tensor made, own;
        if (!out) made = new_tensor({x->size(0), bb.O}, ot, x->device());
        const at::Tensor &y = out ? *out : made;
        if (res && !(res->is_cuda() && res->is_contiguous() && res->sizes() == y.sizes() && res->scalar_type() == y.scalar_type())) {
            fail_assert("residual must be a contiguous CUDA tensor of the output's shape and dtype");
            return nullptr;
        }
        d.M = (int32_t)x->size(0); d.I = (int32_t)x->size(1); d.O = bb.O;
        if (!dtype_of(x->scalar_type(), d.x_dtype) || !dtype_of(y.scalar_type(), d.y_dtype)) return nullptr;
        d.relu = relu; d.has_bias = bias != nullptr; d.has_residual = res != nullptr;
        void *w = nullptr, *yp = y.data_ptr();
        size_t wb = 0;
        if (!workspace_arg(ws, *x, own, w, wb)) return nullptr;
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        npas_status s;
        Py_BEGIN_ALLOW_THREADS
        s = npas_linear_bb(&d, &bb, x->data_ptr(), blob->data_ptr(), static_cast<const float *>(ptr(bias)), ptr(res), yp, w, wb, st);
        Py_END_ALLOW_THREADS
        return result(s, out ? a[7] : nullptr, std::move(made));
    });
}

// ---- packing and pruning ------------------------------------------------------------------------------------------

// The sums a blob's size follows from.  Kept bits per mask word below `live`.
struct MaskSums { uint64_t total; uint32_t most; };
__attribute__((target_clones("popcnt", "default"))) MaskSums count_bits(const uint64_t *m, size_t n, uint64_t live)
{
    MaskSums s{0, 0};
    for (size_t i = 0; i < n; ++i) {
        const uint32_t c = (uint32_t)__builtin_popcountll(m[i] & live);
        s.total += c;
        s.most = c > s.most ? c : s.most;
    }
    return s;
}
// stored values of a block-based layer (rows x columns of every block, rounded up to eight) and its fullest column set
__attribute__((target_clones("popcnt", "default"))) MaskSums count_values(const uint64_t *r, const uint64_t *c, size_t n, uint64_t rlive, uint64_t clive)
{
    MaskSums s{0, 0};
    for (size_t i = 0; i < n; ++i) {
        const uint32_t nc = (uint32_t)__builtin_popcountll(c[i] & clive);
        s.total += ((uint64_t)__builtin_popcountll(r[i] & rlive) * nc + 7) / 8 * 8;
        s.most = nc > s.most ? nc : s.most;
    }
    return s;
}
uint64_t low_bits(int n) { return n >= 64 ? ~0ull : (1ull << n) - 1; }

// Mask words that come from the host: counted here, uploaded for the packers.
struct Mask { at::Tensor dev, host; };
bool upload(const at::Tensor &m, int64_t n, const at::Device &dev, cudaStream_t st, Mask &out)
{
    out.host = at::empty({n}, at::TensorOptions().dtype(at::kLong));
    memcpy(out.host.data_ptr(), m.data_ptr(), (size_t)n * 8);
    out.dev = new_tensor({n}, at::kLong, dev);
    const cudaError_t e = cudaMemcpyAsync(out.dev.data_ptr(), out.host.data_ptr(), (size_t)n * 8, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) { PyErr_SetString(PyExc_RuntimeError, cudaGetErrorString(e)); return false; }
    return true;
}
bool mask_arg(const at::Tensor &m, int64_t n)
{
    return (m.scalar_type() == at::kLong && m.is_contiguous() && m.numel() >= n) || fail_assert("mask words: contiguous int64, one per block");
}

// Mask words on the device: what is kept has to be known here before the blob can be allocated, and other streams and
// threads may change the words meanwhile.  The plan reads them once and posts the counts as one word of page-locked memory,
// on which this thread spins (copying the masks to the host, waiting for the stream and counting, with the scan
// of the masks behind that: prune + pack of 512x3x3x512 38.3 us, now 27.8 together with the selection).  Should the stream end, or fail, without a post, so does the call.
template <typename F>
bool planned(cudaStream_t st, F launch, MaskSums &sums)
{
    const at::Tensor word = at::empty({1}, at::TensorOptions().dtype(at::kLong).pinned_memory(true));
    uint64_t *p = static_cast<uint64_t *>(word.data_ptr()), v = 0;
    *p = 0;
    cudaError_t e = cudaErrorNotReady;
    npas_status s;
    Py_BEGIN_ALLOW_THREADS
    s = launch(p);
    for (uint32_t spins = 1; s == NPAS_OK && e == cudaErrorNotReady; ++spins) {
        if ((v = __atomic_load_n(p, __ATOMIC_ACQUIRE)) != 0) break;
        if (spins % 4096 == 0) e = cudaStreamQuery(st);
    }
    if (s == NPAS_OK && v == 0) v = __atomic_load_n(p, __ATOMIC_ACQUIRE);
    Py_END_ALLOW_THREADS
    if (v == 0) {
        PyErr_SetString(PyExc_RuntimeError, s != NPAS_OK ? npas_status_string(s) : cudaGetErrorString(e));
        return false;
    }
    sums = MaskSums{v & 0xFFFFFFFFu, (uint32_t)(v >> 32) & 0x7FFFFFFFu};
    return true;
}
// A blob object: blob_type(data, desc) with a desc_type instance that holds d; or the status as an int.
template <typename D>
PyObject *packed(npas_status s, at::Tensor &&blob, const D &d, PyObject *desc_type, PyObject *blob_type)
{
    if (s != NPAS_OK) return PyLong_FromLong((long)s);
    PyObject *desc = PyObject_CallNoArgs(desc_type);
    if (!desc) return nullptr;
    Py_buffer view;
    bool ok = PyObject_GetBuffer(desc, &view, PyBUF_WRITABLE) == 0;
    if (ok) {
        ok = view.len == (Py_ssize_t)sizeof(D);
        if (ok) memcpy(view.buf, &d, sizeof(D));
        PyBuffer_Release(&view);
        if (!ok) PyErr_SetString(PyExc_TypeError, "descriptor of the wrong type");
    }
    PyObject *data = ok ? THPVariable_Wrap(std::move(blob)) : nullptr, *r = nullptr;
    if (data) {
        PyObject *args[2] = {data, desc};
        r = PyObject_Vectorcall(blob_type, args, 2, nullptr);
    }
    Py_XDECREF(data);
    Py_DECREF(desc);
    return r;
}

// Mask words as the packers take them, an int64 tensor on w's device or on the CPU: the argument itself, or what the Python
// function `words`(mask, device) makes of it.  `made` keeps what was made.
struct Owned {
    PyObject *p = nullptr;
    ~Owned() { Py_XDECREF(p); }
};
bool mask_words(PyObject *o, PyObject *w_obj, const at::Tensor &w, PyObject *words, Owned &made, const at::Tensor *&m)
{
    if (THPVariable_Check(o)) {
        m = &THPVariable_Unpack(o);
        if (m->scalar_type() == at::kLong && m->device() == w.device() && m->is_contiguous()) return true;
    }
    Owned dev;
    dev.p = PyObject_GetAttrString(w_obj, "device");
    if (!dev.p) return false;
    PyObject *args[2] = {o, dev.p};
    made.p = PyObject_Vectorcall(words, args, 2, nullptr);
    return made.p && tensor_arg(made.p, m, false, "mask");
}

// the types of the weights and of the packed weights (None: the same)
bool weight_types(const at::Tensor &w, PyObject *packed_dtype, int32_t &in, int32_t &out)
{
    at::ScalarType t;
    if (!dtype_of(w.scalar_type(), in)) return false;
    if (packed_dtype != Py_None && !THPDtype_Check(packed_dtype)) { PyErr_Format(PyExc_TypeError, "unsupported dtype %R", packed_dtype); return false; }
    return dtype_arg(packed_dtype, w.scalar_type(), t) && dtype_of(t, out);
}

bool whole_arg(PyObject *o, long long &v)             // int(o)
{
    Owned i;
    i.p = PyNumber_Long(o);
    if (!i.p) return false;
    v = PyLong_AsLongLong(i.p);
    return !(v == -1 && PyErr_Occurred());
}

// pack_bp(w, mask, Mb, Nb, packed_dtype, words, desc_type, blob_type) -> blob, or the status
PyObject *pack_bp(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *w, *m;
        Owned made;
        npas_bp_desc d = {};
        if (n != 8) { PyErr_SetString(PyExc_TypeError, "pack_bp takes 8 arguments"); return nullptr; }
        if (!tensor_arg(a[0], w, false, "w")) return nullptr;
        if (!(w->is_cuda() && w->is_contiguous() && w->dim() == 4)) { fail_assert("w must be a contiguous 4-D CUDA tensor"); return nullptr; }
        d.K = (int32_t)w->size(0); d.R = (int32_t)w->size(1); d.S = (int32_t)w->size(2); d.C = (int32_t)w->size(3);
        if (!weight_types(*w, a[4], d.w_in, d.w_packed) || !mask_words(a[1], a[0], *w, a[5], made, m) || !int_arg(a[2], d.Mb) || !int_arg(a[3], d.Nb)) return nullptr;
        size_t bytes = 0;
        npas_status s = npas_internal_bp_size(&d, 0, &bytes);
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        const cudaStream_t st = c10::cuda::getCurrentCUDAStream().stream();
        const int64_t blocks = (int64_t)(d.K / d.Mb) * (d.C / d.Nb);
        if (!mask_arg(*m, blocks)) return nullptr;
        Mask mask;
        at::Tensor scratch;
        MaskSums sums;
        if (m->is_cuda()) {
            size_t need = 0;
            npas_internal_plan_bp_bytes(&d, &need);
            scratch = new_tensor({(int64_t)need}, at::kByte, w->device());
            if (!planned(st, [&](uint64_t *host) { return npas_internal_plan_bp(&d, static_cast<const uint64_t *>(m->data_ptr()), scratch.data_ptr(), host, st); }, sums)) return nullptr;
        } else {
            if (!upload(*m, blocks, w->device(), st, mask)) return nullptr;
            sums = count_bits(static_cast<const uint64_t *>(mask.host.data_ptr()), (size_t)blocks, low_bits(d.R * d.S));
        }
        d.max_taps = sums.most ? (int32_t)sums.most : 1;
        s = npas_internal_bp_size(&d, sums.total, &bytes);
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        at::Tensor blob = new_tensor({(int64_t)bytes}, at::kByte, w->device());
        Py_BEGIN_ALLOW_THREADS
        s = m->is_cuda() ? npas_internal_pack_bp_planned(&d, w->data_ptr(), scratch.data_ptr(), sums.total, blob.data_ptr(), bytes, st)
                         : npas_internal_pack_bp(&d, w->data_ptr(), static_cast<const uint64_t *>(mask.dev.data_ptr()), blob.data_ptr(), bytes, st);
        Py_END_ALLOW_THREADS
        return packed(s, std::move(blob), d, a[6], a[7]);
    });
}

// pack_bb(w, rows, cols, Bo, Bi, packed_dtype, words, desc_type, blob_type) -> blob, or the status
PyObject *pack_bb(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *w, *mr, *mc;
        Owned made_r, made_c;
        npas_bb_desc d = {};
        if (n != 9) { PyErr_SetString(PyExc_TypeError, "pack_bb takes 9 arguments"); return nullptr; }
        if (!tensor_arg(a[0], w, false, "w")) return nullptr;
        if (!(w->is_cuda() && w->is_contiguous() && w->dim() == 2)) { fail_assert("w must be a contiguous 2-D CUDA tensor"); return nullptr; }
        d.O = (int32_t)w->size(0); d.I = (int32_t)w->size(1);
        if (!weight_types(*w, a[5], d.w_in, d.w_packed) || !mask_words(a[1], a[0], *w, a[6], made_r, mr) || !mask_words(a[2], a[0], *w, a[6], made_c, mc) ||
            !int_arg(a[3], d.Bo) || !int_arg(a[4], d.Bi))
            return nullptr;
        size_t bytes = 0;
        npas_status s = npas_internal_bb_size(&d, 0, 0, &bytes);
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        const cudaStream_t st = c10::cuda::getCurrentCUDAStream().stream();
        const int64_t blocks = (int64_t)(d.O / d.Bo) * (d.I / d.Bi);
        if (!mask_arg(*mr, blocks) || !mask_arg(*mc, blocks)) return nullptr;
        Mask rows, cols;
        at::Tensor scratch;
        MaskSums sums;
        if (!mr->is_cuda() && !upload(*mr, blocks, w->device(), st, rows)) return nullptr;
        if (!mc->is_cuda() && !upload(*mc, blocks, w->device(), st, cols)) return nullptr;
        const uint64_t *dr = static_cast<const uint64_t *>(mr->is_cuda() ? mr->data_ptr() : rows.dev.data_ptr());
        const uint64_t *dc = static_cast<const uint64_t *>(mc->is_cuda() ? mc->data_ptr() : cols.dev.data_ptr());
        const bool plan = mr->is_cuda() || mc->is_cuda();
        if (plan) {
            size_t need = 0;
            npas_internal_plan_bb_bytes(&d, &need);
            scratch = new_tensor({(int64_t)need}, at::kByte, w->device());
            if (!planned(st, [&](uint64_t *host) { return npas_internal_plan_bb(&d, dr, dc, scratch.data_ptr(), host, st); }, sums)) return nullptr;
        } else {
            sums = count_values(static_cast<const uint64_t *>(rows.host.data_ptr()), static_cast<const uint64_t *>(cols.host.data_ptr()), (size_t)blocks,
                                low_bits(d.Bo), low_bits(d.Bi));
        }
        d.max_cols = sums.most ? (int32_t)sums.most : 1;
        s = npas_internal_bb_size(&d, sums.total, sums.most, &bytes);
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        at::Tensor blob = new_tensor({(int64_t)bytes}, at::kByte, w->device());
        Py_BEGIN_ALLOW_THREADS
        s = plan ? npas_internal_pack_bb_planned(&d, w->data_ptr(), scratch.data_ptr(), sums.total, sums.most, blob.data_ptr(), bytes, st)
                 : npas_internal_pack_bb(&d, w->data_ptr(), dr, dc, blob.data_ptr(), bytes, st);
        Py_END_ALLOW_THREADS
        return packed(s, std::move(blob), d, a[7], a[8]);
    });
}

// prune_bp_global(w, Mb, Nb, rate, n_keep) -> masks, or the status; one of the last two is None
PyObject *prune_bp_global(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *w;
        npas_bp_desc d = {};
        if (n != 5) { PyErr_SetString(PyExc_TypeError, "prune_bp_global takes 5 arguments"); return nullptr; }
        if (!tensor_arg(a[0], w, false, "w")) return nullptr;
        if (!(w->is_cuda() && w->is_contiguous() && w->dim() == 4)) { fail_assert("w must be a contiguous 4-D CUDA tensor"); return nullptr; }
        if ((a[3] == Py_None) == (a[4] == Py_None)) { fail_assert("either rate or n_keep"); return nullptr; }
        if (!int_arg(a[1], d.Mb) || !int_arg(a[2], d.Nb) || !dtype_of(w->scalar_type(), d.w_in)) return nullptr;
        d.K = (int32_t)w->size(0); d.R = (int32_t)w->size(1); d.S = (int32_t)w->size(2); d.C = (int32_t)w->size(3);
        d.w_packed = d.w_in;
        long long n_keep = 0;
        if (a[3] == Py_None) {
            if (!whole_arg(a[4], n_keep)) return nullptr;
        } else {
            Owned f;
            f.p = PyNumber_Float(a[3]);
            if (!f.p) return nullptr;
            const double rate = PyFloat_AS_DOUBLE(f.p);
            if (d.Mb == 0 || d.Nb == 0 || rate == 0.0) { PyErr_SetString(PyExc_ZeroDivisionError, "division by zero"); return nullptr; }
            const double keep = std::floor((double)((long long)(d.K / d.Mb) * (d.C / d.Nb) * d.R * d.S) / rate + 0.5);
            if (!(std::fabs(keep) < 9e18)) { PyErr_SetString(std::isnan(keep) ? PyExc_ValueError : PyExc_OverflowError, "cannot keep that many groups"); return nullptr; }
            n_keep = (long long)keep;
        }
        size_t bytes = 0;
        npas_status s = npas_prune_bp_global_workspace(&d, &bytes);
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        at::Tensor ws = new_tensor({(int64_t)bytes}, at::kByte, w->device()), tm = new_tensor({d.K / d.Mb, d.C / d.Nb}, at::kLong, w->device());
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        Py_BEGIN_ALLOW_THREADS
        s = npas_prune_bp_magnitude_global(&d, w->data_ptr(), n_keep, static_cast<uint64_t *>(tm.data_ptr()), ws.data_ptr(), bytes, st);
        Py_END_ALLOW_THREADS
        return result(s, nullptr, std::move(tm));
    });
}

// prune_bb(w, Bo, Bi, keep_rows, keep_cols) -> (rows, columns), or the status
PyObject *prune_bb(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *w;
        npas_bb_desc d = {};
        long long kr, kc;
        if (n != 5) { PyErr_SetString(PyExc_TypeError, "prune_bb takes 5 arguments"); return nullptr; }
        if (!tensor_arg(a[0], w, false, "w") || !int_arg(a[1], d.Bo) || !int_arg(a[2], d.Bi) || !dtype_of(w->scalar_type(), d.w_in) || !whole_arg(a[3], kr) || !whole_arg(a[4], kc))
            return nullptr;
        if (!(w->is_cuda() && w->is_contiguous() && w->dim() == 2)) { fail_assert("w must be a contiguous 2-D CUDA tensor"); return nullptr; }
        d.O = (int32_t)w->size(0); d.I = (int32_t)w->size(1);
        d.w_packed = d.w_in;
        if (d.Bo == 0 || d.Bi == 0) { PyErr_SetString(PyExc_ZeroDivisionError, "block size is zero"); return nullptr; }
        at::Tensor rk = new_tensor({d.O / d.Bo, d.I / d.Bi}, at::kLong, w->device()), ck = new_tensor({d.O / d.Bo, d.I / d.Bi}, at::kLong, w->device());
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        npas_status s;
        Py_BEGIN_ALLOW_THREADS
        s = npas_prune_bb_magnitude(&d, w->data_ptr(), (int32_t)kr, (int32_t)kc, static_cast<uint64_t *>(rk.data_ptr()), static_cast<uint64_t *>(ck.data_ptr()), st);
        Py_END_ALLOW_THREADS
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        return Py_BuildValue("(NN)", THPVariable_Wrap(std::move(rk)), THPVariable_Wrap(std::move(ck)));
    });
}

// unpack_bb(blob, desc) -> (weights, rows, columns), or the status
PyObject *unpack_bb(PyObject *, PyObject *const *a, Py_ssize_t n)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *blob;
        npas_bb_desc d;
        if (n != 2) { PyErr_SetString(PyExc_TypeError, "unpack_bb takes 2 arguments"); return nullptr; }
        if (!tensor_arg(a[0], blob, false, "blob.data") || !desc_arg(a[1], d)) return nullptr;
        if (d.Bo == 0 || d.Bi == 0) { PyErr_SetString(PyExc_ZeroDivisionError, "block size is zero"); return nullptr; }
        const at::Device dev = blob->device();
        at::Tensor w = new_tensor({d.O, d.I}, d.w_packed == NPAS_F32 ? at::kFloat : at::kBFloat16, dev);
        at::Tensor rk = new_tensor({d.O / d.Bo, d.I / d.Bi}, at::kLong, dev), ck = new_tensor({d.O / d.Bo, d.I / d.Bi}, at::kLong, dev);
        void *st = c10::cuda::getCurrentCUDAStream().stream();
        npas_status s;
        Py_BEGIN_ALLOW_THREADS
        s = npas_unpack_bb(&d, blob->data_ptr(), (size_t)blob->numel(), w.data_ptr(), static_cast<uint64_t *>(rk.data_ptr()), static_cast<uint64_t *>(ck.data_ptr()), st);
        Py_END_ALLOW_THREADS
        if (s != NPAS_OK) return PyLong_FromLong((long)s);
        return Py_BuildValue("(NNN)", THPVariable_Wrap(std::move(w)), THPVariable_Wrap(std::move(rk)), THPVariable_Wrap(std::move(ck)));
    });
}

// ---- a whole stack of layers --------------------------------------------------------------------------------------
// One call for the forward pass of a chain of layers: what Python did between the layers (shapes, keys, liveness, two
// allocations) took longer than the layers of a small batch.  The activations lie in one buffer, placed by first fit over
// the layers' lifetimes; only the result is a tensor of its own.

struct Span { int64_t lo, hi; };

// First-fit placement of buffers with known lifetimes in [0, size): `busy` is kept sorted.
class Arena {
public:
    int64_t take(int64_t bytes)
    {
        bytes = (bytes + 255) & ~int64_t(255);
        int64_t at = 0;
        size_t i = 0;
        for (; i < busy_.size() && busy_[i].lo - at < bytes; ++i) at = busy_[i].hi;
        busy_.insert(busy_.begin() + (long)i, Span{at, at + bytes});
        if (at + bytes > size_) size_ = at + bytes;
        return at;
    }
    void give(int64_t at)
    {
        for (size_t i = 0; i < busy_.size(); ++i)
            if (busy_[i].lo == at) { busy_.erase(busy_.begin() + (long)i); return; }
    }
    int64_t size() const { return size_; }

private:
    std::vector<Span> busy_;
    int64_t size_ = 0;
};

// One row of the topology: kind 0 first layer (followed by the max-pool), 1 convolution, 2 GEMM over the pixels.
enum { kApart = 1, kTogether = 2 };
struct LayerRow { int32_t kind, stride, pad, relu, cout, src, res, reserved; };

// A second stream and the two events that tie it to the caller's, one set per thread (made for the device it last used, given
// back when the thread ends).
struct SideStream {
    int dev = -1;
    cudaStream_t stream = nullptr;
    cudaEvent_t ready = nullptr, done = nullptr;
    void give_back()
    {
        if (ready) cudaEventDestroy(ready);
        if (done) cudaEventDestroy(done);
        if (stream) cudaStreamDestroy(stream);
        stream = nullptr; ready = done = nullptr; dev = -1;
    }
    // usable for work of the current device forked from `main`?  (Nothing is created while `main` is being captured.)
    bool prepare(cudaStream_t main)
    {
        int d = -1;
        if (cudaGetDevice(&d) != cudaSuccess) return false;
        if (d == dev) return true;
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(main, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
        give_back();
        if (cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking) != cudaSuccess || cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&done, cudaEventDisableTiming) != cudaSuccess) {
            give_back();
            cudaGetLastError();
            return false;
        }
        dev = d;
        return true;
    }
    ~SideStream() { give_back(); }
};
thread_local SideStream side;

// stack_forward(x, rows, blobs, biases, ws, routes): rows = bytes of LayerRow; routes = None, or [path, variant, with_next] of every
// layer as a flat list.  src / res: index of a layer, -1 the network's input, -2 the pooled tensor, -3 (res only) none.
// with_next: whether a layer and the one behind it were measured faster one by one (kApart) or in one launch (kTogether, whatever
// their own plans); not measured (0), they share a launch where that is preferred and neither has a plan of its own.
PyObject *stack_forward(PyObject *, PyObject *const *a, Py_ssize_t nargs)
{
    return guarded([&]() -> PyObject * {
        const at::Tensor *x, *ws;
        if (nargs != 6) { PyErr_SetString(PyExc_TypeError, "stack_forward takes 6 arguments"); return nullptr; }
        if (!tensor_arg(a[0], x, false, "x") || !tensor_arg(a[4], ws, false, "ws")) return nullptr;
        if (!PyBytes_Check(a[1]) || !PyList_Check(a[2]) || !PyList_Check(a[3])) { PyErr_SetString(PyExc_TypeError, "stack_forward: rows, blobs, biases"); return nullptr; }
        const int L = (int)(PyBytes_GET_SIZE(a[1]) / (Py_ssize_t)sizeof(LayerRow));
        const LayerRow *rows = reinterpret_cast<const LayerRow *>(PyBytes_AS_STRING(a[1]));
        if (L < 1 || PyList_GET_SIZE(a[2]) != L || PyList_GET_SIZE(a[3]) != L) { fail_assert("stack_forward: one blob and one bias per layer"); return nullptr; }
        if (!(x->is_cuda() && x->is_contiguous() && x->dim() == 4 && x->scalar_type() == at::kBFloat16)) { fail_assert("x must be a contiguous 4-D bf16 CUDA tensor"); return nullptr; }
        struct Step {
            npas_conv_desc cd; npas_linear_desc ld; npas_bp_desc bp; npas_bb_desc bb;
            const void *blob; const float *bias;
            int64_t h, w, p, q, out, sub;          // input and output height / width, buffer of the output, of the subsampled input (-1: none)
            int64_t in_at, res_at;                  // -1: the network's input / none
        };
        std::vector<Step> steps((size_t)L);
        struct Shape { int64_t h, w, c, at; };
        std::vector<Shape> made((size_t)L);
        std::vector<int> last((size_t)L, -1);
        int pooled_last = -1;
        for (int i = 0; i < L; ++i)
            for (int s : {rows[i].src, rows[i].res}) {
                if (s >= i || s < -3) { fail_assert("stack_forward: a layer reads a later one"); return nullptr; }
                if (s >= 0) last[(size_t)s] = i;
                if (s == -2) pooled_last = i;
            }
        if (a[5] != Py_None && (!PyList_Check(a[5]) || PyList_GET_SIZE(a[5]) != 3 * (Py_ssize_t)L)) { fail_assert("stack_forward: three numbers per layer in routes"); return nullptr; }
        auto route = [&](int i, int which, int32_t &v) { return int_arg(PyList_GET_ITEM(a[5], 3 * i + which), v); };
        Shape pooled{0, 0, 0, -1};
        Arena arena;
        const int64_t N = x->size(0);
        // Layers that can run beside others: a GEMM whose input was there before the layers just ahead of it (the projection of
        // a shortcut, beside the block's first two convolutions).  It starts on a second stream when layer from[i] has finished
        // and is waited for before layer join[i], the first that reads it; its buffers are taken when it may start and its input
        // is kept until the join.  Only where it leaves most of the chip free (fewer 128 x 128 tiles than half the SMs): one image
        // of 224 x 224 270 us instead of 278, of 64 x 64 224 instead of 240; larger batches fill the chip one layer at a time.
        std::vector<int> from((size_t)L, -1), join((size_t)L, -1), begins((size_t)L, -1);     // begins[s]: the layer that starts after s
        c10::cuda::CUDAStream main_stream = c10::cuda::getCurrentCUDAStream();
        int dev = 0, sms = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 0;
        bool forks = false;
        for (int i = 2; i < L; ++i) {
            int s = rows[i].src;
            if (s == -2)
                for (int j = 0; j < i; ++j)
                    if (rows[j].kind == 0) s = j;
            if (rows[i].kind != 2 || rows[i].res != -3 || s < 0 || s >= i - 1 || begins[(size_t)s] >= 0) continue;
            int j = i + 1;
            while (j < L && rows[j].src != i && rows[j].res != i) ++j;
            bool free_between = j < L;
            for (int k = s + 1; k < j && k < L; ++k) free_between = free_between && (k == i || (from[(size_t)k] < 0 && begins[(size_t)k] < 0));
            if (!free_between) continue;
            from[(size_t)i] = s; join[(size_t)i] = j; begins[(size_t)s] = i;
        }
        // Two 1x1 layers behind one another, the second reading nothing but the first: one launch where that is the faster way.
        // Its outputs are written while its inputs are still being read, so what is free behind the first layer is given back
        // behind the second only.
        std::vector<char> two((size_t)L, 0);
        std::vector<int64_t> held;
        auto give = [&](int i, int64_t at) {
            if (two[(size_t)i]) held.push_back(at);
            else arena.give(at);
        };
        for (int i = 0; i < L; ++i) {
            const LayerRow &r = rows[i];
            Step &st = steps[(size_t)i];
            PyObject *bo = PyList_GET_ITEM(a[2], i);
            PyObject *data = PyObject_GetAttrString(bo, "data");
            if (!data) return nullptr;
            Py_DECREF(data);                        // (the blob object keeps it)
            PyObject *desc = PyObject_GetAttrString(bo, "desc");
            if (!desc) return nullptr;
            Py_DECREF(desc);
            const at::Tensor *blob, *bias;
            if (!tensor_arg(data, blob, false, "blob.data") || !tensor_arg(PyList_GET_ITEM(a[3], i), bias, false, "bias")) return nullptr;
            st.blob = blob->data_ptr(); st.bias = static_cast<const float *>(bias->data_ptr());
            int32_t path = 0, variant = 0;
            if (a[5] != Py_None && (!route(i, 0, path) || !route(i, 1, variant))) return nullptr;
            const Shape in = r.src == -1 ? Shape{x->size(1), x->size(2), x->size(3), -1} : r.src == -2 ? pooled : made[(size_t)r.src];
            st.h = in.h; st.w = in.w; st.in_at = in.at;
            if (from[(size_t)i] < 0) st.sub = -1;
            st.res_at = r.res == -2 ? pooled.at : r.res >= 0 ? made[(size_t)r.res].at : -1;
            const bool has_res = r.res == -2 || r.res >= 0;
            if (r.kind == 2) {
                if (!desc_arg(desc, st.bb)) return nullptr;
                st.p = (in.h - 1) / r.stride + 1; st.q = (in.w - 1) / r.stride + 1;
                if (r.stride != 1 && from[(size_t)i] < 0) st.sub = arena.take(N * st.p * st.q * in.c * 2);
                st.ld = npas_linear_desc{(int32_t)(N * st.p * st.q), (int32_t)in.c, r.cout, NPAS_BF16, NPAS_BF16, r.relu, 1, has_res, path, variant};
            } else {
                if (!desc_arg(desc, st.bp)) return nullptr;
                st.p = (in.h + 2 * r.pad - st.bp.R) / r.stride + 1; st.q = (in.w + 2 * r.pad - st.bp.S) / r.stride + 1;
                st.cd = npas_conv_desc{(int32_t)N, (int32_t)in.h, (int32_t)in.w, (int32_t)in.c, r.cout, st.bp.R, st.bp.S, r.stride, r.pad,
                                       NPAS_BF16, NPAS_BF16, r.relu, 1, has_res, path, variant};
                if (r.kind == 0) { st.p = (st.p + 2 - 3) / 2 + 1; st.q = (st.q + 2 - 3) / 2 + 1; }      // the pooled tensor
            }
            if (from[(size_t)i] < 0) st.out = i == L - 1 ? -1 : arena.take(N * st.p * st.q * r.cout * 2);
            if (i > 0 && two[(size_t)i - 1]) st.ld.path = st.ld.variant = 0;
            else if (r.kind == 2 && r.stride == 1 && from[(size_t)i] < 0 && i + 1 < L) {
                const LayerRow &t = rows[i + 1];
                int32_t with_next = 0, path2 = 0, variant2 = 0;
                if (a[5] != Py_None && (!route(i, 2, with_next) || !route(i + 1, 0, path2) || !route(i + 1, 1, variant2))) return nullptr;
                npas_linear_desc one = st.ld;
                one.path = one.variant = 0;
                const npas_linear_desc b{st.ld.M, r.cout, t.cout, NPAS_BF16, NPAS_BF16, t.relu, 1, 0, 0, 0};
                two[(size_t)i] = t.kind == 2 && t.stride == 1 && t.src == i && t.res == -3 && from[(size_t)i + 1] < 0 && begins[(size_t)i + 1] < 0 &&
                                 (with_next == kTogether || (with_next == 0 && !path && !variant && !path2 && !variant2)) && npas_internal_linear_two_preferred(&one, &b);
                if (two[(size_t)i]) st.ld = one;
            }
            made[(size_t)i] = Shape{st.p, st.q, r.cout, st.out};
            if (r.kind == 0) pooled = made[(size_t)i];
            if (st.sub >= 0 && from[(size_t)i] < 0) give(i, st.sub);
            // buffers that no later layer reads (the pooled tensor has one of its own name)
            for (int j = 0; j <= i; ++j)
                if (made[(size_t)j].at >= 0 && j != L - 1 && rows[j].kind != 0 && last[(size_t)j] <= i && (last[(size_t)j] == i || j == i)) give(i, made[(size_t)j].at);
            if (pooled.at >= 0 && pooled_last == i) give(i, pooled.at);
            for (int k = 0; k < i; ++k)                     // a layer beside these ends here: its subsampled input is free
                if (from[(size_t)k] >= 0 && join[(size_t)k] == i && steps[(size_t)k].sub >= 0) give(i, steps[(size_t)k].sub);
            if (i > 0 && two[(size_t)i - 1]) {
                for (const int64_t at : held) arena.give(at);
                held.clear();
            }
            const int f = begins[(size_t)i];
            if (f >= 0) {
                const Shape &o = made[(size_t)i];
                const int64_t p = (o.h - 1) / rows[f].stride + 1, q = (o.w - 1) / rows[f].stride + 1;
                const bool small = ((N * p * q + 127) / 128) * ((rows[f].cout + 127) / 128) * 2 <= sms;
                if (!small || (!forks && !side.prepare(main_stream.stream()))) { from[(size_t)f] = -1; begins[(size_t)i] = -1; }
                else {
                    forks = true;
                    steps[(size_t)f].sub = rows[f].stride != 1 ? arena.take(N * p * q * o.c * 2) : -1;
                    steps[(size_t)f].out = arena.take(N * p * q * rows[f].cout * 2);
                    int &kept = rows[f].src == -2 ? pooled_last : last[(size_t)rows[f].src];
                    if (kept < join[(size_t)f]) kept = join[(size_t)f];
                }
            }
        }
        const Step &end = steps[(size_t)L - 1];
        at::Tensor y = new_tensor({N, end.p, end.q, rows[L - 1].cout}, at::kBFloat16, x->device());
        at::Tensor buf = new_tensor({arena.size()}, at::kByte, x->device());
        uint8_t *base = static_cast<uint8_t *>(buf.data_ptr());
        void *xin = x->data_ptr(), *yout = y.data_ptr(), *w = ws->data_ptr();
        cudaStream_t main = main_stream.stream();
        const size_t wb = (size_t)ws->numel();
        npas_status s = NPAS_OK;
        int at_layer = 0, pending = -1;                // pending: the layer that runs, or will run, on the second stream
        Py_BEGIN_ALLOW_THREADS
        for (int i = 0; i < L && s == NPAS_OK; ++i) {
            const LayerRow &r = rows[i];
            const Step &st = steps[(size_t)i];
            const void *in = st.in_at < 0 ? xin : base + st.in_at, *res = st.res_at < 0 ? nullptr : base + st.res_at;
            void *out = st.out < 0 ? yout : base + st.out;
            at_layer = i;
            // nothing in this call writes a blob, and a layer beside starts behind an event recorded after the first layer
            const int32_t chain = i == 0 ? NPAS_CHAIN_FIRST : NPAS_CHAIN_LATER;
            const bool beside = from[(size_t)i] >= 0;
            void *stream = beside ? side.stream : main;
            if (pending >= 0 && join[(size_t)pending] == i) {
                if (cudaStreamWaitEvent(main, side.done, 0) != cudaSuccess) s = NPAS_ERR_CUDA;
                pending = -1;
                if (s != NPAS_OK) break;
            }
            if (i > 0 && two[(size_t)i - 1]) continue;     // (done together with the layer before)
            if (two[(size_t)i]) {
                const Step &t = steps[(size_t)i + 1];
                s = npas_internal_linear_two(&st.ld, &st.bb, &t.ld, &t.bb, in, st.blob, st.bias, res, out, t.blob, t.bias, t.out < 0 ? yout : base + t.out, w, wb,
                                             chain, stream);
            } else if (r.kind == 2) {
                if (st.sub >= 0) {
                    s = npas_subsample2d((int32_t)N, (int32_t)st.h, (int32_t)st.w, st.ld.I, r.stride, 2, in, base + st.sub, stream);
                    if (s != NPAS_OK) break;
                    in = base + st.sub;
                }
                s = npas_internal_linear_bb(&st.ld, &st.bb, in, st.blob, st.bias, res, out, w, wb, chain, stream);
            } else if (r.kind == 0) {
                s = npas_internal_conv2d_bp_maxpool(&st.cd, &st.bp, 3, 2, 1, in, st.blob, st.bias, out, w, wb, chain, stream);
            } else {
                s = npas_internal_conv2d_bp(&st.cd, &st.bp, in, st.blob, st.bias, res, out, w, wb, chain, stream);
            }
            if (beside && s == NPAS_OK && cudaEventRecord(side.done, side.stream) != cudaSuccess) s = NPAS_ERR_CUDA;
            if (s == NPAS_OK && begins[(size_t)i] >= 0) {
                if (cudaEventRecord(side.ready, main) != cudaSuccess || cudaStreamWaitEvent(side.stream, side.ready, 0) != cudaSuccess) s = NPAS_ERR_CUDA;
                else pending = begins[(size_t)i];
            }
        }
        // (left early: what already runs beside is still the caller's stream's to wait for)
        if (pending >= 0 && cudaEventRecord(side.done, side.stream) == cudaSuccess) cudaStreamWaitEvent(main, side.done, 0);
        Py_END_ALLOW_THREADS
        if (s != NPAS_OK) return Py_BuildValue("(ii)", (int)s, at_layer);
        return THPVariable_Wrap(std::move(y));
    });
}

PyMethodDef kMethods[] = {
    {"conv2d_bp", (PyCFunction)(void (*)(void))conv2d_bp, METH_FASTCALL, nullptr},
    {"conv2d_bp_maxpool", (PyCFunction)(void (*)(void))conv2d_bp_maxpool, METH_FASTCALL, nullptr},
    {"linear_bb", (PyCFunction)(void (*)(void))linear_bb, METH_FASTCALL, nullptr},
    {"pack_bp", (PyCFunction)(void (*)(void))pack_bp, METH_FASTCALL, nullptr},
    {"pack_bb", (PyCFunction)(void (*)(void))pack_bb, METH_FASTCALL, nullptr},
    {"prune_bp_global", (PyCFunction)(void (*)(void))prune_bp_global, METH_FASTCALL, nullptr},
    {"prune_bb", (PyCFunction)(void (*)(void))prune_bb, METH_FASTCALL, nullptr},
    {"unpack_bb", (PyCFunction)(void (*)(void))unpack_bb, METH_FASTCALL, nullptr},
    {"stack_forward", (PyCFunction)(void (*)(void))stack_forward, METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_npas_host", nullptr, -1, kMethods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__npas_host() { return PyModule_Create(&kModule); }
