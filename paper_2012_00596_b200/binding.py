"""Binding over libnpas.so: argument marshalling only, every step runs in the CUDA kernels.

The function names mirror the C ABI (include/npas.h).  Tensors are torch CUDA tensors used purely
as device buffers; calls are enqueued on torch's current stream.  The compute calls go through a
CPython extension (csrc/host_ext.cpp), the rest through ctypes.  There is no CPU fallback: when
a shared library is missing or a call fails, an exception is raised.
"""
from __future__ import annotations

import ctypes
import importlib.util
import os
from dataclasses import dataclass

import numpy as np
import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libnpas.so")
HOST_PATH = os.path.join(_HERE, "_npas_host.so")
WORKSPACE_BYTES = 256
F32, BF16 = 0, 1
_lib = None
_host = None                     # the extension module, from the first load() on


class NpasError(RuntimeError):
    def __init__(self, code: int, what: str):
        super().__init__(f"{what}: {status_string(code)} (npas_status {code})")
        self.code = code


class BpDesc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("K", "C", "R", "S", "Mb", "Nb", "w_in", "w_packed", "max_taps")]


class BbDesc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("O", "I", "Bo", "Bi", "w_in", "w_packed", "max_cols")]


class ConvDesc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("N", "H", "W", "C", "K", "R", "S", "stride", "pad", "x_dtype",
                                              "y_dtype", "relu", "has_bias", "has_residual", "path", "variant")]


class LinearDesc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int32) for n in ("M", "I", "O", "x_dtype", "y_dtype", "relu", "has_bias", "has_residual", "path",
                                              "variant")]


EXPORTS = ["npas_status_string", "npas_abi_version", "npas_mask_bp_from_dense", "npas_mask_bb_from_dense",
           "npas_pack_bp_size", "npas_pack_bp", "npas_unpack_bp", "npas_pack_bb_size", "npas_pack_bb",
           "npas_unpack_bb", "npas_conv2d_bp", "npas_linear_bb", "npas_blob_check",
           "npas_check_device_status", "npas_launch_count", "npas_maxpool2d", "npas_conv2d_bp_static_ws",
           "npas_subsample2d", "npas_prune_bp_magnitude", "npas_prune_bb_magnitude",
           "npas_conv2d_bp_workspace", "npas_linear_bb_workspace", "npas_conv2d_bp_kernel", "npas_linear_bb_kernel",
           "npas_tune_conv2d_bp", "npas_tune_linear_bb", "npas_prune_bp_global_workspace", "npas_prune_bp_magnitude_global", "npas_conv2d_bp_maxpool"]


def load() -> ctypes.CDLL:
    """Load the CUDA library; raises if it has not been built (there is no other code path)."""
    global _lib, _host
    if _lib is None:
        for path in (LIB_PATH, HOST_PATH):
            if not os.path.exists(path):
                raise FileNotFoundError(f"{path} is missing: build it with paper_2012_00596_b200/build.py")
        lib = ctypes.CDLL(LIB_PATH)
        for name in EXPORTS:
            getattr(lib, name)
        lib.npas_status_string.restype = ctypes.c_char_p
        lib.npas_status_string.argtypes = [ctypes.c_int]
        lib.npas_abi_version.restype = ctypes.c_uint32
        lib.npas_launch_count.restype = ctypes.c_uint64
        for name in EXPORTS[2:]:
            if name == "npas_launch_count":
                continue
            getattr(lib, name).restype = ctypes.c_int
        spec = importlib.util.spec_from_file_location("_npas_host", HOST_PATH)
        host = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(host)
        _host, _lib = host, lib
    return _lib


def _refused(code: int, what: str):
    raise NpasError(code, what)


def status_string(code: int) -> str:
    return load().npas_status_string(int(code)).decode()


def launch_count() -> int:
    return int(load().npas_launch_count())


def _check(code: int, what: str):
    if code != 0:
        raise NpasError(code, what)


def _p(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _dt_code(dtype: torch.dtype) -> int:
    if dtype == torch.float32:
        return F32
    if dtype == torch.bfloat16:
        return BF16
    raise TypeError(f"unsupported dtype {dtype}")


def _dt(t: torch.Tensor) -> int:
    return _dt_code(t.dtype)


def _torch_dt(code: int):
    return torch.float32 if code == F32 else torch.bfloat16


def _mask_to_device(mask, device) -> torch.Tensor:
    """uint64 bitsets (numpy or tensor) -> contiguous int64 CUDA tensor holding the same bits."""
    if isinstance(mask, torch.Tensor):
        return mask.to(device=device, dtype=torch.int64).contiguous()
    return torch.from_numpy(np.ascontiguousarray(mask, dtype=np.uint64).view(np.int64)).to(device)


def _mask_words(mask, device) -> torch.Tensor:
    """Mask words as the packers take them: an int64 tensor on ``device``, or on the CPU."""
    if isinstance(mask, torch.Tensor):
        if mask.dtype == torch.int64 and mask.device == device and mask.is_contiguous():
            return mask
        mask = mask_to_numpy(mask)
    return torch.from_numpy(np.ascontiguousarray(mask, dtype=np.uint64).view(np.int64))


def mask_to_numpy(mask: torch.Tensor) -> np.ndarray:
    return mask.cpu().numpy().view(np.uint64)


@dataclass
class BpBlob:
    data: torch.Tensor          # uint8 device buffer holding the blob
    desc: BpDesc


@dataclass
class BbBlob:
    data: torch.Tensor
    desc: BbDesc


def workspace(device="cuda") -> torch.Tensor:
    """Zeroed device scratch for the compute calls (holds the device status words)."""
    return torch.zeros(WORKSPACE_BYTES, dtype=torch.uint8, device=device)


# ---------------------------------------------------------------------------- packers ----------

def pack_bp(w: torch.Tensor, tap_mask, Mb: int, Nb: int, packed_dtype=None) -> BpBlob:
    """npas_pack_bp: dense KRSC weights + per-block tap bitsets -> blob (on w's device)."""
    if _host is None:
        load()
    r = _host.pack_bp(w, tap_mask, Mb, Nb, packed_dtype, _mask_words, BpDesc, BpBlob)
    return r if type(r) is not int else _refused(r, "npas_pack_bp")


def unpack_bp(blob: BpBlob):
    """npas_unpack_bp -> (masked dense weights in the blob's dtype [K,R,S,C], tap_mask int64 [nFB,nCB])."""
    lib = load()
    d = blob.desc
    w = torch.empty((d.K, d.R, d.S, d.C), dtype=_torch_dt(d.w_packed), device=blob.data.device)
    tm = torch.empty((d.K // d.Mb, d.C // d.Nb), dtype=torch.int64, device=blob.data.device)
    _check(lib.npas_unpack_bp(ctypes.byref(d), _p(blob.data), ctypes.c_size_t(blob.data.numel()), _p(w), _p(tm),
                              _stream()), "npas_unpack_bp")
    return w, tm


def pack_bb(w: torch.Tensor, row_keep, col_keep, Bo: int, Bi: int, packed_dtype=None) -> BbBlob:
    if _host is None:
        load()
    r = _host.pack_bb(w, row_keep, col_keep, Bo, Bi, packed_dtype, _mask_words, BbDesc, BbBlob)
    return r if type(r) is not int else _refused(r, "npas_pack_bb")


def unpack_bb(blob: BbBlob):
    if _host is None:
        load()
    r = _host.unpack_bb(blob.data, blob.desc)
    return r if type(r) is not int else _refused(r, "npas_unpack_bb")


def prune_bp_magnitude(w: torch.Tensor, Mb: int, Nb: int, keep_taps: int) -> torch.Tensor:
    """npas_prune_bp_magnitude: dense KRSC weights -> per-block tap bitsets (int64 tensor on the device)."""
    lib = load()
    assert w.is_cuda and w.is_contiguous() and w.dim() == 4
    K, R, S, C = w.shape
    d = BpDesc(K, C, R, S, Mb, Nb, _dt(w), _dt(w), 0)
    tm = torch.empty((K // Mb, C // Nb), dtype=torch.int64, device=w.device)
    _check(lib.npas_prune_bp_magnitude(ctypes.byref(d), _p(w), int(keep_taps), _p(tm), _stream()), "npas_prune_bp_magnitude")
    return tm


def prune_bp_magnitude_global(w: torch.Tensor, Mb: int, Nb: int, *, rate: float = None, n_keep: int = None) -> torch.Tensor:
    """npas_prune_bp_magnitude_global: keep the ``n_keep`` highest-scoring (block, tap) groups of the whole
    layer (``rate``: n_keep = round(groups / rate), e.g. 2.5 or 7); tap bitsets as an int64 device tensor."""
    if _host is None:
        load()
    r = _host.prune_bp_global(w, Mb, Nb, rate, n_keep)
    return r if type(r) is not int else _refused(r, "npas_prune_bp_magnitude_global")


def prune_bb_magnitude(w: torch.Tensor, Bo: int, Bi: int, keep_rows: int, keep_cols: int):
    """npas_prune_bb_magnitude: dense [O,I] weights -> (row bitsets, column bitsets), int64 tensors on the device."""
    if _host is None:
        load()
    r = _host.prune_bb(w, Bo, Bi, keep_rows, keep_cols)
    return r if type(r) is not int else _refused(r, "npas_prune_bb_magnitude")


def mask_bp_from_dense(dense_mask: torch.Tensor, Mb: int, Nb: int) -> torch.Tensor:
    """npas_mask_bp_from_dense: uint8 [K,R,S,C] 0/1 mask -> tap bitsets; raises on a bad structure."""
    lib = load()
    K, R, S, C = dense_mask.shape
    d = BpDesc(K, C, R, S, Mb, Nb, F32, F32)
    m = dense_mask.to(torch.uint8).contiguous()
    tm = torch.empty((K // Mb, C // Nb), dtype=torch.int64, device=m.device)
    viol = torch.zeros(1, dtype=torch.int32, device=m.device)
    _check(lib.npas_mask_bp_from_dense(ctypes.byref(d), _p(m), _p(tm), _p(viol), _stream()),
           "npas_mask_bp_from_dense")
    return tm


def mask_bb_from_dense(dense_mask: torch.Tensor, Bo: int, Bi: int):
    lib = load()
    O, I = dense_mask.shape
    d = BbDesc(O, I, Bo, Bi, F32, F32)
    m = dense_mask.to(torch.uint8).contiguous()
    rk = torch.empty((O // Bo, I // Bi), dtype=torch.int64, device=m.device)
    ck = torch.empty_like(rk)
    viol = torch.zeros(1, dtype=torch.int32, device=m.device)
    _check(lib.npas_mask_bb_from_dense(ctypes.byref(d), _p(m), _p(rk), _p(ck), _p(viol), _stream()),
           "npas_mask_bb_from_dense")
    return rk, ck


def blob_check(blob) -> None:
    lib = load()
    bp = ctypes.byref(blob.desc) if isinstance(blob, BpBlob) else None
    bb = ctypes.byref(blob.desc) if isinstance(blob, BbBlob) else None
    _check(lib.npas_blob_check(bp, bb, _p(blob.data), ctypes.c_size_t(blob.data.numel()), _stream()),
           "npas_blob_check")


# ---------------------------------------------------------------------------- compute ----------

def conv2d_bp(x: torch.Tensor, blob: BpBlob, bias=None, residual=None, *, stride=1, pad=1, relu=False,
              out_dtype=None, out=None, ws=None, path=0, variant=0) -> torch.Tensor:
    """npas_conv2d_bp on NHWC x; returns NHWC y (allocated here unless ``out`` is given)."""
    if _host is None:
        load()
    y = _host.conv2d_bp(x, blob.data, blob.desc, bias, residual, stride, pad, relu, out_dtype, out, ws, path, variant)
    return y if type(y) is not int else _refused(y, "npas_conv2d_bp")


def linear_bb(x: torch.Tensor, blob: BbBlob, bias=None, residual=None, *, relu=False, out_dtype=None, out=None,
              ws=None, path=0, variant=0) -> torch.Tensor:
    if _host is None:
        load()
    y = _host.linear_bb(x, blob.data, blob.desc, bias, residual, relu, out_dtype, out, ws, path, variant)
    return y if type(y) is not int else _refused(y, "npas_linear_bb")


def subsample2d(x: torch.Tensor, stride: int) -> torch.Tensor:
    """Y[n,p,q,:] = X[n, p*stride, q*stride, :] (the input of a strided 1x1 convolution run as a GEMM)."""
    lib = load()
    assert x.is_cuda and x.is_contiguous() and x.dim() == 4
    N, H, W, C = x.shape
    y = torch.empty((N, (H - 1) // stride + 1, (W - 1) // stride + 1, C), dtype=x.dtype, device=x.device)
    _check(lib.npas_subsample2d(N, H, W, C, stride, x.element_size(), _p(x), _p(y), _stream()), "npas_subsample2d")
    return y


def check_device_status(ws: torch.Tensor) -> None:
    """Synchronises and raises NpasError(NPAS_ERR_TIMEOUT) if a kernel gave up on a bounded wait."""
    lib = load()
    detail = ctypes.c_int32(0)
    code = lib.npas_check_device_status(_p(ws), _stream(), ctypes.byref(detail))
    if code != 0:
        raise NpasError(code, f"device status (detail 0x{detail.value:x})")


def maxpool2d(x: torch.Tensor, R=3, stride=2, pad=1) -> torch.Tensor:
    lib = load()
    N, H, W, C = x.shape
    P = (H + 2 * pad - R) // stride + 1
    Q = (W + 2 * pad - R) // stride + 1
    y = torch.empty((N, P, Q, C), dtype=x.dtype, device=x.device)
    _check(lib.npas_maxpool2d(N, H, W, C, R, stride, pad, _p(x), _p(y), _stream()), "npas_maxpool2d")
    return y


def conv2d_bp_maxpool(x: torch.Tensor, blob: BpBlob, bias=None, *, stride=1, pad=1, relu=True, pool=(3, 2, 1), out=None,
                      ws=None, path=0) -> torch.Tensor:
    """npas_conv2d_bp_maxpool: convolution + bias + ReLU + max-pool fused in one kernel; returns the pooled
    NHWC tensor.  Raises NpasError(8) where no kernel has the fused epilogue (run the two calls then)."""
    if _host is None:
        load()
    pr, ps, pp = pool
    y = _host.conv2d_bp_maxpool(x, blob.data, blob.desc, bias, stride, pad, relu, pr, ps, pp, out, ws, path)
    return y if type(y) is not int else _refused(y, "npas_conv2d_bp_maxpool")


def conv2d_bp_static_ws(x: torch.Tensor, blob: BpBlob, bias=None, residual=None, *, stride=1, pad=1, relu=False,
                        out_dtype=None, out=None, path=0, check=True) -> torch.Tensor:
    """npas_conv2d_bp_static_ws: same result as ``conv2d_bp`` without caller-provided scratch.

    For callers that may not allocate device memory (fixed-budget or real-time inference loops,
    plug-ins whose host owns all allocations): the library's own 256-byte device array takes the
    place of the workspace.  ``out`` is still the caller's (this helper allocates it only when it
    is not passed).  With ``check`` the call synchronises and raises on a device-side time-out.
    """
    lib = load()
    assert x.is_cuda and x.is_contiguous() and x.dim() == 4
    N, H, W, C = x.shape
    d = blob.desc
    P = (H + 2 * pad - d.R) // stride + 1
    Q = (W + 2 * pad - d.S) // stride + 1
    if out is None:
        out = torch.empty((N, P, Q, d.K), dtype=x.dtype if out_dtype is None else out_dtype, device=x.device)
    cd = ConvDesc(N, H, W, C, d.K, d.R, d.S, stride, pad, _dt(x), _dt(out), int(bool(relu)),
                  int(bias is not None), int(residual is not None), path, 0)
    status = ctypes.c_int32(0)
    _check(lib.npas_conv2d_bp_static_ws(ctypes.byref(cd), ctypes.byref(d), _p(x), _p(blob.data), _p(bias),
                                        _p(residual), _p(out), ctypes.byref(status) if check else None, _stream()),
           "npas_conv2d_bp_static_ws")
    return out


# ---------------------------------------------------------------------------- kernel choice ----

CONV_KERNELS = {1: "conv_bp_simt_kernel", 3: "conv_bp_tc_kernel", 5: "conv_stem_kernel", 6: "conv_bp_dn_kernel",
                7: "conv_bp_d2_kernel", 8: "conv_bp_kr_kernel"}
LINEAR_KERNELS = {1: "linear_bb_simt_kernel", 3: "linear_bb_tc_kernel", 5: "linear_bb_dn_kernel", 6: "linear_bb_d2_kernel"}


def conv2d_bp_kernel(x_shape, blob: BpBlob, *, stride=1, pad=1, dtype=torch.bfloat16, out_dtype=None, relu=False,
                     bias=False, residual=False, path=0, variant=0) -> int:
    """npas_conv2d_bp_kernel: id of the kernel the call would run (host only; raises NpasError(8) when the
    requested path declines the geometry)."""
    lib = load()
    N, H, W, C = x_shape
    d = blob.desc
    t = torch.empty(0, dtype=dtype)
    to = t if out_dtype is None else torch.empty(0, dtype=out_dtype)
    cd = ConvDesc(N, H, W, C, d.K, d.R, d.S, stride, pad, _dt(t), _dt(to), int(bool(relu)), int(bool(bias)),
                  int(bool(residual)), path, variant)
    kid = ctypes.c_int32(0)
    _check(lib.npas_conv2d_bp_kernel(ctypes.byref(cd), ctypes.byref(d), ctypes.byref(kid)), "npas_conv2d_bp_kernel")
    return kid.value


def conv2d_bp_workspace(x_shape, blob: BpBlob, *, stride=1, pad=1, dtype=torch.bfloat16, out_dtype=None, relu=False,
                        bias=False, residual=False, path=0, variant=0, device="cuda") -> torch.Tensor:
    """npas_conv2d_bp_workspace: zeroed device scratch of the size the call needs for this layer (the status words)."""
    lib = load()
    N, H, W, C = x_shape
    d = blob.desc
    t = torch.empty(0, dtype=dtype)
    to = t if out_dtype is None else torch.empty(0, dtype=out_dtype)
    cd = ConvDesc(N, H, W, C, d.K, d.R, d.S, stride, pad, _dt(t), _dt(to), int(bool(relu)), int(bool(bias)),
                  int(bool(residual)), path, variant)
    n = ctypes.c_size_t(0)
    _check(lib.npas_conv2d_bp_workspace(ctypes.byref(cd), ctypes.byref(d), ctypes.byref(n)), "npas_conv2d_bp_workspace")
    return torch.zeros(max(n.value, WORKSPACE_BYTES), dtype=torch.uint8, device=device)


def linear_bb_kernel(M: int, blob: BbBlob, *, dtype=torch.bfloat16, out_dtype=None, relu=False, bias=False,
                     residual=False, path=0, variant=0) -> int:
    lib = load()
    d = blob.desc
    t = torch.empty(0, dtype=dtype)
    to = t if out_dtype is None else torch.empty(0, dtype=out_dtype)
    ld = LinearDesc(M, d.I, d.O, _dt(t), _dt(to), int(bool(relu)), int(bool(bias)), int(bool(residual)), path, variant)
    kid = ctypes.c_int32(0)
    _check(lib.npas_linear_bb_kernel(ctypes.byref(ld), ctypes.byref(d), ctypes.byref(kid)), "npas_linear_bb_kernel")
    return kid.value


def tune_conv2d_bp(x: torch.Tensor, blob: BpBlob, bias=None, residual=None, *, stride=1, pad=1, relu=False,
                   out=None, ws=None, reps=10):
    """npas_tune_conv2d_bp: times every kernel / tile shape that takes the layer on these buffers and returns
    (path, variant, microseconds) of the fastest; pass the first two to ``conv2d_bp``."""
    lib = load()
    N, H, W, C = x.shape
    d = blob.desc
    P = (H + 2 * pad - d.R) // stride + 1
    Q = (W + 2 * pad - d.S) // stride + 1
    if out is None:
        out = torch.empty((N, P, Q, d.K), dtype=x.dtype, device=x.device)
    if ws is None:
        ws = workspace(x.device)
    cd = ConvDesc(N, H, W, C, d.K, d.R, d.S, stride, pad, _dt(x), _dt(out), int(bool(relu)),
                  int(bias is not None), int(residual is not None), 0, 0)
    path, variant, us = ctypes.c_int32(0), ctypes.c_int32(0), ctypes.c_float(0)
    _check(lib.npas_tune_conv2d_bp(ctypes.byref(cd), ctypes.byref(d), _p(x), _p(blob.data), _p(bias), _p(residual),
                                   _p(out), _p(ws), ctypes.c_size_t(ws.numel()), int(reps), ctypes.byref(path),
                                   ctypes.byref(variant), ctypes.byref(us), _stream()), "npas_tune_conv2d_bp")
    return path.value, variant.value, us.value


def tune_linear_bb(x: torch.Tensor, blob: BbBlob, bias=None, residual=None, *, relu=False, out=None, ws=None, reps=10):
    lib = load()
    M, I = x.shape
    d = blob.desc
    if out is None:
        out = torch.empty((M, d.O), dtype=x.dtype, device=x.device)
    if ws is None:
        ws = workspace(x.device)
    ld = LinearDesc(M, I, d.O, _dt(x), _dt(out), int(bool(relu)), int(bias is not None), int(residual is not None), 0, 0)
    path, variant, us = ctypes.c_int32(0), ctypes.c_int32(0), ctypes.c_float(0)
    _check(lib.npas_tune_linear_bb(ctypes.byref(ld), ctypes.byref(d), _p(x), _p(blob.data), _p(bias), _p(residual),
                                   _p(out), _p(ws), ctypes.c_size_t(ws.numel()), int(reps), ctypes.byref(path),
                                   ctypes.byref(variant), ctypes.byref(us), _stream()), "npas_tune_linear_bb")
    return path.value, variant.value, us.value


def tune_linear_two(x: torch.Tensor, blob1: BbBlob, bias1, residual, blob2: BbBlob, bias2, *, relu, plans=((0, 0), (0, 0)), ws=None, reps=10):
    """Two GEMMs behind one another, the second on the first one's result: measures them as one launch and one by one on their
    ``plans``.  (True where one launch is the faster way, microseconds of the faster way), or None where there is no such launch."""
    lib = load()
    M, I = x.shape
    d1, d2 = blob1.desc, blob2.desc
    a = LinearDesc(M, I, d1.O, BF16, BF16, int(bool(relu[0])), int(bias1 is not None), int(residual is not None), *plans[0])
    b = LinearDesc(M, d1.O, d2.O, BF16, BF16, int(bool(relu[1])), int(bias2 is not None), 0, *plans[1])
    if ws is None:
        ws = workspace(x.device)
    y1, y2 = (torch.empty((M, d.O), dtype=torch.bfloat16, device=x.device) for d in (d1, d2))
    together, us = ctypes.c_int32(0), ctypes.c_float(0)
    code = lib.npas_internal_tune_linear_two(ctypes.byref(a), ctypes.byref(d1), ctypes.byref(b), ctypes.byref(d2), _p(x), _p(blob1.data), _p(bias1), _p(residual),
                                             _p(y1), _p(blob2.data), _p(bias2), _p(y2), _p(ws), ctypes.c_size_t(ws.numel()), int(reps), ctypes.byref(together),
                                             ctypes.byref(us), _stream())
    if code == 8:                                # NPAS_ERR_UNSUPPORTED
        return None
    _check(code, "npas_internal_tune_linear_two")
    return bool(together.value), us.value


class PlanCache:
    """Tuned (path, variant) pairs keyed by what the choice depends on: the call geometry, the block
    sizes and the mask statistic the kernels plan with (largest kept count of a block).  Plain JSON on
    disk, so a tuning run on one process serves later ones on the same GPU model."""

    def __init__(self):
        self.plans = {}

    @staticmethod
    def conv_key(x_shape, blob: BpBlob, stride, pad, relu, has_bias, has_residual) -> str:
        d = blob.desc
        return "conv:" + ",".join(str(int(v)) for v in (*x_shape, d.K, d.R, d.S, d.Mb, d.Nb, d.max_taps, stride, pad,
                                                         relu, has_bias, has_residual))

    @staticmethod
    def linear_key(M, blob: BbBlob, relu, has_bias, has_residual) -> str:
        d = blob.desc
        return "linear:" + ",".join(str(int(v)) for v in (M, d.I, d.O, d.Bo, d.Bi, d.max_cols, relu, has_bias, has_residual))

    @staticmethod
    def two_key(first: str, second: str) -> str:
        """Two GEMMs behind one another, by their own keys; the plan is (2, 0) in one launch, (1, 0) one by one."""
        return f"two:{first}|{second}"

    def get(self, key: str):
        v = self.plans.get(key)
        return None if v is None else (int(v[0]), int(v[1]))

    def put(self, key: str, path: int, variant: int, us: float) -> None:
        self.plans[key] = [int(path), int(variant), round(float(us), 3)]

    def to_json(self) -> str:
        import json
        return json.dumps({"version": 1, "plans": self.plans}, sort_keys=True)

    @classmethod
    def from_json(cls, text: str) -> "PlanCache":
        import json
        obj = json.loads(text)
        if obj.get("version") != 1 or not isinstance(obj.get("plans"), dict):
            raise ValueError("not a plan cache")
        c = cls()
        for k, v in obj["plans"].items():
            if not (isinstance(v, list) and len(v) == 3):
                raise ValueError(f"bad plan entry {k!r}")
            c.plans[str(k)] = [int(v[0]), int(v[1]), float(v[2])]
        return c
