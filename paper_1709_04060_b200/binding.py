"""Binding of the C ABI in ``include/qnn.h`` (argument marshalling only): ctypes, and for the calls that
launch kernels an extension module (``csrc/fastcall.c``) in front of it.

The ``qnn_*`` functions mirror the C entry points one to one and return the
status code.  Pointer arguments accept a ``torch.Tensor`` (its ``data_ptr()``
is passed; the tensor must be contiguous and live on the GPU), an ``int``
address, or ``None``.  ``stream=None`` means torch's current CUDA stream.

The helpers below them (``pack``, ``qgemm``, ``qconv``, ...) only allocate the
output tensor with torch, build the descriptor and call the entry point; every
step of the computation runs in the library's kernels.  There is no fallback:
if the shared library is missing, importing this module raises.
"""
import ctypes
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libqnn_b200.so")

if not os.path.exists(LIB_PATH):
    raise ImportError(
        f"{LIB_PATH} not found: build it with `python -m paper_1709_04060_b200.build` "
        "(there is no CPU fallback)")
_lib = ctypes.CDLL(LIB_PATH)

QNN_OK = 0
QNN_ERR_INVALID_ARG, QNN_ERR_UNSUPPORTED, QNN_ERR_ALIGNMENT = -1, -2, -3
QNN_ERR_WORKSPACE, QNN_ERR_CUDA, QNN_ERR_DEVICE_TIMEOUT = -4, -5, -6
QNN_ENC_UNSIGNED, QNN_ENC_SIGNED, QNN_ENC_BIPOLAR = 0, 1, 2
QNN_FMT_BITPLANES, QNN_FMT_INT8, QNN_FMT_FIELDS = 0, 1, 2
QNN_PATH_AUTO, QNN_PATH_BITSERIAL, QNN_PATH_TCGEN05_I8 = 0, 1, 2

EXPORTS = (
    "qnn_packed_ld", "qnn_packed_bytes", "qnn_pack", "qnn_planes_to_int8", "qnn_gemm_workspace_bytes",
    "qnn_gemm_out_bytes", "qnn_qgemm", "qnn_qgemm_kernel", "qnn_qgemm_kernel_name", "qnn_conv_out_h", "qnn_conv_out_w",
    "qnn_conv_lowered_k", "qnn_conv_lowered_bytes", "qnn_conv_workspace_bytes",
    "qnn_conv_out_bytes", "qnn_im2col", "qnn_qconv", "qnn_conv_boxes", "qnn_conv_in_place", "qnn_conv_maxpool_fuses", "qnn_qconv_maxpool", "qnn_qconv_static", "qnn_maxpool",
    "qnn_streamline", "qnn_peak_mma_i8", "qnn_peak_popc", "qnn_peak_popc_sink_bytes", "qnn_validate_thresholds", "qnn_device_status", "qnn_launch_count",
    "qnn_status_string", "qnn_version",
)


class qnn_pack_desc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("rows", "K", "bits", "enc", "fmt")]


class qnn_gemm_desc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in (
        "M", "N", "K", "w_bits", "a_bits", "out_bits", "w_enc", "a_enc",
        "w_fmt", "a_fmt", "out_fmt", "path", "skip_planes")]


class qnn_conv_desc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in (
        "B", "H", "W", "C", "in_pitch", "OC", "KH", "KW", "stride", "pad",
        "w_bits", "a_bits", "out_bits", "w_enc", "a_enc", "fmt", "out_fmt", "path")]


class qnn_channel_params(ctypes.Structure):
    _fields_ = [(n, ctypes.c_double) for n in ("a_prev", "b_prev", "alpha", "gamma", "beta", "mu", "sigma")] + \
               [("row_sum", ctypes.c_longlong)]


class qnn_pool_desc(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("B", "H", "W", "C", "k", "stride", "bits", "fmt")]


_vp, _sz, _ci = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
_P = ctypes.POINTER
_lib.qnn_packed_ld.restype = _sz
_lib.qnn_packed_ld.argtypes = [_ci, _ci]
_lib.qnn_packed_bytes.restype = _sz
_lib.qnn_packed_bytes.argtypes = [_P(qnn_pack_desc)]
_lib.qnn_pack.restype = _ci
_lib.qnn_pack.argtypes = [_P(qnn_pack_desc), _vp, _vp, _vp]
_lib.qnn_planes_to_int8.argtypes = [_P(qnn_pack_desc), _vp, _vp, _vp]
_lib.qnn_planes_to_int8.restype = _ci
_lib.qnn_gemm_workspace_bytes.restype = _sz
_lib.qnn_gemm_workspace_bytes.argtypes = [_P(qnn_gemm_desc)]
_lib.qnn_gemm_out_bytes.restype = _sz
_lib.qnn_gemm_out_bytes.argtypes = [_P(qnn_gemm_desc), _ci]
_lib.qnn_qgemm_kernel.restype = _ci
_lib.qnn_qgemm_kernel.argtypes = [_P(qnn_gemm_desc), _ci]
_lib.qnn_qgemm_kernel_name.restype = ctypes.c_char_p
_lib.qnn_qgemm_kernel_name.argtypes = [_P(qnn_gemm_desc), _ci]
_lib.qnn_qgemm.restype = _ci
_lib.qnn_qgemm.argtypes = [_P(qnn_gemm_desc), _vp, _vp, _vp, _vp, _vp, _sz, _vp]
for _n in ("qnn_conv_out_h", "qnn_conv_out_w", "qnn_conv_lowered_k"):
    getattr(_lib, _n).restype = _ci
    getattr(_lib, _n).argtypes = [_P(qnn_conv_desc)]
for _n in ("qnn_conv_lowered_bytes", "qnn_conv_workspace_bytes"):
    getattr(_lib, _n).restype = _sz
    getattr(_lib, _n).argtypes = [_P(qnn_conv_desc)]
_lib.qnn_conv_out_bytes.restype = _sz
_lib.qnn_conv_out_bytes.argtypes = [_P(qnn_conv_desc), _ci]
_lib.qnn_im2col.restype = _ci
_lib.qnn_im2col.argtypes = [_P(qnn_conv_desc), _vp, _vp, _vp]
_lib.qnn_qconv.restype = _ci
_lib.qnn_qconv.argtypes = [_P(qnn_conv_desc), _vp, _vp, _vp, _vp, _vp, _sz, _vp]
_lib.qnn_conv_boxes.restype = _ci
_lib.qnn_conv_boxes.argtypes = [_P(qnn_conv_desc), _ci, _P(_ci), _P(_ci), _P(_ci)]
_lib.qnn_conv_in_place.restype = _ci
_lib.qnn_conv_in_place.argtypes = [_P(qnn_conv_desc), _ci]
_lib.qnn_conv_maxpool_fuses.restype = _ci
_lib.qnn_conv_maxpool_fuses.argtypes = [_P(qnn_conv_desc), _ci, _ci]
_lib.qnn_qconv_maxpool.restype = _ci
_lib.qnn_qconv_maxpool.argtypes = [_P(qnn_conv_desc), _ci, _ci, _vp, _vp, _vp, _vp, _vp]
_lib.qnn_qconv_static.restype = _ci
_lib.qnn_qconv_static.argtypes = [_P(qnn_conv_desc), _vp, _vp, _vp, _vp, _vp]
_lib.qnn_maxpool.restype = _ci
_lib.qnn_maxpool.argtypes = [_P(qnn_pool_desc), _vp, _vp, _vp]
_lib.qnn_streamline.restype = _ci
_lib.qnn_streamline.argtypes = [_P(qnn_channel_params), _ci, _P(ctypes.c_double), _ci, ctypes.c_longlong,
                                ctypes.c_longlong, _P(ctypes.c_int32), _P(ctypes.c_uint8)]
_lib.qnn_peak_mma_i8.restype = _ci
_lib.qnn_peak_mma_i8.argtypes = [_ci, _ci, _ci, _P(ctypes.c_double), _vp]
_lib.qnn_peak_popc.restype = _ci
_lib.qnn_peak_popc.argtypes = [_ci, _vp, _sz, _P(ctypes.c_double), _vp]
_lib.qnn_peak_popc_sink_bytes.restype = _sz
_lib.qnn_peak_popc_sink_bytes.argtypes = []
_lib.qnn_validate_thresholds.restype = _ci
_lib.qnn_validate_thresholds.argtypes = [_vp, _ci, _ci, _P(_ci), _vp]
_lib.qnn_device_status.restype = _ci
_lib.qnn_device_status.argtypes = [_P(_ci)]
_lib.qnn_launch_count.restype = ctypes.c_ulonglong
_lib.qnn_launch_count.argtypes = []
_lib.qnn_status_string.restype = ctypes.c_char_p
_lib.qnn_status_string.argtypes = [_ci]
_lib.qnn_version.restype = _ci
_lib.qnn_version.argtypes = []


class QnnError(RuntimeError):
    def __init__(self, status):
        self.status = status
        super().__init__(f"qnn status {status}: {qnn_status_string(status)}")


def check(status: int) -> None:
    if status != QNN_OK:
        raise QnnError(status)


def _ptr(x):
    if x is None:
        return None
    if isinstance(x, _Tensor):
        assert x.is_contiguous(), "device buffers must be contiguous"
        return x.data_ptr()
    if isinstance(x, int):
        return x
    raise TypeError(type(x))


_Tensor = torch.Tensor
# The current stream's handle without building a torch.cuda.Stream around it (0.2 us
# instead of 3.5 us a call), where this build of torch has these two functions: without
# them the library can still be imported and queried on the host.
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)
_device = getattr(torch._C, "_cuda_getDevice", None)


def _stream(stream):
    if stream is None:
        if _raw_stream is None or _device is None or not _initialized():
            return torch.cuda.current_stream().cuda_stream
        return _raw_stream(_device())
    return int(stream)


_initialized = torch.cuda.is_initialized

try:
    from . import _fastcall
except ImportError:              # a tree whose extension is not built: the same calls through ctypes
    _fastcall = None


def _entry(name, kinds, desc_type):
    """The entry point ``name`` as a callable; kinds of its arguments: d descriptor, p pointer, n number,
    s stream.  The extension takes the plain forms (0.8 us of host time instead of 2.2) and hands every
    other one to the ctypes call below."""
    fn = getattr(_lib, name)
    convert = [{"d": ctypes.byref, "p": _ptr, "n": lambda x: x, "s": _stream}[k] for k in kinds]

    def slow(*args):
        return fn(*[c(x) for c, x in zip(convert, args)])

    if _fastcall is None:
        return slow
    return _fastcall.bind(ctypes.cast(fn, _vp).value, kinds, desc_type, _Tensor, slow, _raw_stream, _device, _initialized)


_pack = _entry("qnn_pack", "dpps", qnn_pack_desc)
_planes_to_int8 = _entry("qnn_planes_to_int8", "dpps", qnn_pack_desc)
_qgemm = _entry("qnn_qgemm", "dpppppns", qnn_gemm_desc)
_im2col = _entry("qnn_im2col", "dpps", qnn_conv_desc)
_qconv = _entry("qnn_qconv", "dpppppns", qnn_conv_desc)
_qconv_maxpool = _entry("qnn_qconv_maxpool", "dnnpppps", qnn_conv_desc)
_qconv_static = _entry("qnn_qconv_static", "dpppps", qnn_conv_desc)
_maxpool = _entry("qnn_maxpool", "dpps", qnn_pool_desc)


# ---- one-to-one entry points -------------------------------------------------
def qnn_version() -> int:
    return _lib.qnn_version()


def qnn_status_string(s: int) -> str:
    return _lib.qnn_status_string(s).decode()


def qnn_launch_count() -> int:
    return int(_lib.qnn_launch_count())


def qnn_packed_ld(K: int, fmt: int) -> int:
    return int(_lib.qnn_packed_ld(K, fmt))


def qnn_packed_bytes(d: qnn_pack_desc) -> int:
    return int(_lib.qnn_packed_bytes(ctypes.byref(d)))


def qnn_pack(d, logical, packed, stream=None) -> int:
    return _pack(d, logical, packed, stream)


def qnn_planes_to_int8(d, planes, containers, stream=None) -> int:
    return _planes_to_int8(d, planes, containers, stream)


def qnn_gemm_workspace_bytes(d) -> int:
    return int(_lib.qnn_gemm_workspace_bytes(ctypes.byref(d)))


def qnn_gemm_out_bytes(d, has_thresholds: bool) -> int:
    return int(_lib.qnn_gemm_out_bytes(ctypes.byref(d), int(has_thresholds)))


QNN_KERNEL_TENSOR, QNN_KERNEL_TENSOR_CTA_PAIR, QNN_KERNEL_BYTES_FEW_COLUMNS = 1, 2, 3
QNN_KERNEL_PLANES_FEW_COLUMNS, QNN_KERNEL_PLANES_TILED, QNN_KERNEL_FIELDS_FEW_COLUMNS = 4, 5, 6


def qnn_qgemm_kernel(d, has_thresholds: bool = True) -> int:
    """The kind of kernel qnn_qgemm would run for this problem (a QNN_KERNEL_* value, or a negative status)."""
    return _lib.qnn_qgemm_kernel(ctypes.byref(d), int(has_thresholds))


def qnn_qgemm_kernel_name(d, has_thresholds: bool = True):
    """The name of the kernel function qnn_qgemm would run for this problem, None where it would refuse it."""
    name = _lib.qnn_qgemm_kernel_name(ctypes.byref(d), int(has_thresholds))
    return None if name is None else name.decode()


def qnn_qgemm(d, W, A, thr, out, workspace=None, workspace_bytes=0, stream=None) -> int:
    return _qgemm(d, W, A, thr, out, workspace, workspace_bytes, stream)


def qnn_conv_out_h(d) -> int:
    return _lib.qnn_conv_out_h(ctypes.byref(d))


def qnn_conv_out_w(d) -> int:
    return _lib.qnn_conv_out_w(ctypes.byref(d))


def qnn_conv_lowered_k(d) -> int:
    return _lib.qnn_conv_lowered_k(ctypes.byref(d))


def qnn_conv_lowered_bytes(d) -> int:
    return int(_lib.qnn_conv_lowered_bytes(ctypes.byref(d)))


def qnn_conv_workspace_bytes(d) -> int:
    return int(_lib.qnn_conv_workspace_bytes(ctypes.byref(d)))


def qnn_conv_out_bytes(d, has_thresholds: bool) -> int:
    return int(_lib.qnn_conv_out_bytes(ctypes.byref(d), int(has_thresholds)))


def qnn_im2col(d, inp, lowered, stream=None) -> int:
    return _im2col(d, inp, lowered, stream)


def qnn_qconv(d, Wpacked, inp, thr, out, workspace, workspace_bytes, stream=None) -> int:
    return _qconv(d, Wpacked, inp, thr, out, workspace, workspace_bytes, stream)


def qnn_conv_boxes(d, has_thresholds: bool = True):
    """Boxes of output pixels that the CTA-pair kernel cuts this layer into: (number, width, height, images), or
    None where it takes consecutive pixels or another kernel takes the layer."""
    w, h, n = _ci(), _ci(), _ci()
    boxes = _lib.qnn_conv_boxes(ctypes.byref(d), int(has_thresholds), ctypes.byref(w), ctypes.byref(h), ctypes.byref(n))
    return (boxes, w.value, h.value, n.value) if boxes else None


def qnn_conv_in_place(d, has_thresholds: bool = True) -> bool:
    """Whether qnn_qconv reads the rows of this three-channel map in place."""
    return bool(_lib.qnn_conv_in_place(ctypes.byref(d), int(has_thresholds)))


def qnn_conv_maxpool_fuses(d, k: int, stride: int) -> bool:
    """Whether qnn_qconv_maxpool takes this layer with this pool."""
    return bool(_lib.qnn_conv_maxpool_fuses(ctypes.byref(d), k, stride))


def qnn_qconv_maxpool(d, k: int, stride: int, Wpacked, inp, thr, out, stream=None) -> int:
    return _qconv_maxpool(d, k, stride, Wpacked, inp, thr, out, stream)


QNN_QCONV_STATIC_MAX_BYTES = 16 << 20


def qnn_qconv_static(d, Wpacked, inp, thr, out, stream=None) -> int:
    """qnn_qconv without a workspace argument: the lowered matrix goes into a fixed
    array inside the library, so the call allocates nothing (see include/qnn.h)."""
    return _qconv_static(d, Wpacked, inp, thr, out, stream)


def qnn_maxpool(d, inp, out, stream=None) -> int:
    return _maxpool(d, inp, out, stream)


def qnn_streamline(channels, qthr, acc_lo: int, acc_hi: int):
    """Host-only.  channels: sequence of qnn_channel_params (or 8-tuples in field order);
    qthr: the quantizer's float thresholds.  Returns (status, thresholds [channels][n_thr] as
    nested lists of ints, negate flags)."""
    arr = (qnn_channel_params * len(channels))(*[c if isinstance(c, qnn_channel_params) else qnn_channel_params(*c)
                                                  for c in channels])
    n = len(qthr)
    q = (ctypes.c_double * n)(*[float(t) for t in qthr])
    out = (ctypes.c_int32 * (len(channels) * n))()
    neg = (ctypes.c_uint8 * len(channels))()
    st = _lib.qnn_streamline(arr, len(channels), q, n, int(acc_lo), int(acc_hi), out, neg)
    thr = [[out[c * n + i] for i in range(n)] for c in range(len(channels))]
    return st, thr, [int(v) for v in neg]


def qnn_peak_mma_i8(pair: int, n: int, mmas_per_cta: int, stream=None):
    """Launches the tensor-pipe issue-rate microbenchmark; returns (status, integer ops of the launch)."""
    ops = ctypes.c_double(0.0)
    st = _lib.qnn_peak_mma_i8(int(pair), int(n), int(mmas_per_cta), ctypes.byref(ops), _stream(stream))
    return st, ops.value


def qnn_peak_popc_sink_bytes() -> int:
    return int(_lib.qnn_peak_popc_sink_bytes())


def qnn_peak_popc(iters: int, sink, stream=None):
    """Launches the POPC issue-rate microbenchmark; returns (status, population counts of the launch)."""
    n = ctypes.c_double(0.0)
    st = _lib.qnn_peak_popc(int(iters), _ptr(sink), sink.numel() * sink.element_size(), ctypes.byref(n),
                            _stream(stream))
    return st, n.value


def qnn_validate_thresholds(thr, M: int, n_thr: int, stream=None):
    """Returns (status, number of unsorted rows).  Synchronises the stream."""
    n_bad = _ci(0)
    st = _lib.qnn_validate_thresholds(_ptr(thr), M, n_thr, ctypes.byref(n_bad), _stream(stream))
    return st, n_bad.value


def qnn_device_status():
    """Returns (status, device status word).  Synchronises the device."""
    v = _ci(0)
    st = _lib.qnn_device_status(ctypes.byref(v))
    return st, v.value


# ---- allocation helpers (marshalling only) -----------------------------------
def _dev_bytes(n: int) -> torch.Tensor:
    return torch.empty(max(int(n), 16), dtype=torch.uint8, device="cuda")


def _scratch(n: int, stream, zeroed: bool = False) -> torch.Tensor:
    """Workspace of one call on ``stream``: allocated (and cleared) there, so that its memory is handed out
    again only behind the call, whichever stream is the current one."""
    if stream is None:
        return torch.zeros(n, dtype=torch.uint8, device="cuda") if zeroed else _dev_bytes(n)
    with torch.cuda.stream(torch.cuda.ExternalStream(int(stream))):
        return _scratch(n, None, zeroed)


def to_device_logical(x, enc: int) -> torch.Tensor:
    """numpy/torch logical integers -> contiguous device bytes (uint8 for
    UNSIGNED, int8 otherwise), the packer's input format."""
    t = torch.as_tensor(x)
    t = t.to(torch.uint8 if enc == QNN_ENC_UNSIGNED else torch.int8)
    return t.contiguous().cuda()


def pack(logical: torch.Tensor, bits: int, enc: int, fmt: int, stream=None) -> torch.Tensor:
    """Pack a [rows][K] device byte matrix; returns the packed device buffer (uint8 view)."""
    rows, K = logical.shape
    d = qnn_pack_desc(rows, K, bits, enc, fmt)
    out = _dev_bytes(qnn_packed_bytes(d))
    check(qnn_pack(d, logical, out, stream))
    return out


def gemm_desc(M, N, K, w_bits, a_bits, out_bits, w_enc, a_enc, fmt, out_fmt,
              path=QNN_PATH_AUTO, skip_planes=0) -> qnn_gemm_desc:
    return qnn_gemm_desc(M, N, K, w_bits, a_bits, out_bits, w_enc, a_enc, fmt, fmt, out_fmt, path, skip_planes)


def qgemm(d: qnn_gemm_desc, W, A, thr, out=None, stream=None) -> torch.Tensor:
    """Fused GEMM + threshold; returns the output buffer (uint8 view, or int32
    [N][M] when thr is None)."""
    if out is None:
        out = _dev_bytes(qnn_gemm_out_bytes(d, thr is not None))
    # the optional workspace starts with flag words that must be zero before the first call
    ws_bytes = qnn_gemm_workspace_bytes(d)
    ws = _scratch(ws_bytes, stream, zeroed=True) if ws_bytes else None
    check(qnn_qgemm(d, W, A, thr, out, ws, ws_bytes, stream))
    if thr is None:
        return out[: d.N * d.M * 4].view(torch.int32).view(d.N, d.M)
    return out


def conv_weight_rows(d: qnn_conv_desc, Wt):
    """Logical filters [OC][KH][KW][C] (numpy) laid out as the rows [OC][qnn_conv_lowered_k]
    that `pack` expects for this convolution: per-pixel padding to 32 channels for bit planes,
    per-filter-row padding to 16 bytes for 8-bit maps whose C is not a multiple of 16."""
    import numpy as np
    OC, KH, KW, C = Wt.shape
    K = qnn_conv_lowered_k(d)
    if d.fmt == QNN_FMT_BITPLANES:
        cp = (C + 31) // 32 * 32
        rows = np.zeros((OC, KH * KW, cp), dtype=Wt.dtype)
        rows[:, :, :C] = Wt.reshape(OC, KH * KW, C)
    elif C % 16 == 0:
        rows = Wt
    else:
        rows = np.zeros((OC, KH, K // KH), dtype=Wt.dtype)
        rows[:, :, :KW * C] = Wt.reshape(OC, KH, KW * C)
    return np.ascontiguousarray(rows.reshape(OC, K))


def qconv(d: qnn_conv_desc, Wpacked, inp, thr, out=None, workspace=None, stream=None) -> torch.Tensor:
    if out is None:
        out = _dev_bytes(qnn_conv_out_bytes(d, thr is not None))
    ws_bytes = qnn_conv_workspace_bytes(d)
    if workspace is None:
        workspace = _scratch(ws_bytes, stream)
    check(qnn_qconv(d, Wpacked, inp, thr, out, workspace, workspace.numel(), stream))
    return out
