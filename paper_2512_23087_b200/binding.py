"""ctypes binding of the C ABI in ``include/dvp.h``.

Argument marshalling only: tensors are turned into raw device pointers and
sizes, outputs are allocated with torch, and every step of the computation
runs in the CUDA library.  There is no fallback: if ``libdvp_b200.so`` has not
been built, the first call raises.
"""
from __future__ import annotations

import contextlib
import ctypes
import os
import struct
from types import SimpleNamespace

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libdvp_b200.so")
BOUNDS_LIB_PATH = os.path.join(_HERE, "libdvp_b200_bounds.so")   # the bounds-checking build

DVP_OK, DVP_ERR_INVALID_ARG, DVP_ERR_UNSUPPORTED, DVP_ERR_WORKSPACE, DVP_ERR_CUDA = range(5)
DVP_F32, DVP_BF16, DVP_F16 = 0, 1, 2
DVP_ID_I64, DVP_ID_I32 = 0, 1
DVP_FLAG_IN_TRAIN, DVP_FLAG_IN_INFER, DVP_FLAG_NO_ID, DVP_FLAG_BAD_ID = 1, 2, 64, 128
DVP_ENTRY_FORWARD, DVP_ENTRY_BACKWARD, DVP_ENTRY_FUSED_LMHEAD = 0, 1, 2
DVP_STATIC_WORKSPACE_BYTES = 32 * 1024 * 1024
DVP_MODE_FINITE_MASK, DVP_MODE_THRESHOLD_IN_LOGITS_DTYPE = 1, 2
DVP_WEIGHT_NONE, DVP_WEIGHT_RATIO, DVP_WEIGHT_TRUNCATE, DVP_WEIGHT_MASK = 0, 1, 2, 3

EXPORTS = ("dvp_forward", "dvp_backward", "dvp_fused_lmhead_forward_backward",
           "dvp_fused_lmhead_forward_backward_static", "dvp_sequence_aggregate", "dvp_monitor", "dvp_gemm_tn",
           "dvp_workspace_bytes", "dvp_status_string", "dvp_version", "dvp_row_wait_status",
           "dvp_static_workspace_status", "dvp_debug_bounds_status")

_DTYPES = {torch.float32: DVP_F32, torch.bfloat16: DVP_BF16, torch.float16: DVP_F16}
_SIDE_FIELDS = ("max", "lse", "lse_safe", "logp", "logp_mp", "comp_mp", "count", "mask", "log_cov")


class DvpError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} ({status})")


class SideOut(ctypes.Structure):
    _fields_ = [(n, ctypes.c_void_p) for n in _SIDE_FIELDS]


class ForwardArgs(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("logits_dtype", ctypes.c_int32),
        ("grad_dtype", ctypes.c_int32),
        ("id_dtype", ctypes.c_int32),
        ("T", ctypes.c_int64),
        ("V", ctypes.c_int64),
        ("ld_train", ctypes.c_int64),
        ("ld_infer", ctypes.c_int64),
        ("ld_grad", ctypes.c_int64),
        ("rho", ctypes.c_double),
        ("train_logits", ctypes.c_void_p),
        ("infer_logits", ctypes.c_void_p),
        ("ids", ctypes.c_void_p),
        ("upstream", ctypes.c_void_p),
        ("grad_train", ctypes.c_void_p),
        ("train", SideOut),
        ("infer", SideOut),
        ("log_ratio", ctypes.c_void_p),
        ("flags", ctypes.c_void_p),
        ("stream", ctypes.c_void_p),
        ("launch_hint", ctypes.c_uint32),
        ("mode", ctypes.c_uint32),
        ("mask_value", ctypes.c_float),
        ("weight_kind", ctypes.c_uint32),
        ("weight_lo", ctypes.c_float),
        ("weight_hi", ctypes.c_float),
        ("weight_out", ctypes.c_void_p),
    ]


class BackwardArgs(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("logits_dtype", ctypes.c_int32),
        ("grad_dtype", ctypes.c_int32),
        ("id_dtype", ctypes.c_int32),
        ("T", ctypes.c_int64),
        ("V", ctypes.c_int64),
        ("ld_train", ctypes.c_int64),
        ("ld_grad", ctypes.c_int64),
        ("rho", ctypes.c_double),
        ("train_logits", ctypes.c_void_p),
        ("ids", ctypes.c_void_p),
        ("upstream", ctypes.c_void_p),
        ("max_t", ctypes.c_void_p),
        ("lse_safe_t", ctypes.c_void_p),
        ("comp_mp_t", ctypes.c_void_p),
        ("flags", ctypes.c_void_p),
        ("grad_train", ctypes.c_void_p),
        ("stream", ctypes.c_void_p),
        ("launch_hint", ctypes.c_uint32),
        ("mode", ctypes.c_uint32),
        ("mask_value", ctypes.c_float),
        ("reserved_", ctypes.c_uint32),
    ]


class FusedArgs(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("id_dtype", ctypes.c_int32),
        ("T", ctypes.c_int64),
        ("H", ctypes.c_int64),
        ("V", ctypes.c_int64),
        ("ld_hidden", ctypes.c_int64),
        ("ld_w", ctypes.c_int64),
        ("ld_infer", ctypes.c_int64),
        ("ld_dh", ctypes.c_int64),
        ("ld_dw", ctypes.c_int64),
        ("rho", ctypes.c_double),
        ("hidden", ctypes.c_void_p),
        ("w_vocab", ctypes.c_void_p),
        ("infer_logits", ctypes.c_void_p),
        ("ids", ctypes.c_void_p),
        ("upstream", ctypes.c_void_p),
        ("d_hidden", ctypes.c_void_p),
        ("d_w", ctypes.c_void_p),
        ("accumulate_dw", ctypes.c_int32),
        ("panel_rows", ctypes.c_int32),
        ("train", SideOut),
        ("infer", SideOut),
        ("log_ratio", ctypes.c_void_p),
        ("flags", ctypes.c_void_p),
        ("workspace", ctypes.c_void_p),
        ("workspace_bytes", ctypes.c_size_t),
        ("stream", ctypes.c_void_p),
        ("weight_kind", ctypes.c_uint32),
        ("weight_lo", ctypes.c_float),
        ("weight_hi", ctypes.c_float),
        ("weight_out", ctypes.c_void_p),
    ]


class SequenceArgs(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("reserved_", ctypes.c_uint32),
        ("T", ctypes.c_int64),
        ("S", ctypes.c_int64),
        ("seq_offsets", ctypes.c_void_p),
        ("log_ratio", ctypes.c_void_p),
        ("veto_threshold", ctypes.c_double),
        ("seq_log_ratio", ctypes.c_void_p),
        ("min_log_ratio", ctypes.c_void_p),
        ("n_valid", ctypes.c_void_p),
        ("n_zero_weight", ctypes.c_void_p),
        ("veto", ctypes.c_void_p),
        ("stream", ctypes.c_void_p),
        ("log_cov", ctypes.c_void_p),
        ("min_cov", ctypes.c_void_p),
        ("mean_cov", ctypes.c_void_p),
    ]


class MonitorArgs(ctypes.Structure):
    _fields_ = [
        ("struct_size", ctypes.c_uint32),
        ("logits_dtype", ctypes.c_int32),
        ("T", ctypes.c_int64),
        ("V", ctypes.c_int64),
        ("ld_train", ctypes.c_int64),
        ("ld_infer", ctypes.c_int64),
        ("train_logits", ctypes.c_void_p),
        ("infer_logits", ctypes.c_void_p),
        ("kl_infer_train", ctypes.c_void_p),
        ("kl_train_infer", ctypes.c_void_p),
        ("entropy_train", ctypes.c_void_p),
        ("entropy_infer", ctypes.c_void_p),
        ("stream", ctypes.c_void_p),
    ]


# The hot entry points are called with their argument structs packed in one go: setting the fields of a ctypes
# structure one by one costs several microseconds a call.
_FORWARD_PACK = struct.Struct("=I3i5qd5Q18Q3QIIfIffQ")
_BACKWARD_PACK = struct.Struct("=I3i4qd9QIIfI")
_MONITOR_PACK = struct.Struct("=Ii4q7Q")
_SEQUENCE_PACK = struct.Struct("=II2q2Qd9Q")
_FUSED_PACK = struct.Struct("=Ii8qd7Qii18Q5QIff4xQ")
assert _FUSED_PACK.size == ctypes.sizeof(FusedArgs)
assert _FORWARD_PACK.size == ctypes.sizeof(ForwardArgs) and _BACKWARD_PACK.size == ctypes.sizeof(BackwardArgs)
assert _MONITOR_PACK.size == ctypes.sizeof(MonitorArgs) and _SEQUENCE_PACK.size == ctypes.sizeof(SequenceArgs)

_lib = None
_host = None


def load_library() -> ctypes.CDLL:
    """Load ``libdvp_b200.so``; raises if it is missing (there is no fallback)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2512_23087_b200.build`; "
                "this package has no CPU or PyTorch fallback")
        global _host
        try:
            from . import _host   # lays outputs over one allocation
        except ImportError as e:
            raise RuntimeError("the helper _host.so is missing or does not load: build it with "
                               "`python -m paper_2512_23087_b200.build`") from e
        from .build import host_target
        if getattr(_host, "built_for", None) != f"[built for {host_target()}]":
            raise RuntimeError(f"the helper _host.so was built for another interpreter or torch than {host_target()}: build "
                               "it with `python -m paper_2512_23087_b200.build`")
        lib = ctypes.CDLL(LIB_PATH)
        lib.dvp_forward.argtypes = [ctypes.POINTER(ForwardArgs)]
        lib.dvp_forward.restype = ctypes.c_int
        lib.dvp_backward.argtypes = [ctypes.POINTER(BackwardArgs)]
        lib.dvp_backward.restype = ctypes.c_int
        lib.dvp_fused_lmhead_forward_backward.argtypes = [ctypes.POINTER(FusedArgs)]
        lib.dvp_fused_lmhead_forward_backward.restype = ctypes.c_int
        lib.dvp_fused_lmhead_forward_backward_static.argtypes = [ctypes.POINTER(FusedArgs)]
        lib.dvp_fused_lmhead_forward_backward_static.restype = ctypes.c_int
        lib.dvp_sequence_aggregate.argtypes = [ctypes.POINTER(SequenceArgs)]
        lib.dvp_sequence_aggregate.restype = ctypes.c_int
        lib.dvp_monitor.argtypes = [ctypes.POINTER(MonitorArgs)]
        lib.dvp_monitor.restype = ctypes.c_int
        lib.dvp_gemm_tn.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_int64,
                                    ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_int64,
                                    ctypes.c_int64, ctypes.c_int32, ctypes.c_float, ctypes.c_int32,
                                    ctypes.c_void_p, ctypes.c_void_p]
        lib.dvp_gemm_tn.restype = ctypes.c_int
        lib.dvp_workspace_bytes.argtypes = [ctypes.c_int, ctypes.c_void_p]
        lib.dvp_workspace_bytes.restype = ctypes.c_size_t
        lib.dvp_status_string.argtypes = [ctypes.c_int]
        lib.dvp_status_string.restype = ctypes.c_char_p
        lib.dvp_version.restype = ctypes.c_int
        lib.dvp_row_wait_status.argtypes = [ctypes.POINTER(ctypes.c_uint32)]
        lib.dvp_row_wait_status.restype = ctypes.c_int
        lib.dvp_static_workspace_status.argtypes = [ctypes.POINTER(ctypes.c_uint32)]
        lib.dvp_static_workspace_status.restype = ctypes.c_int
        lib.dvp_debug_bounds_status.argtypes = [ctypes.POINTER(ctypes.c_uint32)]
        lib.dvp_debug_bounds_status.restype = ctypes.c_int
        lib.packed = {}   # the entry points that take a packed struct
        for name in ("dvp_forward", "dvp_backward", "dvp_monitor", "dvp_sequence_aggregate"):
            fn = lib[name]   # a function object of its own, with its own argtypes
            fn.argtypes, fn.restype = [ctypes.c_char_p], ctypes.c_int
            lib.packed[name] = fn
        lib.forward_at = ctypes.cast(lib.dvp_forward, ctypes.c_void_p).value
        _lib = lib
    return _lib


@contextlib.contextmanager
def bounds_checking_library():
    """Inside the block every call of this module goes to the bounds-checking build of the
    library (``python -m paper_2512_23087_b200.build --debug-bounds``), whose kernels compare
    every index of their on-chip tables and every global offset with its extent;
    ``dvp_debug_bounds_status()`` then tells whether any check failed."""
    global _lib, LIB_PATH
    if not os.path.exists(BOUNDS_LIB_PATH):
        raise RuntimeError(f"{BOUNDS_LIB_PATH} is missing: build it with "
                           "`python -m paper_2512_23087_b200.build --debug-bounds`")
    saved = (_lib, LIB_PATH)
    _lib, LIB_PATH = None, BOUNDS_LIB_PATH
    try:
        yield load_library()
    finally:
        _lib, LIB_PATH = saved


def dvp_debug_bounds_status() -> int:
    """Waits for the current device and returns (and clears) the word into which the
    bounds-checking build ORs a code for every index it found out of range; raises
    ``DvpError(DVP_ERR_UNSUPPORTED)`` on the ordinary build, which has no checks."""
    out = ctypes.c_uint32(0)
    st = load_library().dvp_debug_bounds_status(ctypes.byref(out))
    if st != DVP_OK:
        raise DvpError(st, "dvp_debug_bounds_status")
    return int(out.value)


def status_string(status: int) -> str:
    return load_library().dvp_status_string(int(status)).decode()


def _ptr(t: torch.Tensor | None):
    return None if t is None else t.data_ptr()


def _address(t: torch.Tensor | None) -> int:
    return 0 if t is None else t.data_ptr()


def _stream(stream) -> int:
    if stream is None:
        return torch._C._cuda_getCurrentRawStream(torch.cuda.current_device())
    return stream.cuda_stream


def _check_matrix(name: str, x: torch.Tensor):
    if x.dim() != 2 or x.stride(1) != 1:
        raise ValueError(f"{name} must be 2-D with unit inner stride")
    if not x.is_cuda:
        raise ValueError(f"{name} must live on a CUDA device")


def _token_outputs(like: torch.Tensor, T: int, sides: int, floats: int):
    """``sides`` side namespaces with their addresses in the order of ``dvp_side_out``, ``floats`` further float32
    vectors of T tokens, and the flags.  All of them lie over one allocation."""
    v, base, step = _host.outputs(like, T, 7 * sides + floats, sides)
    out, n = [], 7 * sides + floats
    for i in range(sides):
        r, at = v[7 * i:7 * i + 7], base + 7 * i * step
        o = SimpleNamespace(max=r[0], lse=r[1], lse_safe=r[2], logp=r[3], logp_mp=r[4], comp_mp=r[5], log_cov=r[6],
                            count=v[n + i], mask=None)
        out.append((o, (at, at + step, at + 2 * step, at + 3 * step, at + 4 * step, at + 5 * step, base + (n + i) * step,
                        0, at + 6 * step)))
    return out, v[7 * sides:n], v[-1]


def _with_mask(side, like: torch.Tensor, T: int, V: int):
    o, addresses = side
    o.mask = like.new_empty((T, (V + 31) // 32), dtype=torch.int32)
    return o, addresses[:7] + (o.mask.data_ptr(), addresses[8])


def _addresses(side):
    """The addresses of a side's tensors, in the order of ``dvp_side_out``."""
    return tuple(_address(getattr(side, n)) for n in _SIDE_FIELDS)


_NO_SIDE = (0,) * 9


def _float32(x: float) -> float:
    """What a C float holds of x: struct refuses to pack a finite value beyond float32's range."""
    return ctypes.c_float(x).value


# What a uint32_t holds of a number, as ctypes takes it: struct refuses to pack what is out of range, where the library's
# own check is to answer.
_UINT32 = 0xffffffff


def _int32(x) -> int:
    """The same for an int32_t."""
    return (int(x) + 0x80000000 & 0xffffffff) - 0x80000000


def _id_dtype(ids: torch.Tensor) -> int:
    if ids.dtype == torch.int64:
        return DVP_ID_I64
    if ids.dtype == torch.int32:
        return DVP_ID_I32
    raise TypeError("ids must be int64 or int32")


def dvp_forward(train_logits: torch.Tensor, ids: torch.Tensor, rho: float, *,
                infer_logits: torch.Tensor | None = None, upstream: torch.Tensor | None = None,
                grad_train: torch.Tensor | None = None, grad_dtype: torch.dtype | None = None,
                want_mask: bool = False, stream=None, launch_hint: int = 0, out=None,
                mask_value: float | None = None, threshold_in_logits_dtype: bool = False,
                weight_kind: int = DVP_WEIGHT_NONE, weight_lo: float = 0.0, weight_hi: float = float("inf")):
    """Pruned log-probabilities of the sampled tokens for the training and the
    inference logits (Def. 5.1, Def. 5.2), their log-ratio, and, when
    ``upstream`` is given, dLoss/dlogits (Prop. 5.4) in the same call.

    ``mask_value`` (finite) switches to the App. A listing's semantics: pruned
    logits are replaced by it instead of by -inf; ``threshold_in_logits_dtype``
    rounds the threshold the way an eager tensor expression would.
    ``weight_kind`` (``DVP_WEIGHT_*``) multiplies each token's upstream gradient
    inside the kernel by the token's importance weight e^{log_ratio}, plain,
    truncated at ``weight_hi`` or masked outside [``weight_lo``, ``weight_hi``]
    (Thm. 5.3 per token); the weights used come back as ``weight``.

    Returns a namespace with ``train`` / ``infer`` (per-token tensors),
    ``log_ratio``, ``flags`` and ``grad_train``.  Pass the namespace of an
    earlier call as ``out`` to reuse its buffers.  The per-token tensors of a
    call lie over one storage (at most eighty bytes a token): keeping one keeps
    that storage, and ``torch.save`` of one writes all of it unless it is cloned.
    """
    lib = load_library()
    mode = (DVP_MODE_FINITE_MASK if mask_value is not None else 0) | \
        (DVP_MODE_THRESHOLD_IN_LOGITS_DTYPE if threshold_in_logits_dtype else 0)
    if out is None and not want_mask:   # all of it in one native call
        res = _host.forward(lib.forward_at, train_logits, ids, float(rho), infer_logits, upstream, grad_train, grad_dtype,
                            None if stream is None else stream.cuda_stream, launch_hint & _UINT32, mode,
                            0.0 if mask_value is None else mask_value, int(weight_kind) & _UINT32, weight_lo, weight_hi)
        if type(res) is int:
            raise DvpError(res, "dvp_forward")
        return res
    packed = lib.packed
    _check_matrix("train_logits", train_logits)
    T, V = train_logits.shape
    dtype = train_logits.dtype
    has_infer, weighted = infer_logits is not None, weight_kind != DVP_WEIGHT_NONE
    if has_infer:
        _check_matrix("infer_logits", infer_logits)
        if infer_logits.dtype != dtype or infer_logits.shape != train_logits.shape:
            raise ValueError("infer_logits must match train_logits in dtype and shape")
    if out is not None:
        res = out
        train_at, infer_at = _addresses(res.train), _addresses(res.infer) if has_infer else _NO_SIDE
    else:
        sides, rest, flags = _token_outputs(train_logits, T, 2 if has_infer else 1, has_infer + weighted)
        sides = [_with_mask(side, train_logits, T, V) for side in sides]   # without masks the call above was made
        res = SimpleNamespace(train=sides[0][0], infer=sides[1][0] if has_infer else None,
                              log_ratio=rest[0] if has_infer else None,
                              flags=flags, grad_train=None)
        train_at, infer_at = sides[0][1], sides[1][1] if has_infer else _NO_SIDE
        if weighted:
            res.weight = rest[-1]
    if weighted and getattr(res, "weight", None) is None:
        res.weight = train_logits.new_empty(T, dtype=torch.float32)
    grad_code = grad_ld = 0
    if upstream is not None:
        if upstream.dtype != torch.float32:
            raise TypeError("upstream must be float32")
        if grad_train is None:
            grad_train = res.grad_train
        if grad_train is None:
            grad_train = train_logits.new_empty((T, V), dtype=grad_dtype or dtype)
        _check_matrix("grad_train", grad_train)
        res.grad_train = grad_train
        grad_code, grad_ld = _DTYPES[grad_train.dtype], grad_train.stride(0)
    else:
        grad_train = None
    st = packed["dvp_forward"](_FORWARD_PACK.pack(
        _FORWARD_PACK.size, _DTYPES[dtype], grad_code, _id_dtype(ids), T, V, train_logits.stride(0),
        infer_logits.stride(0) if has_infer else 0, grad_ld, float(rho), train_logits.data_ptr(),
        _address(infer_logits), ids.data_ptr(), _address(upstream), _address(grad_train), *train_at, *infer_at,
        res.log_ratio.data_ptr() if has_infer else 0, res.flags.data_ptr(), _stream(stream), launch_hint & _UINT32, mode,
        _float32(mask_value) if mask_value is not None else 0.0, int(weight_kind) & _UINT32, _float32(weight_lo),
        _float32(weight_hi), res.weight.data_ptr() if weighted else 0))
    if st != DVP_OK:
        raise DvpError(st, "dvp_forward")
    return res


def dvp_backward(train_logits: torch.Tensor, ids: torch.Tensor, rho: float, upstream: torch.Tensor,
                 saved, *, grad_train: torch.Tensor | None = None,
                 grad_dtype: torch.dtype | None = None, use_comp: bool = True, stream=None,
                 launch_hint: int = 0, mask_value: float | None = None,
                 threshold_in_logits_dtype: bool = False) -> torch.Tensor:
    """dLoss/dlogits from the vectors an earlier ``dvp_forward`` saved
    (``saved`` = its result namespace) and a per-token upstream gradient."""
    packed = load_library().packed
    _check_matrix("train_logits", train_logits)
    T, V = train_logits.shape
    if grad_train is None:
        grad_train = train_logits.new_empty((T, V), dtype=grad_dtype or train_logits.dtype)
    _check_matrix("grad_train", grad_train)
    mode = (DVP_MODE_FINITE_MASK if mask_value is not None else 0) | \
        (DVP_MODE_THRESHOLD_IN_LOGITS_DTYPE if threshold_in_logits_dtype else 0)
    st = packed["dvp_backward"](_BACKWARD_PACK.pack(
        _BACKWARD_PACK.size, _DTYPES[train_logits.dtype], _DTYPES[grad_train.dtype], _id_dtype(ids), T, V,
        train_logits.stride(0), grad_train.stride(0), float(rho), train_logits.data_ptr(), ids.data_ptr(),
        upstream.data_ptr(), saved.train.max.data_ptr(), saved.train.lse_safe.data_ptr(),
        saved.train.comp_mp.data_ptr() if use_comp else 0, saved.flags.data_ptr(), grad_train.data_ptr(),
        _stream(stream), launch_hint & _UINT32, mode, _float32(mask_value) if mask_value is not None else 0.0, 0))
    if st != DVP_OK:
        raise DvpError(st, "dvp_backward")
    return grad_train


def dvp_row_wait_status() -> int:
    """Synchronises the current device and returns (and clears) the status word of
    the resident-row kernel: 0 unless one of its bounded waits ran out."""
    out = ctypes.c_uint32(0)
    st = load_library().dvp_row_wait_status(ctypes.byref(out))
    if st != 0:
        raise DvpError(st, "dvp_row_wait_status")
    return int(out.value)


def dvp_gemm_tn(a: torch.Tensor, b: torch.Tensor, *, alpha: float = 1.0, out: torch.Tensor | None = None,
                accumulate: bool = False, single_block_tiles: bool = False, stream=None,
                a_transposed: bool = False, split_k: bool = False, b_transposed: bool = False):
    """``out (+)= alpha * a @ b.T`` on the tensor cores; a [m, k] and b [n, k] are
    both bf16 or both f16 with k contiguous, out is float32.  With ``a_transposed``
    ``a`` is given as [k, m] with m contiguous (``out (+)= alpha * a.T @ b.T``),
    with ``b_transposed`` ``b`` as [k, n] with n contiguous.
    ``split_k`` computes every tile as two halves of the k range added into ``out``.
    Returns (out, status) where status is a device int32 that is non-zero if the
    kernel gave up waiting."""
    lib = load_library()
    _check_matrix("a", a)
    _check_matrix("b", b)
    if a.dtype != b.dtype or a.dtype not in (torch.bfloat16, torch.float16):
        raise TypeError("a and b must both be bfloat16 or both float16")
    m, k = (a.shape[1], a.shape[0]) if a_transposed else a.shape
    n = b.shape[1] if b_transposed else b.shape[0]
    if out is None:
        out = torch.empty(m, n, dtype=torch.float32, device=a.device)
    status = torch.zeros(1, dtype=torch.int32, device=a.device)
    mode = int(accumulate) | (2 if single_block_tiles else 0) | (4 if a_transposed else 0) | (8 if split_k else 0) | \
        (16 if b_transposed else 0)
    st = lib.dvp_gemm_tn(_ptr(a), a.stride(0), _ptr(b), b.stride(0), _ptr(out), out.stride(0), m, n, k,
                         _DTYPES[a.dtype], float(alpha), mode, _ptr(status), _stream(stream))
    if st != DVP_OK:
        raise DvpError(st, "dvp_gemm_tn")
    return out, status


def dvp_workspace_bytes(entry_point: int, args: ctypes.Structure) -> int:
    return int(load_library().dvp_workspace_bytes(int(entry_point), ctypes.byref(args)))


def _fused_args(hidden, w_vocab, ids, rho, upstream, infer_logits, d_w, accumulate_dw, panel_rows, stream,
                want_mask=False):
    """Marshals the arguments both fused entry points share; creates the output tensors."""
    _check_matrix("hidden", hidden)
    _check_matrix("w_vocab", w_vocab)
    T, H = hidden.shape
    V = w_vocab.shape[0]
    if hidden.dtype != torch.bfloat16 or w_vocab.dtype != torch.bfloat16:
        raise TypeError("hidden and w_vocab must be bfloat16")
    has_infer = infer_logits is not None
    if has_infer:
        _check_matrix("infer_logits", infer_logits)
        if infer_logits.dtype != torch.bfloat16:
            raise TypeError("infer_logits must be bfloat16")
    sides, rest, flags = _token_outputs(hidden, T, 2 if has_infer else 1, has_infer)
    if want_mask:
        sides[0] = _with_mask(sides[0], hidden, T, V)
    res = SimpleNamespace(train=sides[0][0], infer=sides[1][0] if has_infer else None,
                          log_ratio=rest[0] if has_infer else None,
                          flags=flags,
                          d_hidden=hidden.new_empty((T, H), dtype=torch.float32),
                          d_w=d_w if d_w is not None else hidden.new_empty((V, H), dtype=torch.float32))
    a = FusedArgs.from_buffer_copy(_FUSED_PACK.pack(
        _FUSED_PACK.size, _id_dtype(ids), T, H, V, hidden.stride(0), w_vocab.stride(0),
        infer_logits.stride(0) if has_infer else 0, res.d_hidden.stride(0), res.d_w.stride(0), float(rho),
        hidden.data_ptr(), w_vocab.data_ptr(), _address(infer_logits), ids.data_ptr(), _address(upstream),
        res.d_hidden.data_ptr(), res.d_w.data_ptr(), _int32(accumulate_dw), _int32(panel_rows), *sides[0][1],
        *(sides[1][1] if has_infer else _NO_SIDE), res.log_ratio.data_ptr() if has_infer else 0, res.flags.data_ptr(),
        0, 0, _stream(stream), 0, 0.0, 0.0, 0))
    return a, res


def dvp_fused_lmhead_forward_backward(hidden: torch.Tensor, w_vocab: torch.Tensor, ids: torch.Tensor,
                                      rho: float, upstream: torch.Tensor, *,
                                      infer_logits: torch.Tensor | None = None,
                                      d_w: torch.Tensor | None = None, accumulate_dw: bool = False,
                                      panel_rows: int = 0, workspace: torch.Tensor | None = None,
                                      stream=None, weight_kind: int = DVP_WEIGHT_NONE,
                                      weight_lo: float = 0.0, weight_hi: float = 1.0, want_mask: bool = False):
    """Pruned log-probabilities and gradients with respect to ``hidden`` and
    ``w_vocab`` with the training logits hidden x w_vocab^T produced panel by
    panel inside the library and never stored as a [T, V] matrix.  With
    ``weight_kind`` (truncate or mask, finite ``weight_hi``) each token's upstream
    gradient is multiplied by its importance weight; the weights come back as
    ``weight``.  ``want_mask`` asks for the packed training safe set."""
    lib = load_library()
    a, res = _fused_args(hidden, w_vocab, ids, rho, upstream, infer_logits, d_w, accumulate_dw, panel_rows,
                         stream, want_mask)
    need = dvp_workspace_bytes(DVP_ENTRY_FUSED_LMHEAD, a)
    if workspace is None:
        workspace = torch.empty(max(need, 256), dtype=torch.uint8, device=hidden.device)
    res.workspace = workspace
    a.workspace, a.workspace_bytes = _ptr(workspace), workspace.numel() * workspace.element_size()
    a.weight_kind = int(weight_kind)
    if weight_kind != DVP_WEIGHT_NONE:
        a.weight_lo, a.weight_hi = float(weight_lo), float(weight_hi)
        res.weight = torch.empty(hidden.shape[0], dtype=torch.float32, device=hidden.device)
        a.weight_out = _ptr(res.weight)
    st = lib.dvp_fused_lmhead_forward_backward(ctypes.byref(a))
    if st != DVP_OK:
        raise DvpError(st, "dvp_fused_lmhead_forward_backward")
    return res


def dvp_fused_lmhead_forward_backward_static(hidden: torch.Tensor, w_vocab: torch.Tensor,
                                             ids: torch.Tensor, rho: float, upstream: torch.Tensor, *,
                                             infer_logits: torch.Tensor | None = None,
                                             d_w: torch.Tensor | None = None,
                                             accumulate_dw: bool = False, panel_rows: int = 0,
                                             stream=None):
    """The fused LM-head computation for callers that have no device memory of
    their own to offer as a workspace: the library uses a fixed 32 MiB array that
    is part of its image instead, and the call allocates nothing (this wrapper
    only creates the output tensors a caller would normally already own).

    Problems whose workspace would not fit raise ``DvpError`` with
    ``DVP_ERR_WORKSPACE``.  All calls on a GPU share that one array, so calls
    that could overlap on the GPU (different streams) must be ordered by the
    caller.  Make the first call on each device outside any stream capture.
    ``dvp_static_workspace_status`` reads the status word of the last call."""
    lib = load_library()
    a, res = _fused_args(hidden, w_vocab, ids, rho, upstream, infer_logits, d_w, accumulate_dw, panel_rows,
                         stream)
    st = lib.dvp_fused_lmhead_forward_backward_static(ctypes.byref(a))
    if st != DVP_OK:
        raise DvpError(st, "dvp_fused_lmhead_forward_backward_static")
    return res


def dvp_static_workspace_status() -> int:
    """Waits for the current device and returns the status word that the tensor-core kernels of
    the last ``dvp_fused_lmhead_forward_backward_static`` call left in the built-in workspace:
    0 when every kernel finished, non-zero when one gave up waiting (results invalid)."""
    out = ctypes.c_uint32(0)
    st = load_library().dvp_static_workspace_status(ctypes.byref(out))
    if st != DVP_OK:
        raise DvpError(st, "dvp_static_workspace_status")
    return int(out.value)


def dvp_sequence_aggregate(log_ratio: torch.Tensor, seq_offsets: torch.Tensor,
                           veto_threshold: float = 1e-4, stream=None, log_cov: torch.Tensor | None = None):
    """Per-sequence sum and minimum of the token log-ratios, token counts and the
    veto flag (Sec. 4.4, Thm. 5.3, App. A protocol 5).  ``seq_offsets`` is an
    int64 device tensor of S + 1 non-decreasing token offsets.  With ``log_cov``
    (ln Z per token from ``dvp_forward``) also the minimum and the mean of the
    coverage Z over each sequence (Def. 5.2; the Z_min of Prop. 5.5)."""
    packed = load_library().packed
    if log_ratio.dtype != torch.float32 or seq_offsets.dtype != torch.int64:
        raise TypeError("log_ratio must be float32 and seq_offsets int64")
    has_cov = log_cov is not None
    if has_cov and (log_cov.dtype != torch.float32 or log_cov.numel() != log_ratio.numel()):
        raise TypeError("log_cov must be float32 with one entry per token")
    S = seq_offsets.numel() - 1
    v, _, _ = _host.outputs(log_ratio, S, 4 if has_cov else 2, 2)
    floats, counts = v[:-3], v[-3:-1]
    res = SimpleNamespace(seq_log_ratio=floats[0], min_log_ratio=floats[1], n_valid=counts[0], n_zero_weight=counts[1],
                          veto=v[-1])
    if has_cov:
        res.min_cov, res.mean_cov = floats[2], floats[3]
    st = packed["dvp_sequence_aggregate"](_SEQUENCE_PACK.pack(
        _SEQUENCE_PACK.size, 0, log_ratio.numel(), S, seq_offsets.data_ptr(), log_ratio.data_ptr(),
        float(veto_threshold), floats[0].data_ptr(), floats[1].data_ptr(), counts[0].data_ptr(), counts[1].data_ptr(),
        res.veto.data_ptr(), _stream(stream), _address(log_cov), floats[2].data_ptr() if has_cov else 0,
        floats[3].data_ptr() if has_cov else 0))
    if st != DVP_OK:
        raise DvpError(st, "dvp_sequence_aggregate")
    return res


def dvp_monitor(train_logits: torch.Tensor, infer_logits: torch.Tensor, stream=None):
    """Per-token KL(infer || train), KL(train || infer) and the two entropies over
    the full vocabulary (Sec. 6's stability metric), in nats."""
    packed = load_library().packed
    _check_matrix("train_logits", train_logits)
    _check_matrix("infer_logits", infer_logits)
    if infer_logits.dtype != train_logits.dtype or infer_logits.shape != train_logits.shape:
        raise ValueError("infer_logits must match train_logits in dtype and shape")
    T, V = train_logits.shape
    rows, at, step = _host.outputs(train_logits, T, 4, 0)
    st = packed["dvp_monitor"](_MONITOR_PACK.pack(
        _MONITOR_PACK.size, _DTYPES[train_logits.dtype], T, V, train_logits.stride(0), infer_logits.stride(0),
        train_logits.data_ptr(), infer_logits.data_ptr(), at, at + step, at + 2 * step, at + 3 * step,
        _stream(stream)))
    if st != DVP_OK:
        raise DvpError(st, "dvp_monitor")
    return SimpleNamespace(kl_infer_train=rows[0], kl_train_infer=rows[1], entropy_train=rows[2],
                           entropy_infer=rows[3])
