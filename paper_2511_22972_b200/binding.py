"""Binding of the C ABI in include/fly_verify.h: ctypes for what is called once, the native extension
(csrc/native_binding.cpp) for what is called every step.

Argument marshalling only: every step of the verification runs in the CUDA
kernels of libfly_verify.so.  There is no CPU fallback; a missing library that
cannot be built raises ImportError.
"""
from __future__ import annotations

import ctypes as C
import importlib.util
import os

from . import build as _build

FLY_OK, FLY_ERR_INVALID_ARG, FLY_ERR_UNSUPPORTED, FLY_ERR_CUDA, FLY_ERR_TIMEOUT, FLY_ERR_TOO_LARGE = range(6)
FLY_STATIC_MAX_BATCH, FLY_STATIC_MAX_PIECES = 1024, 16384
FLY_F32, FLY_BF16 = 0, 1
FLY_THETA_NATS, FLY_THETA_NORMALIZED = 0, 1
FLY_BOUNDARY_REJECT, FLY_BOUNDARY_CARRY = 0, 1
FLY_OPT_SPLITS, FLY_OPT_SCAN_MODE, FLY_OPT_WEIGHT_LAYOUT = 0, 1, 3

EXPORTS = (
    "fly_verify_create", "fly_verify_destroy", "fly_verify_run", "fly_verify_run_host", "fly_verify_run_static",
    "fly_verify_device_status", "fly_verify_selftest_wait", "fly_verify_reduce_shard", "fly_verify_run_partials",
    "fly_pld_draft", "fly_verify_plan",
    "fly_verify_set_option", "fly_verify_last_launch_count", "fly_verify_last_cuda_error",
    "fly_status_string",
)


class fly_verify_config_t(C.Structure):
    _fields_ = [("device", C.c_int32), ("max_batch", C.c_int32), ("max_k", C.c_int32),
                ("vocab", C.c_int32), ("logits_dtype", C.c_int), ("hidden", C.c_int32)]


class fly_verify_args_t(C.Structure):
    _fields_ = [
        ("B", C.c_int32), ("K", C.c_int32),
        ("logits", C.c_void_p), ("row_stride", C.c_int64),
        ("hidden", C.c_void_p), ("weight", C.c_void_p),
        ("draft", C.c_void_p),
        ("theta", C.c_double), ("theta_unit", C.c_int), ("W", C.c_int32), ("boundary", C.c_int),
        ("state_in", C.c_void_p), ("state_out", C.c_void_p),
        ("accept_len", C.c_void_p), ("rollback", C.c_void_p), ("out_tokens", C.c_void_p),
        ("target_argmax", C.c_void_p), ("entropy", C.c_void_p), ("row_flags", C.c_void_p),
        ("target_tokens", C.c_void_p),
        ("temperature", C.c_double), ("inputs_ready", C.c_int32),
    ]


class fly_plan_t(C.Structure):
    _fields_ = [("grid", C.c_int32), ("slots", C.c_int32), ("units_per_block", C.c_int64), ("units_per_row", C.c_int64),
                ("row_span", C.c_int64)]


class FlyError(RuntimeError):
    def __init__(self, status: int, what: str, cuda_error: int = 0):
        self.status = status
        self.cuda_error = cuda_error
        super().__init__(f"{what}: {status_string(status)} (status {status}, cuda error {cuda_error})")


_lib = None
_native = None


def lib() -> C.CDLL:
    """Loads (building first if a source is newer) libfly_verify.so."""
    global _lib, _native
    if _lib is not None:
        return _lib
    what = "libfly_verify.so is missing and could not be built"
    try:
        path = _build.ensure_built()
        what = "libfly_verify.so could not be loaded"
        L = C.CDLL(path)
        what = os.path.basename(_build.NATIVE_PATH) + " could not be loaded"
        import torch  # noqa: F401  (the extension resolves its symbols in torch's libraries)
        spec = importlib.util.spec_from_file_location(__package__ + "._native", _build.NATIVE_PATH)
        native = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(native)
        native.init(*[C.cast(getattr(L, f), C.c_void_p).value for f in (
            "fly_verify_run", "fly_verify_run_host", "fly_verify_reduce_shard", "fly_verify_run_partials",
            "fly_verify_run_static", "fly_pld_draft")])
    except Exception as e:  # no silent fallback: the CUDA library is the product
        raise ImportError(f"{what}: {e}") from e
    L.fly_verify_create.argtypes = [C.POINTER(fly_verify_config_t), C.POINTER(C.c_void_p)]
    L.fly_verify_create.restype = C.c_int
    L.fly_verify_destroy.argtypes = [C.c_void_p]
    L.fly_verify_destroy.restype = C.c_int
    L.fly_verify_run.argtypes = [C.c_void_p, C.POINTER(fly_verify_args_t), C.c_void_p]
    L.fly_verify_run.restype = C.c_int
    L.fly_verify_run_host.argtypes = [C.c_void_p, C.POINTER(fly_verify_args_t), C.c_void_p]
    L.fly_verify_run_host.restype = C.c_int
    L.fly_verify_run_static.argtypes = [C.c_int32, C.c_int32, C.c_int, C.POINTER(fly_verify_args_t), C.c_void_p]
    L.fly_verify_run_static.restype = C.c_int
    L.fly_verify_device_status.argtypes = [C.c_void_p, C.c_void_p]
    L.fly_verify_device_status.restype = C.c_int
    L.fly_verify_selftest_wait.argtypes = [C.c_void_p, C.c_void_p]
    L.fly_verify_selftest_wait.restype = C.c_int
    L.fly_verify_reduce_shard.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_int64, C.c_int32, C.c_double, C.c_void_p,
                                          C.c_void_p]
    L.fly_verify_reduce_shard.restype = C.c_int
    L.fly_verify_run_partials.argtypes = [C.c_void_p, C.POINTER(fly_verify_args_t), C.c_void_p, C.c_int32, C.c_int32,
                                          C.c_void_p]
    L.fly_verify_run_partials.restype = C.c_int
    L.fly_pld_draft.argtypes = [C.c_int32, C.c_int32, C.c_void_p, C.c_int64, C.c_void_p, C.c_int32, C.c_int32, C.c_int32,
                                C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    L.fly_pld_draft.restype = C.c_int
    L.fly_verify_plan.argtypes = [C.c_int32, C.c_int64, C.c_int32, C.c_int, C.c_int32, C.c_int32, C.c_int32,
                                  C.POINTER(fly_plan_t)]
    L.fly_verify_plan.restype = C.c_int
    L.fly_verify_set_option.argtypes = [C.c_void_p, C.c_int, C.c_int32]
    L.fly_verify_set_option.restype = C.c_int
    L.fly_verify_last_launch_count.argtypes = [C.c_void_p]
    L.fly_verify_last_launch_count.restype = C.c_int32
    L.fly_verify_last_cuda_error.argtypes = [C.c_void_p]
    L.fly_verify_last_cuda_error.restype = C.c_int32
    L.fly_status_string.argtypes = [C.c_int]
    L.fly_status_string.restype = C.c_char_p
    _native = native
    _lib = L
    return L


def status_string(status: int) -> str:
    return lib().fly_status_string(int(status)).decode()


class FlyVerify:
    """Handle of one verifier (fly_verify_create / fly_verify_destroy).

    Tensors are torch tensors used purely as typed device (or, for run_host,
    pinned host) buffers; the caller owns them.
    """

    def __init__(self, max_batch: int, max_k: int, vocab: int, dtype: str = "bf16", device: int = 0,
                 hidden: int = 0):
        self._h = C.c_void_p()
        self.weight_vd = False
        self.vocab = int(vocab)
        self.dtype = dtype
        cfg = fly_verify_config_t(int(device), int(max_batch), int(max_k), int(vocab),
                                  FLY_BF16 if dtype == "bf16" else FLY_F32, int(hidden))
        st = lib().fly_verify_create(C.byref(cfg), C.byref(self._h))
        if st != FLY_OK:
            self._h = C.c_void_p()
            raise FlyError(st, "fly_verify_create")

    def _raise(self, status: int, what: str):
        raise FlyError(status, what, lib().fly_verify_last_cuda_error(self._h))

    def close(self):
        if getattr(self, "_h", None) is not None and self._h.value:
            lib().fly_verify_destroy(self._h)
            self._h = C.c_void_p()

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass

    def set_option(self, option: int, value: int):
        st = lib().fly_verify_set_option(self._h, int(option), int(value))
        if st != FLY_OK:
            raise FlyError(st, "fly_verify_set_option")

    def set_splits(self, splits: int):
        self.set_option(FLY_OPT_SPLITS, splits)

    def set_scan_mode(self, separate_kernel: bool):
        self.set_option(FLY_OPT_SCAN_MODE, 1 if separate_kernel else 0)

    def set_weight_layout(self, vocab_major: bool):
        """Fused path: True if the weight is stored [V, hidden] (hidden contiguous), False for [hidden, V]."""
        self.set_option(FLY_OPT_WEIGHT_LAYOUT, 1 if vocab_major else 0)
        self.weight_vd = bool(vocab_major)

    def device_status(self, stream: int = 0) -> int:
        """fly_verify_device_status: synchronises the stream; FLY_OK or FLY_ERR_TIMEOUT."""
        return int(lib().fly_verify_device_status(self._h, C.c_void_p(stream)))

    def reduce_shard(self, logits, vocab_offset: int, partial_out, stream: int = 0, temperature: float = 0.0):
        """fly_verify_reduce_shard: logits [rows, vocab_slice] (a strided view is fine) -> partial_out
        [rows, 4] (any 16-byte element type, e.g. float32 x 4)."""
        st = _native.reduce_shard(self._h.value or 0, self.vocab, logits, vocab_offset, partial_out, stream or 0, temperature)
        if st:
            self._raise(st, "fly_verify_reduce_shard")

    def run_partials(self, args: fly_verify_args_t, partials, world: int, total_vocab: int, stream: int = 0):
        """fly_verify_run_partials: partials [world, rows, 4] gathered from the ranks."""
        st = _native.run_partials(self._h.value or 0, C.addressof(args), partials, world, total_vocab, stream or 0)
        if st:
            self._raise(st, "fly_verify_run_partials")

    def selftest_wait(self, stream: int = 0) -> int:
        """fly_verify_selftest_wait: makes one bounded device-side wait run out on purpose (no fault)."""
        return int(lib().fly_verify_selftest_wait(self._h, C.c_void_p(stream)))

    @property
    def last_launch_count(self) -> int:
        return int(lib().fly_verify_last_launch_count(self._h))

    def make_args(self, B, K, draft, accept_len, out_tokens, logits=None, row_stride=0, hidden=None,
                  weight=None, theta=1.0, theta_unit="nats", W=3, boundary="reject", state_in=None,
                  state_out=None, rollback=None, target_argmax=None, entropy=None, row_flags=None,
                  target_tokens=None, temperature=0.0, inputs_ready=False):
        if _native is None:
            lib()  # (called without a handle)
        a = fly_verify_args_t()
        _native.fill(C.addressof(a), B, K, draft, accept_len, out_tokens, logits, row_stride, hidden, weight, theta,
                     theta_unit, W, boundary, state_in, state_out, rollback, target_argmax, entropy, row_flags,
                     target_tokens, temperature, inputs_ready)
        return a

    def run(self, args: fly_verify_args_t, stream: int = 0):
        """fly_verify_run: device buffers, asynchronous on `stream` (a raw cudaStream_t value)."""
        st = _native.run(self._h.value or 0, C.addressof(args), stream or 0, False)
        if st:
            self._raise(st, "fly_verify_run")

    def run_host(self, args: fly_verify_args_t, stream: int = 0):
        """fly_verify_run_host: host buffers, copies in and out, synchronises."""
        st = _native.run(self._h.value or 0, C.addressof(args), stream or 0, True)
        if st:
            self._raise(st, "fly_verify_run_host")


def run_static(args: fly_verify_args_t, vocab: int, dtype: str = "bf16", device: int = 0, stream: int = 0):
    """fly_verify_run_static: the logits-path step without a handle, for callers that must not allocate
    device memory (its scratch is a fixed array inside the library).  `args` is the same struct that
    FlyVerify.run takes; `static_args` fills one without needing a handle.  Calls on one device must not
    overlap on the GPU."""
    lib()  # (no handle has loaded it for the caller)
    st = _native.run_static(C.addressof(args), vocab, FLY_BF16 if dtype == "bf16" else FLY_F32, device, stream or 0)
    if st:
        raise FlyError(st, "fly_verify_run_static")


def pld_draft(tokens, lengths, K: int, max_ngram: int = 3, min_ngram: int = 1, device: int = 0, stream: int = 0):
    """fly_pld_draft on tokens [B, Lmax] int32 and lengths [B] int32 (device tensors).  Returns
    (draft [B, K], count [B], match_pos [B], match_ngram [B]) as new device tensors."""
    lib()
    st, draft, count, pos, ng = _native.pld_draft(tokens, lengths, K, max_ngram, min_ngram, device, stream or 0)
    if st:
        raise FlyError(st, "fly_pld_draft")
    return draft, count, pos, ng


def static_args(*a, **kw) -> fly_verify_args_t:
    """Fills a fly_verify_args_t (same parameters as FlyVerify.make_args) without creating a handle."""
    return FlyVerify.make_args(None, *a, **kw)


class VerifyBuffers:
    """Output buffers of one step, allocated once with torch and reused."""

    def __init__(self, B: int, K: int, device, pinned: bool = False):
        import torch
        kw = dict(device=device)
        if pinned:
            kw = dict(device="cpu", pin_memory=True)
        self.accept_len = torch.empty(B, dtype=torch.int32, **kw)
        self.rollback = torch.empty(B, dtype=torch.int32, **kw)
        self.out_tokens = torch.empty(B, K + 1, dtype=torch.int32, **kw)
        self.target_argmax = torch.empty(B, K + 1, dtype=torch.int32, **kw)
        self.entropy = torch.empty(B, K + 1, dtype=torch.float32, **kw)
        self.row_flags = torch.empty(B, K + 1, dtype=torch.int32, **kw)
        zero = torch.tensor([[0, 0, -1]] * B, dtype=torch.int32)   # the zero state of every sequence
        self.state = zero.pin_memory() if pinned else zero.to(device)


def plan(sm_count: int, rows: int, vocab: int, dtype: str = "bf16", vector_path: bool = True, inputs_ready: bool = False,
         forced_pieces: int = 0) -> fly_plan_t:
    """fly_verify_plan: the launch geometry of the row reduction (host arithmetic only, no CUDA call)."""
    out = fly_plan_t()
    st = lib().fly_verify_plan(int(sm_count), int(rows), int(vocab), FLY_BF16 if dtype == "bf16" else FLY_F32,
                               1 if vector_path else 0, 1 if inputs_ready else 0, int(forced_pieces), C.byref(out))
    if st != FLY_OK:
        raise FlyError(st, "fly_verify_plan")
    return out


def verify(fv: FlyVerify, logits, draft, out: VerifyBuffers, theta=1.0, W=3, theta_unit="nats",
           boundary="reject", stream: int = 0, host: bool = False, temperature=0.0, inputs_ready=False):
    """One verification step on logits [B, K+1, V] and draft [B, K] (int32).
    In carry mode out.state is both the carried-in and the carried-out state."""
    st = _native.verify(fv._h.value or 0, fv.vocab, logits, draft, out, theta, W, theta_unit, boundary, stream or 0, host,
                        temperature, inputs_ready)
    if st:
        fv._raise(st, "fly_verify_run_host" if host else "fly_verify_run")
    return out


def verify_fused(fv: FlyVerify, hidden, weight, draft, out: VerifyBuffers, theta=1.0, W=3, theta_unit="nats",
                 boundary="reject", stream: int = 0, host: bool = False, temperature=0.0):
    """One verification step on the fused LM-head path: hidden [B*(K+1), D] bf16 and weight [D, V] bf16
    (device; with host=True hidden, draft and the outputs are host buffers, the weight stays on the device).
    The logits hidden @ weight are formed and reduced inside the kernel and never stored."""
    st = _native.verify_fused(fv._h.value or 0, fv.vocab, fv.weight_vd, hidden, weight, draft, out, theta, W, theta_unit,
                              boundary, stream or 0, host, temperature)
    if st:
        fv._raise(st, "fly_verify_run_host" if host else "fly_verify_run")
    return out
