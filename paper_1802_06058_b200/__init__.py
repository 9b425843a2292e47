"""Variance-based gradient compression hot path on NVIDIA B200 -- Python binding.

Thin marshalling over the C ABI declared in ``include/vgc.h`` (same entry-point names).
Every step of the path runs in the CUDA library ``libvgc.so`` built from ``csrc/``; the extension module
``_vgc_native`` checks tensors and passes pointers and sizes, this module raises on a non-zero status
(workspace sizes and other plain queries go through ctypes).  PyTorch is
used for device memory and streams.  There is no CPU fallback: if the library is missing or
was not built, every call raises.
"""
from __future__ import annotations

import ctypes
import importlib.util
import os
from typing import Optional, Sequence

import torch

from ._build import LIB_PATH, NATIVE_PATH, build  # noqa: F401  (build is re-exported)

VGC_OK = 0
VGC_DEV_CAPACITY = 1
VGC_DEV_TIMEOUT = 2
VGC_DEV_RANGE = 4
VGC_EXP_NONE = -(2 ** 31)
VGC_MAX_PARAMS = 1 << 28

EXPORTS = [
    "vgc_status_string", "vgc_version", "vgc_kernel_launch_count",
    "vgc_sqgrad_linear_workspace_bytes", "vgc_sqgrad_linear",
    "vgc_sqgrad_conv_workspace_bytes", "vgc_sqgrad_conv",
    "vgc_sqgrad_conv_batch_workspace_bytes", "vgc_sqgrad_conv_batch", "vgc_sqgrad_plan_hint",
    "vgc_sqgrad_conv_exact_workspace_bytes", "vgc_sqgrad_conv_exact",
    "vgc_sqgrad_conv_exact_batch_workspace_bytes", "vgc_sqgrad_conv_exact_batch",
    "vgc_compress_workspace_bytes", "vgc_compress", "vgc_compress_static",
    "vgc_decode_accumulate", "vgc_step_host",
    "vgc_compress_hybrid_workspace_bytes", "vgc_compress_hybrid", "vgc_decode_accumulate_hybrid",
    "vgc_decode_sum", "vgc_decode_sum_hybrid",
    "vgc_pack_bound_bytes", "vgc_pack_workspace_bytes", "vgc_pack_indices", "vgc_unpack_indices",
]


class VgcError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: status {status} ({_status_string(status)})")


class _MessageStruct(ctypes.Structure):      # mirrors vgc_message
    _fields_ = [("words", ctypes.c_void_p), ("capacity", ctypes.c_uint32), ("group_exp", ctypes.c_void_p),
                ("nnz", ctypes.c_void_p), ("n_criterion", ctypes.c_void_p), ("n_dropped", ctypes.c_void_p),
                ("mask", ctypes.c_void_p), ("dev_status", ctypes.c_void_p)]


class _LayerHostStruct(ctypes.Structure):    # mirrors vgc_layer_host
    _fields_ = [(name, ctypes.c_int) for name in ("is_conv", "B", "C", "H", "W", "Cout", "Kh", "Kw", "stride_h",
                                                  "stride_w", "pad_h", "pad_w")] + \
               [("x_host", ctypes.c_void_p), ("delta_host", ctypes.c_void_p), ("x_dev", ctypes.c_void_p),
                ("delta_dev", ctypes.c_void_p)]


class _HybridMessageStruct(ctypes.Structure):    # mirrors vgc_hybrid_message
    _fields_ = [("words", ctypes.c_void_p), ("capacity", ctypes.c_uint32), ("nnz", ctypes.c_void_p),
                ("mask", ctypes.c_void_p), ("dev_status", ctypes.c_void_p)]


class _ViewStruct(ctypes.Structure):         # mirrors vgc_message_view
    _fields_ = [("words", ctypes.c_void_p), ("nnz", ctypes.c_void_p), ("group_exp", ctypes.c_void_p),
                ("max_words", ctypes.c_uint32)]


_lib = None


def load_library():
    """Load libvgc.so (raises if it has not been built) and declare the entry points."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise RuntimeError(f"{LIB_PATH} is missing: run paper_1802_06058_b200.build() "
                           "(needs nvcc); there is no fallback path")
    lib = ctypes.CDLL(LIB_PATH)
    vp, i, f, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_float, ctypes.c_size_t
    lib.vgc_status_string.argtypes = [i]; lib.vgc_status_string.restype = ctypes.c_char_p
    lib.vgc_version.argtypes = []; lib.vgc_version.restype = i
    lib.vgc_kernel_launch_count.argtypes = []; lib.vgc_kernel_launch_count.restype = ctypes.c_uint64
    lib.vgc_sqgrad_linear_workspace_bytes.argtypes = [i, i, i]
    lib.vgc_sqgrad_linear_workspace_bytes.restype = sz
    lib.vgc_sqgrad_linear.argtypes = [vp, vp, i, i, i, f, i, vp, vp, sz, vp]
    lib.vgc_sqgrad_linear.restype = i
    lib.vgc_sqgrad_conv_workspace_bytes.argtypes = [i] * 11
    lib.vgc_sqgrad_conv_workspace_bytes.restype = sz
    lib.vgc_sqgrad_conv.argtypes = [vp, vp] + [i] * 11 + [f, i, vp, vp, sz, vp]
    lib.vgc_sqgrad_conv.restype = i
    lib.vgc_sqgrad_conv_batch_workspace_bytes.argtypes = [i] * 12
    lib.vgc_sqgrad_conv_batch_workspace_bytes.restype = sz
    lib.vgc_sqgrad_conv_batch.argtypes = [i, vp, vp, vp] + [i] * 11 + [f, i, vp, sz, vp]
    lib.vgc_sqgrad_conv_batch.restype = i
    lib.vgc_sqgrad_plan_hint.argtypes = [i]; lib.vgc_sqgrad_plan_hint.restype = None
    lib.vgc_sqgrad_conv_exact_workspace_bytes.argtypes = [i] * 11
    lib.vgc_sqgrad_conv_exact_workspace_bytes.restype = sz
    lib.vgc_sqgrad_conv_exact.argtypes = lib.vgc_sqgrad_conv.argtypes
    lib.vgc_sqgrad_conv_exact.restype = i
    lib.vgc_sqgrad_conv_exact_batch_workspace_bytes.argtypes = [i] * 12
    lib.vgc_sqgrad_conv_exact_batch_workspace_bytes.restype = sz
    lib.vgc_sqgrad_conv_exact_batch.argtypes = lib.vgc_sqgrad_conv_batch.argtypes
    lib.vgc_sqgrad_conv_exact_batch.restype = i
    lib.vgc_compress_workspace_bytes.argtypes = [sz, i]
    lib.vgc_compress_workspace_bytes.restype = sz
    lib.vgc_compress.argtypes = [vp, vp, vp, vp, sz, vp, i, f, f, ctypes.POINTER(_MessageStruct), vp, sz, vp]
    lib.vgc_compress.restype = i
    lib.vgc_compress_static.argtypes = [vp, vp, vp, vp, sz, vp, i, f, f, ctypes.POINTER(_MessageStruct), vp]
    lib.vgc_compress_static.restype = i
    lib.vgc_step_host.argtypes = [ctypes.POINTER(_LayerHostStruct), i, vp, vp, vp, vp, vp, sz, vp, i, f, f, f,
                                  ctypes.POINTER(_MessageStruct), vp, vp, vp, sz, vp, sz, vp]
    lib.vgc_step_host.restype = i
    lib.vgc_decode_accumulate.argtypes = [ctypes.POINTER(_ViewStruct), i, vp, i, f, vp, sz, vp, vp]
    lib.vgc_decode_accumulate.restype = i
    lib.vgc_decode_sum.argtypes = lib.vgc_decode_accumulate.argtypes
    lib.vgc_decode_sum.restype = i
    lib.vgc_compress_hybrid_workspace_bytes.argtypes = [sz]
    lib.vgc_compress_hybrid_workspace_bytes.restype = sz
    lib.vgc_compress_hybrid.argtypes = [vp, vp, vp, vp, sz, f, f, f, i, ctypes.POINTER(_HybridMessageStruct), vp, sz, vp]
    lib.vgc_compress_hybrid.restype = i
    lib.vgc_decode_accumulate_hybrid.argtypes = [ctypes.POINTER(_ViewStruct), i, f, f, vp, sz, vp, vp]
    lib.vgc_decode_accumulate_hybrid.restype = i
    lib.vgc_decode_sum_hybrid.argtypes = lib.vgc_decode_accumulate_hybrid.argtypes
    lib.vgc_decode_sum_hybrid.restype = i
    lib.vgc_pack_bound_bytes.argtypes = [ctypes.c_uint32]; lib.vgc_pack_bound_bytes.restype = sz
    lib.vgc_pack_workspace_bytes.argtypes = [ctypes.c_uint32]; lib.vgc_pack_workspace_bytes.restype = sz
    lib.vgc_pack_indices.argtypes = [vp, vp, ctypes.c_uint32, vp, sz, vp, vp, vp, sz, vp]
    lib.vgc_pack_indices.restype = i
    lib.vgc_unpack_indices.argtypes = [vp, vp, ctypes.c_uint32, vp, vp, vp]
    lib.vgc_unpack_indices.restype = i
    _lib = lib
    return lib


_native = None


def load_native():
    """Load the extension module that marshals the calls (raises if it has not been built)."""
    global _native
    if _native is None:
        load_library()
        if not os.path.exists(NATIVE_PATH):
            raise RuntimeError(f"{NATIVE_PATH} is missing: run paper_1802_06058_b200.build(); there is no fallback path")
        spec = importlib.util.spec_from_file_location("_vgc_native", NATIVE_PATH)
        mod = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(mod)
        mod.use_classes(MessageBuffers, HybridMessageBuffers)
        _native = mod
    return _native


def _status_string(status: int) -> str:
    try:
        return load_library().vgc_status_string(int(status)).decode()
    except Exception:  # pragma: no cover
        return "?"


def _check(status: int, where: str):
    if status != VGC_OK:
        raise VgcError(status, where)


def vgc_version() -> int:
    return load_library().vgc_version()


def vgc_kernel_launch_count() -> int:
    return load_library().vgc_kernel_launch_count()


# ------------------------------------------------------------------------------------------ (1)
def vgc_sqgrad_linear_workspace_bytes(B: int, n_in: int, n_out: int) -> int:
    return load_library().vgc_sqgrad_linear_workspace_bytes(B, n_in, n_out)


def vgc_sqgrad_linear(x, delta, scale: float, S, accumulate: bool = False, ws=None, stream=None):
    """S[out,in] (+)= scale * sum_z delta[z,:]^2 (outer) x[z,:]^2 ; x [B,in], delta [B,out]."""
    st = (_native or load_native()).sqgrad_linear(x, delta, scale, S, accumulate, ws, stream)
    if st:
        _check(st, "vgc_sqgrad_linear")
    return S


def vgc_sqgrad_conv_workspace_bytes(B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw) -> int:
    return load_library().vgc_sqgrad_conv_workspace_bytes(B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw)


def vgc_sqgrad_conv(x, delta, kernel, stride, padding, scale: float, S, accumulate: bool = False,
                    ws=None, stream=None):
    """S[Cout,C,Kh,Kw] (+)= scale * sum over (example, output position) of squared contributions."""
    st = (_native or load_native()).sqgrad_conv(x, delta, kernel, stride, padding, scale, S, accumulate, ws, stream, False)
    if st:
        _check(st, "vgc_sqgrad_conv")
    return S


def vgc_sqgrad_conv_exact_workspace_bytes(B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw) -> int:
    return load_library().vgc_sqgrad_conv_exact_workspace_bytes(B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw)


def vgc_sqgrad_conv_exact(x, delta, kernel, stride, padding, scale: float, S, accumulate: bool = False,
                          ws=None, stream=None):
    """S[Cout,C,Kh,Kw] (+)= scale * sum over examples of the squared per-example weight gradient."""
    st = (_native or load_native()).sqgrad_conv(x, delta, kernel, stride, padding, scale, S, accumulate, ws, stream, True)
    if st:
        _check(st, "vgc_sqgrad_conv_exact")
    return S


def vgc_sqgrad_plan_hint(concurrent_launches: int) -> None:
    """Tell the planner how many sqgrad calls run side by side (streams with separate workspaces): each then
    takes that share of the SMs.  Set it before asking for workspace sizes."""
    load_library().vgc_sqgrad_plan_hint(int(concurrent_launches))


def vgc_sqgrad_conv_batch_workspace_bytes(n_layers, B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw, exact: bool = False) -> int:
    lib = load_library()
    fn = lib.vgc_sqgrad_conv_exact_batch_workspace_bytes if exact else lib.vgc_sqgrad_conv_batch_workspace_bytes
    return fn(n_layers, B, C, H, W, Cout, Kh, Kw, sh, sw, ph, pw)


def vgc_sqgrad_conv_exact_batch(xs, deltas, kernel, stride, padding, scale: float, Ss, accumulate: bool = False,
                                ws=None, stream=None):
    """vgc_sqgrad_conv_exact for several layers of one geometry in one call."""
    return vgc_sqgrad_conv_batch(xs, deltas, kernel, stride, padding, scale, Ss, accumulate, ws, stream, exact=True)


def vgc_sqgrad_conv_batch(xs, deltas, kernel, stride, padding, scale: float, Ss, accumulate: bool = False,
                          ws=None, stream=None, exact: bool = False):
    """vgc_sqgrad_conv for several layers of one geometry (lists of tensors of equal shapes) in one call
    (``exact``: the per-example statistic, vgc_sqgrad_conv_exact_batch)."""
    if len(deltas) != len(xs) or len(Ss) != len(xs):
        raise ValueError("xs, deltas, Ss must have the same length")
    if not len(xs):
        return Ss
    st = (_native or load_native()).sqgrad_conv_batch(xs, deltas, kernel, stride, padding, scale, Ss, accumulate, ws, stream,
                                                      exact)
    if st:
        _check(st, "vgc_sqgrad_conv_exact_batch" if exact else "vgc_sqgrad_conv_batch")
    return Ss


# ------------------------------------------------------------------------------------------ (2)
class MessageBuffers:
    """Device buffers behind a vgc_message: words, per-group exponents, counters, optional mask.

    ``counters`` is int32[4] on the device: nnz, n_criterion, n_dropped, dev_status."""

    def __init__(self, capacity: int, K: int, n: int = 0, with_mask: bool = False, device="cuda"):
        self.capacity = int(capacity)
        self.K = int(K)
        self.words = torch.empty(max(self.capacity, 1), dtype=torch.int32, device=device)
        self.group_exp = torch.empty(max(self.K, 1), dtype=torch.int32, device=device)
        self.counters = torch.zeros(4, dtype=torch.int32, device=device)
        self.mask = torch.zeros(n, dtype=torch.uint8, device=device) if with_mask else None

    def struct(self) -> _MessageStruct:
        c = self.counters.data_ptr()
        return _MessageStruct(self.words.data_ptr(), self.capacity, self.group_exp.data_ptr(), c, c + 4, c + 8,
                              self.mask.data_ptr() if self.mask is not None else None, c + 12)

    def view(self) -> _ViewStruct:
        return _ViewStruct(self.words.data_ptr(), self.counters.data_ptr(), self.group_exp.data_ptr(),
                           min(self.capacity, self.words.numel()))

    def read(self):
        """Device -> host copy (synchronises): dict with words (numpy uint32), group_exp, counters."""
        nnz, n_criterion, n_dropped, dev_status = (int(c) & 0xFFFFFFFF for c in self.counters.tolist())
        kept = min(nnz, self.capacity)
        return {"words": self.words[:kept].cpu().numpy().view("uint32"),
                "group_exp": self.group_exp[:self.K].cpu().numpy(),
                "nnz": nnz, "n_criterion": n_criterion, "n_dropped": n_dropped, "dev_status": dev_status,
                "mask": None if self.mask is None else self.mask.cpu().numpy()}


def vgc_compress_workspace_bytes(n: int, K: int) -> int:
    return load_library().vgc_compress_workspace_bytes(n, K)


def vgc_compress(g, s, r, v, group_offsets, alpha: float, zeta: float, out: MessageBuffers, ws, stream=None):
    """One step of Algorithm 1 over the flat buffer + Encode(); r, v updated in place.
    ``s=None``: v already contains this step's squared-gradient sums (sqgrad with accumulate into v)."""
    st = (_native or load_native()).compress(g, s, r, v, group_offsets, alpha, zeta, out, ws, stream)
    if st:
        _check(st, "vgc_compress")
    return out


VGC_COMPRESS_STATIC_MAX_PARAMS = 1 << 21
VGC_COMPRESS_STATIC_MAX_GROUPS = 1024


def vgc_compress_static(g, s, r, v, group_offsets, alpha: float, zeta: float, out: MessageBuffers, stream=None):
    """vgc_compress for callers that cannot allocate a workspace (memory planned up front, plug-ins
    running inside someone else's step, hosts that lend only the call's tensors): the scratch is a fixed
    array inside the library, so n is limited to VGC_COMPRESS_STATIC_MAX_PARAMS.  Nothing is allocated by
    this call -- the binding passes pointers only.  Calls on one device share the scratch: do not let
    two of them overlap on the GPU.  Make the first call on a device outside any stream capture."""
    st = (_native or load_native()).compress_static(g, s, r, v, group_offsets, alpha, zeta, out, stream)
    if st:
        _check(st, "vgc_compress_static")
    return out


# ------------------------------------------------------------------------------------------ (3)
def vgc_decode_accumulate(messages: Sequence, group_offsets, scale: float, u, dev_status, stream=None,
                          overwrite: bool = False):
    """u[idx] += scale * decoded value over all words of all messages.

    ``messages``: MessageBuffers objects, or (words int32, nnz int32[1], group_exp int32) tensor triples; the
    decoder reads at most as many words as the words tensor holds.
    ``dev_status``: int32[1] device tensor (zeroed by the caller) receiving VGC_DEV_* bits.
    ``overwrite``: write u = scale * sum instead (vgc_decode_sum): u is neither read nor needs clearing."""
    st = (_native or load_native()).decode(messages, group_offsets, scale, u, dev_status, stream, overwrite)
    if st:
        _check(st, "vgc_decode_sum" if overwrite else "vgc_decode_accumulate")
    return u


def vgc_decode_sum(messages: Sequence, group_offsets, scale: float, u, dev_status, stream=None):
    """u = scale * (sum of all words of all messages); every element of u is written."""
    return vgc_decode_accumulate(messages, group_offsets, scale, u, dev_status, stream, overwrite=True)


# ------------------------------------------------------------------------------------------ (4)
class HybridMessageBuffers:
    """Device buffers behind a vgc_hybrid_message.  ``counters`` is int32[2]: nnz, dev_status."""

    def __init__(self, capacity: int, n: int = 0, with_mask: bool = False, device="cuda"):
        self.capacity = int(capacity)
        self.words = torch.empty(max(self.capacity, 1), dtype=torch.int32, device=device)
        self.counters = torch.zeros(2, dtype=torch.int32, device=device)
        self.mask = torch.zeros(n, dtype=torch.uint8, device=device) if with_mask else None

    def struct(self) -> _HybridMessageStruct:
        c = self.counters.data_ptr()
        return _HybridMessageStruct(self.words.data_ptr(), self.capacity, c,
                                    self.mask.data_ptr() if self.mask is not None else None, c + 4)

    def view(self) -> _ViewStruct:
        return _ViewStruct(self.words.data_ptr(), self.counters.data_ptr(), None, min(self.capacity, self.words.numel()))

    def read(self):
        nnz, dev_status = (int(c) & 0xFFFFFFFF for c in self.counters.tolist())
        return {"words": self.words[:min(nnz, self.capacity)].cpu().numpy().view("uint32"), "nnz": nnz,
                "dev_status": dev_status, "mask": None if self.mask is None else self.mask.cpu().numpy()}


def vgc_compress_hybrid_workspace_bytes(n: int) -> int:
    return load_library().vgc_compress_hybrid_workspace_bytes(n)


def vgc_compress_hybrid(g, s, r, v, alpha: float, zeta: float, tau: float, out: HybridMessageBuffers, ws,
                        correction_from_updated_r: bool = False, stream=None):
    """One step of Algorithm 2 over the flat buffer; r, v updated in place.  ``s=None`` as for vgc_compress."""
    st = (_native or load_native()).compress_hybrid(g, s, r, v, alpha, zeta, tau, correction_from_updated_r, out, ws, stream)
    if st:
        _check(st, "vgc_compress_hybrid")
    return out


def vgc_decode_sum_hybrid(messages: Sequence, tau: float, scale: float, u, dev_status, stream=None):
    """u = scale * (sum of +-tau over all words); every element of u is written."""
    return vgc_decode_accumulate_hybrid(messages, tau, scale, u, dev_status, stream, overwrite=True)


def vgc_decode_accumulate_hybrid(messages: Sequence, tau: float, scale: float, u, dev_status, stream=None,
                                 overwrite: bool = False):
    """u[idx] += scale * (+-tau) over all words of all messages (HybridMessageBuffers or (words, nnz) pairs)."""
    st = (_native or load_native()).decode_hybrid(messages, tau, scale, u, dev_status, stream, overwrite)
    if st:
        _check(st, "vgc_decode_accumulate_hybrid")
    return u


# ------------------------------------------------------------------------------------------ (5)
def vgc_pack_bound_bytes(max_words: int) -> int:
    return load_library().vgc_pack_bound_bytes(int(max_words))


def vgc_pack_workspace_bytes(max_words: int) -> int:
    return load_library().vgc_pack_workspace_bytes(int(max_words))


def vgc_pack_indices(words, nnz, packed, packed_bytes, dev_status, ws, stream=None):
    """words int32 [max_words] + nnz int32 [1] (device) -> packed uint8 (device): the index field as differences in
    the base-128 code; packed_bytes int32 [1] (device) receives the stream's length."""
    st = (_native or load_native()).pack_indices(words, nnz, packed, packed_bytes, dev_status, ws, stream)
    if st:
        _check(st, "vgc_pack_indices")
    return packed


def vgc_unpack_indices(packed, nnz, words, dev_status, stream=None):
    """The inverse of vgc_pack_indices: rebuilds min(nnz, words.numel()) words (device int32)."""
    st = (_native or load_native()).unpack_indices(packed, nnz, words, dev_status, stream)
    if st:
        _check(st, "vgc_unpack_indices")
    return words


def vgc_step_host(layers, g_host, g_dev, s_dev, r, v, group_offsets, alpha, zeta, scale, out: MessageBuffers,
                  words_host, counters_host, ws_sqgrad, ws_compress, stream=None):
    """One worker step from host buffers.  ``layers``: list of dicts with keys is_conv, B, C, H, W, Cout,
    Kh, Kw, stride, pad, x_host, delta_host (CPU, ideally pinned) and x_dev, delta_dev (CUDA staging).
    Returns (nnz, n_criterion, n_dropped, dev_status) as read back into ``counters_host``."""
    st = (_native or load_native()).step_host(layers, g_host, g_dev, s_dev, r, v, group_offsets, alpha, zeta, scale, out,
                                              words_host, counters_host, ws_sqgrad, ws_compress, stream)
    if st:
        _check(st, "vgc_step_host")
    return tuple(int(c) & 0xFFFFFFFF for c in counters_host.tolist())


def offsets_tensor(offsets, device="cuda") -> torch.Tensor:
    """Group offsets (uint32 values < 2^31) as the int32 device tensor the binding passes."""
    import numpy as np
    return torch.from_numpy(np.asarray(offsets, dtype=np.int64).astype(np.int32)).to(device)
