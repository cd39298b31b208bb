"""Python binding of liblopro.so: the same entry points as include/lopro.h, argument marshalling only.

What a program calls for every batch goes through the CPython extension built from csrc/binding.cpp (0.35 us of host
time per call besides the launches); sizes, checks and one-time steps go through ctypes.

Tensors are torch tensors (torch supplies device memory and streams); every computation runs in the
library's CUDA kernels.  The library must have been built (`python -m paper_2601_19675_b200.build`);
loading fails loudly otherwise -- there is no fallback path.
"""
from __future__ import annotations

import ctypes
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
# LOPRO_LIBRARY names another build of the library (A/B timing of kernel variants)
LIB_PATH = os.environ.get("LOPRO_LIBRARY") or os.path.join(_HERE, "liblopro.so")

OK, ERR_INVALID_ARG, ERR_UNSUPPORTED, ERR_BUFFER_TOO_SMALL, ERR_CUDA, ERR_TIMEOUT, ERR_INVALID_DATA = range(7)
OUT_BF16, OUT_F32 = 0, 1
LAYOUT_CANONICAL, LAYOUT_FRAGMENT, LAYOUT_ROWBLOCK = 0, 1, 2
SEC_HEADER, SEC_CODES, SEC_SCALEZERO, SEC_PERM, SEC_A, SEC_B, SEC_SIGMA, SEC_S = range(8)

# every symbol include/lopro.h declares
SYMBOLS = ["lopro_version", "lopro_status_str", "lopro_check_desc", "lopro_packed_bytes", "lopro_packed_section",
           "lopro_workspace_bytes", "lopro_pack", "lopro_unpack", "lopro_rotate", "lopro_linear_fwd",
           "lopro_linear_fwd_path", "lopro_host_staging_bytes", "lopro_linear_fwd_host", "lopro_linear_fwd_noalloc",
           "lopro_configure", "lopro_selftest_wait", "lopro_group_workspace_bytes", "lopro_linear_fwd_group_path",
           "lopro_linear_fwd_group", "lopro_pack_lr8", "lopro_unpack_lr8", "lopro_r1svd_workspace_bytes", "lopro_r1svd",
           "lopro_residual_rotate", "lopro_rtn_quantize", "lopro_quantize_workspace_bytes", "lopro_quantize_layer",
           "lopro_block_add_rmsnorm", "lopro_block_rope_append", "lopro_block_attention_workspace_bytes",
           "lopro_block_attention_decode", "lopro_block_silu_mul", "lopro_experts_workspace_bytes",
           "lopro_linear_fwd_experts_path", "lopro_linear_fwd_experts", "lopro_vq_packed_bytes", "lopro_vq_workspace_bytes",
           "lopro_vq_pack", "lopro_vq_linear_fwd", "lopro_product_kernel"]


class Desc(ctypes.Structure):
    _fields_ = [("d_in", ctypes.c_int32), ("d_out", ctypes.c_int32), ("bits", ctypes.c_int32),
                ("group_size", ctypes.c_int32), ("block_size", ctypes.c_int32), ("identity_cols", ctypes.c_int32),
                ("rank", ctypes.c_int32), ("layout", ctypes.c_int32), ("lowrank_format", ctypes.c_int32)]

    def __repr__(self):
        return "Desc(" + ", ".join(f"{n}={getattr(self, n)}" for n, _ in self._fields_) + ")"


class LoproError(RuntimeError):
    def __init__(self, status, where):
        self.status = int(status)
        super().__init__(f"{where}: {status_str(status)} (status {int(status)})")


_lib = None
_native = None      # the CPython extension, bound to the library by lib()
# the entry points it calls, by address
_NATIVE_SYMBOLS = ["lopro_linear_fwd", "lopro_linear_fwd_host", "lopro_linear_fwd_noalloc", "lopro_linear_fwd_group",
                   "lopro_linear_fwd_experts", "lopro_vq_linear_fwd", "lopro_rotate", "lopro_block_add_rmsnorm",
                   "lopro_block_rope_append", "lopro_block_attention_decode", "lopro_block_silu_mul"]


class VqDesc(ctypes.Structure):
    """lopro_vq_desc: the vector-quantized record (4-D centroids with 8-bit indices, or 2-D with 6-bit indices)."""
    _fields_ = [("d_in", ctypes.c_int32), ("d_out", ctypes.c_int32), ("cb_rows", ctypes.c_int32), ("cb_cols", ctypes.c_int32),
                ("block_size", ctypes.c_int32), ("identity_cols", ctypes.c_int32), ("rank", ctypes.c_int32),
                ("dim", ctypes.c_int32)]


def lib():
    """The loaded library (loads it, and binds the CPython extension to it, on first use)."""
    global _lib, _native
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(f"{LIB_PATH} is missing: build it with `python -m paper_2601_19675_b200.build`")
        L = ctypes.CDLL(LIB_PATH)
        vp, i32, i64, sz = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_size_t
        dp = ctypes.POINTER(Desc)
        L.lopro_version.restype = ctypes.c_int
        L.lopro_version.argtypes = []
        L.lopro_status_str.restype = ctypes.c_char_p
        L.lopro_status_str.argtypes = [ctypes.c_int]
        L.lopro_check_desc.restype = ctypes.c_int
        L.lopro_check_desc.argtypes = [dp]
        L.lopro_packed_bytes.restype = sz
        L.lopro_packed_bytes.argtypes = [dp]
        L.lopro_packed_section.restype = ctypes.c_int
        L.lopro_packed_section.argtypes = [dp, i32, ctypes.POINTER(sz), ctypes.POINTER(sz)]
        L.lopro_workspace_bytes.restype = sz
        L.lopro_workspace_bytes.argtypes = [dp, i32]
        L.lopro_pack.restype = ctypes.c_int
        L.lopro_pack.argtypes = [dp, vp, vp, vp, vp, vp, vp, vp, sz, vp]
        L.lopro_unpack.restype = ctypes.c_int
        L.lopro_unpack.argtypes = [dp, vp, vp, vp, vp, vp, vp, vp, vp, vp]
        L.lopro_rotate.restype = ctypes.c_int
        L.lopro_rotate.argtypes = [dp, vp, vp, i64, vp, i64, i32, vp]
        L.lopro_linear_fwd.restype = ctypes.c_int
        L.lopro_linear_fwd.argtypes = [dp, vp, vp, i64, vp, i64, i32, i32, vp, sz, vp]
        L.lopro_linear_fwd_path.restype = i32
        L.lopro_linear_fwd_path.argtypes = [dp, i32, ctypes.POINTER(i32)]
        L.lopro_host_staging_bytes.restype = sz
        L.lopro_host_staging_bytes.argtypes = [dp, i32, i32]
        L.lopro_linear_fwd_host.restype = ctypes.c_int
        L.lopro_linear_fwd_host.argtypes = [dp, vp, vp, vp, i32, i32, vp, sz, vp]
        L.lopro_linear_fwd_noalloc.restype = ctypes.c_int
        L.lopro_linear_fwd_noalloc.argtypes = [dp, vp, vp, i64, vp, i64, i32, i32, vp]
        dpp = ctypes.POINTER(ctypes.POINTER(Desc))
        L.lopro_group_workspace_bytes.restype = sz
        L.lopro_group_workspace_bytes.argtypes = [i32, dpp, i32]
        L.lopro_product_kernel.restype = i32
        L.lopro_product_kernel.argtypes = [i32, dpp, ctypes.POINTER(i32), i32, ctypes.POINTER(i32)]
        L.lopro_linear_fwd_group_path.restype = i32
        L.lopro_linear_fwd_group_path.argtypes = [i32, dpp, i32, ctypes.POINTER(i32)]
        L.lopro_linear_fwd_group.restype = ctypes.c_int
        L.lopro_linear_fwd_group.argtypes = [i32, dpp, ctypes.POINTER(vp), vp, i64, ctypes.POINTER(vp), ctypes.POINTER(i64), i32,
                                             i32, vp, sz, vp]
        L.lopro_pack_lr8.restype = ctypes.c_int
        L.lopro_pack_lr8.argtypes = [dp, vp, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp]
        L.lopro_unpack_lr8.restype = ctypes.c_int
        L.lopro_unpack_lr8.argtypes = [dp, vp, vp, vp, vp, vp, vp]
        L.lopro_configure.restype = ctypes.c_int
        L.lopro_configure.argtypes = [i32, i32]
        L.lopro_selftest_wait.restype = ctypes.c_int
        L.lopro_selftest_wait.argtypes = [vp, vp]
        L.lopro_r1svd_workspace_bytes.restype = sz
        L.lopro_r1svd_workspace_bytes.argtypes = [i32, i32]
        L.lopro_r1svd.restype = ctypes.c_int
        L.lopro_r1svd.argtypes = [vp, i32, i32, i32, i32, vp, i32, vp, vp, vp, vp, sz, vp]
        L.lopro_residual_rotate.restype = ctypes.c_int
        L.lopro_residual_rotate.argtypes = [dp, vp, vp, vp, vp, vp, vp, vp]
        L.lopro_rtn_quantize.restype = ctypes.c_int
        L.lopro_rtn_quantize.argtypes = [dp, vp, vp, vp, vp, vp, vp]
        L.lopro_quantize_workspace_bytes.restype = sz
        L.lopro_quantize_workspace_bytes.argtypes = [dp]
        L.lopro_quantize_layer.restype = ctypes.c_int
        L.lopro_quantize_layer.argtypes = [dp, vp, vp, vp, vp, i32, vp, vp, vp, vp, vp, vp, vp, vp, sz, vp]
        f32 = ctypes.c_float
        vdp = ctypes.POINTER(VqDesc)
        L.lopro_vq_packed_bytes.restype = sz
        L.lopro_vq_packed_bytes.argtypes = [vdp]
        L.lopro_vq_workspace_bytes.restype = sz
        L.lopro_vq_workspace_bytes.argtypes = [vdp, i32]
        L.lopro_vq_pack.restype = ctypes.c_int
        L.lopro_vq_pack.argtypes = [vdp, vp, vp, vp, vp, vp, vp, sz, vp]
        L.lopro_vq_linear_fwd.restype = ctypes.c_int
        L.lopro_vq_linear_fwd.argtypes = [vdp, vp, vp, i64, vp, i64, i32, i32, vp, sz, vp]
        L.lopro_experts_workspace_bytes.restype = sz
        L.lopro_experts_workspace_bytes.argtypes = [dp, i32, i32]
        L.lopro_linear_fwd_experts_path.restype = i32
        L.lopro_linear_fwd_experts_path.argtypes = [dp, i32, ctypes.POINTER(i32), ctypes.POINTER(i32)]
        L.lopro_linear_fwd_experts.restype = ctypes.c_int
        L.lopro_linear_fwd_experts.argtypes = [dp, i32, ctypes.POINTER(vp), ctypes.POINTER(i32), vp, i64, vp, i64, i32, vp, sz, vp]
        L.lopro_block_add_rmsnorm.restype = ctypes.c_int
        L.lopro_block_add_rmsnorm.argtypes = [vp, i64, vp, i64, vp, f32, vp, i64, i32, i32, vp]
        L.lopro_block_rope_append.restype = ctypes.c_int
        L.lopro_block_rope_append.argtypes = [vp, i64, vp, i64, vp, i64, vp, vp, vp, i32, i32, i32, i32, f32, vp, vp]
        L.lopro_block_attention_workspace_bytes.restype = sz
        L.lopro_block_attention_workspace_bytes.argtypes = [i32, i32, i32, i32]
        L.lopro_block_attention_decode.restype = ctypes.c_int
        L.lopro_block_attention_decode.argtypes = [vp, i64, vp, vp, vp, vp, i64, i32, i32, i32, i32, f32, vp, sz, vp, vp]
        L.lopro_block_silu_mul.restype = ctypes.c_int
        L.lopro_block_silu_mul.argtypes = [vp, i64, vp, i64, vp, i64, i32, i32, vp]
        try:
            from . import _binding
        except ImportError as e:
            path = os.path.join(os.path.dirname(LIB_PATH), "_binding.so")
            what = f"cannot be loaded here ({e})" if os.path.exists(path) else "is missing"
            raise RuntimeError(f"{path} {what}: build it with `python -m paper_2601_19675_b200.build`") from e
        _binding.bind({name: ctypes.cast(getattr(L, name), vp).value for name in _NATIVE_SYMBOLS})
        _native = _binding
        _lib = L
    return _lib


def _calls():
    """The extension's functions (loads the library on first use)."""
    if _native is None:
        lib()
    return _native


OPT_NO_WIDE, OPT_NO_TALL, OPT_NO_CHUNKS, OPT_NO_TCGEN05, OPT_PREFILL_PAIRS, OPT_ONE_KERNEL_SET, OPT_NO_CTA_PAIRS, \
    OPT_NO_STEP_RUNS = range(8)


def configure(option, value):
    """lopro_configure: set one tuning switch for the process (which kernels run, never what they compute)."""
    _check(lib().lopro_configure(int(option), int(value)), "lopro_configure")


class configured:
    """Context manager: a tuning switch set for the duration of a block, then back to its default (0; -1 for
    OPT_PREFILL_PAIRS)."""

    def __init__(self, option, value):
        self.option, self.value = option, value

    def __enter__(self):
        configure(self.option, self.value)

    def __exit__(self, *exc):
        configure(self.option, -1 if self.option == OPT_PREFILL_PAIRS else 0)


def selftest_wait(status_word):
    """lopro_selftest_wait: status_word is a device int32 tensor of one element; read it after synchronising."""
    _check(lib().lopro_selftest_wait(_ptr(status_word), _stream()), "lopro_selftest_wait")


def version():
    return lib().lopro_version()


def status_str(status):
    return lib().lopro_status_str(int(status)).decode()


LOWRANK_FOLDED_F16, LOWRANK_FP8 = 0, 1


def make_desc(d_in, d_out, bits, group_size, block_size, identity_cols=None, rank=0, layout=LAYOUT_FRAGMENT,
              lowrank_format=LOWRANK_FOLDED_F16):
    """Descriptor of one layer; identity_cols defaults to block_size (the paper's b_I = b_H)."""
    if identity_cols is None:
        identity_cols = block_size
    return Desc(d_in, d_out, bits, group_size, block_size, identity_cols, rank, layout, lowrank_format)


def check_desc(desc):
    return lib().lopro_check_desc(ctypes.byref(desc))


def packed_bytes(desc):
    return int(lib().lopro_packed_bytes(ctypes.byref(desc)))


def packed_section(desc, section):
    off, nbytes = ctypes.c_size_t(0), ctypes.c_size_t(0)
    st = lib().lopro_packed_section(ctypes.byref(desc), section, ctypes.byref(off), ctypes.byref(nbytes))
    if st != OK:
        raise LoproError(st, "lopro_packed_section")
    return int(off.value), int(nbytes.value)


def workspace_bytes(desc, T):
    return int(lib().lopro_workspace_bytes(ctypes.byref(desc), int(T)))


PATH_STREAM, PATH_GENERAL, PATH_PREFILL, PATH_TALL, PATH_WIDE, PATH_ROWBLOCK = 2, 3, 4, 5, 6, 7
PATH_NAMES = {PATH_TALL: "tall", PATH_WIDE: "wide", PATH_STREAM: "stream", PATH_GENERAL: "general", PATH_PREFILL: "prefill",
              PATH_ROWBLOCK: "rowblock"}


def linear_fwd_path(desc, T):
    """(path, launches) of lopro_linear_fwd for this layer and token count; path 0 = bad arguments."""
    n = ctypes.c_int32(0)
    path = int(lib().lopro_linear_fwd_path(ctypes.byref(desc), int(T), ctypes.byref(n)))
    return path, int(n.value)


def host_staging_bytes(desc, T, out_dtype=OUT_BF16):
    return int(lib().lopro_host_staging_bytes(ctypes.byref(desc), int(T), int(out_dtype)))


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def _check(st, where):
    if st != OK:
        raise LoproError(st, where)


def _dev(t, dtype_bytes):
    assert t.is_cuda and t.is_contiguous() and t.element_size() == dtype_bytes, "expects a contiguous device tensor"
    return t


def pack(desc, codes, scales_f16, zeros_f16, perm, A_f16=None, B_f16=None, out=None):
    """lopro_pack: device tensors in (uint8 codes [m][n]; 2-byte scales/zeros/A/B; int32 perm) -> uint8 blob."""
    nbytes = packed_bytes(desc)
    if nbytes == 0:
        raise LoproError(check_desc(desc) or ERR_INVALID_ARG, "lopro_packed_bytes")
    if out is None:
        out = torch.empty(nbytes, dtype=torch.uint8, device=codes.device)
    st = lib().lopro_pack(ctypes.byref(desc), _ptr(_dev(codes, 1)), _ptr(_dev(scales_f16, 2)), _ptr(_dev(zeros_f16, 2)),
                          _ptr(_dev(perm, 4)), _ptr(A_f16), _ptr(B_f16), _ptr(out), out.numel(), _stream())
    _check(st, "lopro_pack")
    return out


def pack_lr8(desc, codes, scales_f16, zeros_f16, perm, U_e4m3, V_e4m3, sigma_f16, s_f16, out=None):
    """lopro_pack_lr8: the record (W_q, U, V, Sigma, p, s) with U, V as fp8 e4m3 bytes, Sigma and s as fp16 bit patterns."""
    nbytes = packed_bytes(desc)
    if nbytes == 0:
        raise LoproError(check_desc(desc) or ERR_INVALID_ARG, "lopro_packed_bytes")
    if out is None:
        out = torch.empty(nbytes, dtype=torch.uint8, device=codes.device)
    st = lib().lopro_pack_lr8(ctypes.byref(desc), _ptr(_dev(codes, 1)), _ptr(_dev(scales_f16, 2)), _ptr(_dev(zeros_f16, 2)),
                              _ptr(_dev(perm, 4)), _ptr(_dev(U_e4m3, 1)), _ptr(_dev(V_e4m3, 1)), _ptr(_dev(sigma_f16, 2)),
                              _ptr(_dev(s_f16, 2)), _ptr(out), out.numel(), _stream())
    _check(st, "lopro_pack_lr8")
    return out


def r1svd_workspace_bytes(m, n):
    return int(lib().lopro_r1svd_workspace_bytes(m, n))


def r1svd(w, r, it, sketches, cast=False, workspace=None):
    """lopro_r1svd on a device fp32 matrix w [m][n] (deflated IN PLACE); returns (U [m][r], sigma [r], V [r][n]) fp32.
    The first word of the workspace (of r1svd_workspace_bytes) is the status word."""
    m, n = w.shape
    dev = w.device
    U = torch.empty((m, r), dtype=torch.float32, device=dev)
    sigma = torch.empty((r,), dtype=torch.float32, device=dev)
    V = torch.empty((r, n), dtype=torch.float32, device=dev)
    ws = workspace
    if ws is None:
        ws = torch.empty(max(r1svd_workspace_bytes(m, n), 256), dtype=torch.uint8, device=dev)
    st = lib().lopro_r1svd(_ptr(_dev(w, 4)), m, n, r, it, _ptr(_dev(sketches, 4)), 1 if cast else 0, _ptr(U), _ptr(sigma),
                           _ptr(V), _ptr(ws), ws.numel(), _stream())
    _check(st, "lopro_r1svd")
    return U, sigma, V


def residual_rotate(desc, W, Af, Bf, perm):
    """lopro_residual_rotate: R' = (W - Af Bf) P Q as fp32 [m][n], and the device status word (int32 tensor)."""
    out = torch.empty((desc.d_out, desc.d_in), dtype=torch.float32, device=W.device)
    status = torch.zeros(1, dtype=torch.int32, device=W.device)
    st = lib().lopro_residual_rotate(ctypes.byref(desc), _ptr(_dev(W, 4)), _ptr(None if Af is None else _dev(Af, 4)),
                                     _ptr(None if Bf is None else _dev(Bf, 4)), _ptr(_dev(perm, 4)), _ptr(out),
                                     _ptr(status), _stream())
    _check(st, "lopro_residual_rotate")
    return out, status


def rtn_quantize(desc, r_rot):
    """lopro_rtn_quantize: (codes uint8 [m][n], scales, zeros int16 fp16 bit patterns [m][n/g], status int32 tensor)."""
    m, n, g, dev = desc.d_out, desc.d_in, desc.group_size, r_rot.device
    codes = torch.empty((m, n), dtype=torch.uint8, device=dev)
    scales = torch.empty((m, n // g), dtype=torch.int16, device=dev)
    zeros = torch.empty((m, n // g), dtype=torch.int16, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    st = lib().lopro_rtn_quantize(ctypes.byref(desc), _ptr(_dev(r_rot, 4)), _ptr(codes), _ptr(scales), _ptr(zeros),
                                  _ptr(status), _stream())
    _check(st, "lopro_rtn_quantize")
    return codes, scales, zeros, status


def quantize_workspace_bytes(desc):
    return lib().lopro_quantize_workspace_bytes(ctypes.byref(desc))


def quantize_layer(desc, W, perm, sketches=None, it=8, s=None, workspace=None):
    """lopro_quantize_layer: a dict with codes, scales, zeros and the low-rank record in the input formats of
    pack / pack_lr8 (A, B int16 fp16 bits; or U, V uint8, sigma, s int16), plus the workspace (its first word is the
    status word)."""
    m, n, g, r, dev = desc.d_out, desc.d_in, desc.group_size, desc.rank, W.device
    nbytes = quantize_workspace_bytes(desc)
    if nbytes == 0:
        raise LoproError(check_desc(desc) or ERR_UNSUPPORTED, "lopro_quantize_workspace_bytes")
    if workspace is None:
        workspace = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    out = dict(codes=torch.empty((m, n), dtype=torch.uint8, device=dev),
               scales=torch.empty((m, n // g), dtype=torch.int16, device=dev),
               zeros=torch.empty((m, n // g), dtype=torch.int16, device=dev), workspace=workspace)
    lr = [None, None, None, None]
    if r > 0 and desc.lowrank_format == LOWRANK_FP8:
        out.update(U=torch.empty((m, r), dtype=torch.uint8, device=dev), V=torch.empty((r, n), dtype=torch.uint8, device=dev),
                   sigma=torch.empty((r,), dtype=torch.int16, device=dev), s=torch.empty((n,), dtype=torch.int16, device=dev))
        lr = [out["U"], out["V"], out["sigma"], out["s"]]
    elif r > 0:
        out.update(A=torch.empty((m, r), dtype=torch.int16, device=dev), B=torch.empty((r, n), dtype=torch.int16, device=dev))
        lr = [out["A"], out["B"], None, None]
    st = lib().lopro_quantize_layer(ctypes.byref(desc), _ptr(_dev(W, 4)), _ptr(None if s is None else _dev(s, 4)),
                                    _ptr(_dev(perm, 4)), _ptr(None if sketches is None else _dev(sketches, 4)), it,
                                    _ptr(out["codes"]), _ptr(out["scales"]), _ptr(out["zeros"]), _ptr(lr[0]), _ptr(lr[1]),
                                    _ptr(lr[2]), _ptr(lr[3]), _ptr(workspace), workspace.numel(), _stream())
    _check(st, "lopro_quantize_layer")
    return out


def block_add_rmsnorm(h, y, w, eps, out=None):
    """lopro_block_add_rmsnorm: h (bf16 [T][d], updated in place when y is given), y or None, w bf16 [d] -> out."""
    if out is None:
        out = torch.empty(tuple(h.shape), dtype=torch.bfloat16, device=h.device)
    _check(_calls().block_add_rmsnorm(h, y, w, eps, out), "lopro_block_add_rmsnorm")
    return out


def block_rope_append(q, k, v, pos, k_cache, v_cache, theta, status):
    """lopro_block_rope_append: q rotated in place; rotated k and v stored at entry pos[t] of the caches
    [T][heads][ctx_max][head_dim]."""
    _check(_calls().block_rope_append(q, k, v, pos, k_cache, v_cache, theta, status), "lopro_block_rope_append")


def block_attention_workspace_bytes(T, n_heads, head_dim, ctx_max):
    return lib().lopro_block_attention_workspace_bytes(T, n_heads, head_dim, ctx_max)


def block_attention_decode(q, k_cache, v_cache, ctx, scale, workspace, status, out=None):
    """lopro_block_attention_decode: q bf16 [T][heads * head_dim] against the caches; ctx int32 [T] valid entries."""
    if out is None:
        T, n_heads, _, head_dim = k_cache.shape
        out = torch.empty((T, n_heads * head_dim), dtype=torch.bfloat16, device=q.device)
    _check(_calls().block_attention_decode(q, k_cache, v_cache, ctx, scale, workspace, status, out), "lopro_block_attention_decode")
    return out


def block_silu_mul(gate, up, out=None):
    if out is None:
        out = torch.empty(tuple(gate.shape), dtype=torch.bfloat16, device=gate.device)
    _check(_calls().block_silu_mul(gate, up, out), "lopro_block_silu_mul")
    return out


def experts_workspace_bytes(desc, n_experts, max_rows):
    return lib().lopro_experts_workspace_bytes(ctypes.byref(desc), n_experts, max_rows)


def _offsets(row_offsets):
    return (ctypes.c_int32 * len(row_offsets))(*[int(v) for v in row_offsets])


def linear_fwd_experts_path(desc, row_offsets):
    """(path, launches) of lopro_linear_fwd_experts: 2 = shared launches, 1 = expert by expert."""
    launches = ctypes.c_int32(0)
    path = lib().lopro_linear_fwd_experts_path(ctypes.byref(desc), len(row_offsets) - 1, _offsets(row_offsets), ctypes.byref(launches))
    return path, launches.value


def linear_fwd_experts(desc, blobs, row_offsets, x, out_dtype=OUT_BF16, workspace=None, y=None):
    """lopro_linear_fwd_experts: x bf16 [rows][d_in] grouped by expert (host list row_offsets of len(blobs) + 1 entries)."""
    n = len(blobs)
    if workspace is None:
        max_rows = max([row_offsets[e + 1] - row_offsets[e] for e in range(n)] + [1])
        workspace = torch.zeros(max(experts_workspace_bytes(desc, n, max_rows), 256), dtype=torch.uint8, device=x.device)
    if y is None:
        y = torch.empty((x.shape[0], desc.d_out), dtype=torch.float32 if out_dtype == OUT_F32 else torch.bfloat16, device=x.device)
    _check(_calls().linear_fwd_experts(desc, blobs, row_offsets, x, out_dtype, workspace, y), "lopro_linear_fwd_experts")
    return y


def make_vq_desc(d_in, d_out, cb_rows, cb_cols, block_size, identity_cols=None, rank=0, dim=4):
    return VqDesc(d_in, d_out, cb_rows, cb_cols, block_size, block_size if identity_cols is None else identity_cols, rank, dim)


def vq_packed_bytes(desc):
    return lib().lopro_vq_packed_bytes(ctypes.byref(desc))


def vq_workspace_bytes(desc, T):
    return lib().lopro_vq_workspace_bytes(ctypes.byref(desc), T)


def vq_pack(desc, idx, codebooks_bf16, perm, A_f16=None, B_f16=None):
    """lopro_vq_pack: idx uint8 [m][n/dim], codebooks int16 bf16 bits [row groups][column groups][256 or 64][dim], perm int32 [n],
    A, B int16 fp16 bits (None with rank 0) -> packed device bytes."""
    nbytes = vq_packed_bytes(desc)
    if nbytes == 0:
        raise LoproError(ERR_UNSUPPORTED, "lopro_vq_packed_bytes")
    out = torch.empty(nbytes, dtype=torch.uint8, device=idx.device)
    st = lib().lopro_vq_pack(ctypes.byref(desc), _ptr(_dev(idx, 1)), _ptr(_dev(codebooks_bf16, 2)), _ptr(_dev(perm, 4)),
                             _ptr(None if A_f16 is None else _dev(A_f16, 2)), _ptr(None if B_f16 is None else _dev(B_f16, 2)),
                             _ptr(out), out.numel(), _stream())
    _check(st, "lopro_vq_pack")
    return out


def vq_linear_fwd(desc, packed, x, out_dtype=OUT_BF16, workspace=None, y=None):
    """lopro_vq_linear_fwd: x bf16 [T][n] device -> y [T][m]."""
    if workspace is None:
        workspace = torch.zeros(max(vq_workspace_bytes(desc, x.shape[0]), 256), dtype=torch.uint8, device=x.device)
    if y is None:
        y = torch.empty((x.shape[0], desc.d_out), dtype=torch.float32 if out_dtype == OUT_F32 else torch.bfloat16, device=x.device)
    _check(_calls().vq_linear_fwd(desc, packed, x, out_dtype, workspace, y), "lopro_vq_linear_fwd")
    return y


def unpack_lr8(desc, packed):
    """lopro_unpack_lr8: dict(U, V uint8; sigma, s int16 bit patterns) of freshly allocated device tensors."""
    m, n, r, dev = desc.d_out, desc.d_in, desc.rank, packed.device
    out = dict(U=torch.empty((m, r), dtype=torch.uint8, device=dev), V=torch.empty((r, n), dtype=torch.uint8, device=dev),
               sigma=torch.empty((r,), dtype=torch.int16, device=dev), s=torch.empty((n,), dtype=torch.int16, device=dev))
    st = lib().lopro_unpack_lr8(ctypes.byref(desc), _ptr(packed), _ptr(out["U"]), _ptr(out["V"]), _ptr(out["sigma"]),
                                _ptr(out["s"]), _stream())
    _check(st, "lopro_unpack_lr8")
    return out


def unpack(desc, packed, want=("codes", "words", "scales", "zeros", "perm", "A", "B")):
    """lopro_unpack: returns a dict of freshly allocated device tensors (16-bit floats as int16 bit patterns)."""
    m, n, g, r = desc.d_out, desc.d_in, desc.group_size, desc.rank
    dev = packed.device
    out = {}
    if "codes" in want:
        out["codes"] = torch.empty((m, n), dtype=torch.uint8, device=dev)
    if "words" in want:
        out["words"] = torch.empty((m, n * desc.bits // 32), dtype=torch.int32, device=dev)
    if "scales" in want:
        out["scales"] = torch.empty((m, n // g), dtype=torch.int16, device=dev)
    if "zeros" in want:
        out["zeros"] = torch.empty((m, n // g), dtype=torch.int16, device=dev)
    if "perm" in want:
        out["perm"] = torch.empty((n,), dtype=torch.int32, device=dev)
    if "A" in want and r > 0 and desc.lowrank_format == LOWRANK_FOLDED_F16:
        out["A"] = torch.empty((m, r), dtype=torch.int16, device=dev)
    if "B" in want and r > 0 and desc.lowrank_format == LOWRANK_FOLDED_F16:
        out["B"] = torch.empty((r, n), dtype=torch.int16, device=dev)
    st = lib().lopro_unpack(ctypes.byref(desc), _ptr(packed), _ptr(out.get("codes")), _ptr(out.get("words")),
                            _ptr(out.get("scales")), _ptr(out.get("zeros")), _ptr(out.get("perm")), _ptr(out.get("A")),
                            _ptr(out.get("B")), _stream())
    _check(st, "lopro_unpack")
    return out


def perm_of(desc, packed):
    """View of the permutation section of a blob (int32 [n], device)."""
    off, nbytes = packed_section(desc, SEC_PERM)
    return packed[off:off + nbytes].view(torch.int32)


def rotate(desc, perm, x, out=None):
    """lopro_rotate: x bf16 [T][n] (rows may be strided) -> rotated bf16 [T][n]."""
    if out is None:
        out = torch.empty((x.shape[0], desc.d_in), dtype=x.dtype, device=x.device)
    _check(_calls().rotate(desc, perm, x, out), "lopro_rotate")
    return out


def linear_fwd(desc, packed, x, out_dtype=OUT_BF16, workspace=None, y=None):
    """lopro_linear_fwd: x bf16 [T][n] device -> y [T][m] (bf16 or fp32)."""
    if workspace is None:
        workspace = torch.empty(max(workspace_bytes(desc, x.shape[0]), 256), dtype=torch.uint8, device=x.device)
    if y is None:
        y = torch.empty((x.shape[0], desc.d_out), dtype=torch.float32 if out_dtype == OUT_F32 else torch.bfloat16,
                        device=x.device)
    _check(_calls().linear_fwd(desc, packed, x, out_dtype, workspace, y), "lopro_linear_fwd")
    return y


def linear_fwd_host(desc, packed, x_host, y_host, workspace, out_dtype=OUT_BF16):
    """lopro_linear_fwd_host: x_host / y_host are HOST tensors (pinned for asynchronous copies); enqueues
    copy-in, forward and copy-out on the current stream and returns without synchronising."""
    _check(_calls().linear_fwd_host(desc, packed, x_host, out_dtype, workspace, y_host), "lopro_linear_fwd_host")
    return y_host


def _desc_array(descs):
    arr = (ctypes.POINTER(Desc) * len(descs))()
    for i, d in enumerate(descs):
        arr[i] = ctypes.pointer(d)
    return arr


def group_workspace_bytes(descs, T):
    return int(lib().lopro_group_workspace_bytes(len(descs), _desc_array(descs), int(T)))


PRODUCT_STREAM, PRODUCT_WIDE, PRODUCT_PERSISTENT, PRODUCT_ROW_RUNS, PRODUCT_STEP_RUNS = 1, 2, 3, 4, 5


def product_kernel(descs, T=0, rows=None):
    """(kernel, form) of the product launch that serves T <= 32 tokens of one layer, of siblings or, with rows, of experts of
    rows[i] rows each that share a launch; kernel 0 = no such launch.  form: (token tiles, tile steps of a batch, batches of a
    warp's ring, CTAs that share K, most row tiles of such CTAs) of PRODUCT_STEP_RUNS, zeros for the others."""
    form = (ctypes.c_int32 * 5)()
    n = None if rows is None else (ctypes.c_int32 * len(rows))(*[int(r) for r in rows])
    kernel = lib().lopro_product_kernel(len(descs), _desc_array(descs), n, int(T), form)
    return int(kernel), tuple(form)


def linear_fwd_group_path(descs, T):
    """(2, launches) when the sibling layers share their two launches, (1, launches) when they run one by one."""
    n = ctypes.c_int32(0)
    path = int(lib().lopro_linear_fwd_group_path(len(descs), _desc_array(descs), int(T), ctypes.byref(n)))
    return path, int(n.value)


def linear_fwd_group(descs, packed, x, out_dtype=OUT_BF16, workspace=None, ys=None):
    """lopro_linear_fwd_group: sibling layers on the same x bf16 [T][n] -> list of y_i [T][m_i]."""
    if workspace is None:
        workspace = torch.empty(max(group_workspace_bytes(descs, x.shape[0]), 256), dtype=torch.uint8, device=x.device)
    if ys is None:
        ys = [torch.empty((x.shape[0], d.d_out), dtype=torch.float32 if out_dtype == OUT_F32 else torch.bfloat16, device=x.device)
              for d in descs]
    _check(_calls().linear_fwd_group(descs, packed, x, out_dtype, workspace, ys), "lopro_linear_fwd_group")
    return ys


NOALLOC_SCRATCH_BYTES = 8 * 1024 * 1024


def linear_fwd_noalloc(desc, packed, x, y, out_dtype=OUT_BF16):
    """lopro_linear_fwd_noalloc: the forward without a workspace argument, for callers that may not allocate
    device memory (the scratch is a fixed array inside the library).  The binding allocates nothing either:
    the caller passes the output tensor y [T][m].  Raises LoproError(ERR_BUFFER_TOO_SMALL) when the layer and
    token count need more than NOALLOC_SCRATCH_BYTES of scratch."""
    _check(_calls().linear_fwd_noalloc(desc, packed, x, out_dtype, y), "lopro_linear_fwd_noalloc")
    return y


def workspace_status(workspace):
    """Status word a kernel leaves at the start of the workspace (synchronises)."""
    return int(workspace[:4].view(torch.int32).item())
