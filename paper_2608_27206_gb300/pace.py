"""Thin ctypes binding of libpace (include/pace.h).

Every function here only marshals arguments: torch CUDA tensors become device
pointers, host index arrays become int32/int64 buffers, and the call goes to the
C ABI of the same name.  PyTorch supplies device memory and the current stream;
all arithmetic runs in the library's CUDA kernels.  If libpace.so has not been
built, the first call raises: there is no fallback path.
"""
from __future__ import annotations

import ctypes
import os
from array import array
from typing import Optional, Sequence

import numpy as np
import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libpace.so")

PACE_OK, PACE_ERR_INVALID_ARG, PACE_ERR_UNSUPPORTED_ARCH = 0, 1, 2
PACE_ERR_WORKSPACE, PACE_ERR_CUDA, PACE_ERR_TIMEOUT = 3, 4, 5
STATS_FIELDS = ("phi", "rho_g", "d_top", "rho_d", "rho", "r", "n_patches", "k_tail", "h_out", "w_out")


class PaceError(RuntimeError):
    def __init__(self, fn: str, status: int, detail: str = ""):
        self.status = status
        super().__init__(f"{fn} failed: {status_string(status)}{detail}")


class ApcParams(ctypes.Structure):
    _fields_ = [("alpha", ctypes.c_float), ("gamma", ctypes.c_float), ("tail_frac", ctypes.c_float),
                ("r_min", ctypes.c_float), ("r_max", ctypes.c_float), ("align", ctypes.c_int32)]


class DdaeParams(ctypes.Structure):
    _fields_ = [("tau", ctypes.c_float), ("fusion", ctypes.c_int32)]


# fusion modes of DdaeParams (pace_ddae_fusion)
DDAE_ADAPTIVE, DDAE_ONLY_LLM, DDAE_ONLY_VIT, DDAE_FIXED = 0, 1, 2, 3
FEATURE_RGB_STATS, FEATURE_COLOR_ENTROPY, FEATURE_EDGE_DENSITY, FEATURE_LAPLACIAN = 0, 1, 2, 3
PIXEL_FEATURES = {"rgb_stats": 0, "color_entropy": 1, "edge_density": 2, "laplacian": 3}
PIXEL_FEATURE_DIM = 8   # floats per feature token (zero-padded)
QUERY_VISION_TEXT, QUERY_TEXT, QUERY_LAST = 0, 1, 2
QUERY_SETS = {"vision_text": QUERY_VISION_TEXT, "text": QUERY_TEXT, "last": QUERY_LAST}


class GatherTensor(ctypes.Structure):
    _fields_ = [("src", ctypes.c_void_p), ("dst", ctypes.c_void_p), ("row_bytes", ctypes.c_int64),
                ("src_row_stride", ctypes.c_int64), ("dst_row_stride", ctypes.c_int64), ("n_slabs", ctypes.c_int64),
                ("src_slab_stride", ctypes.c_int64), ("dst_slab_stride", ctypes.c_int64),
                ("n_src_rows", ctypes.c_int64)]


GATHER_MAX_TENSORS = 16


_P = ctypes.c_void_p   # device addresses and host index arrays alike
_SIGS = {
    "pace_status_string": (ctypes.c_char_p, [ctypes.c_int]),
    "pace_last_cuda_error": (ctypes.c_int, []),
    "pace_kernel_launch_count": (ctypes.c_uint64, []),
    "pace_selftest_wait_timeout": (ctypes.c_int, [ctypes.c_uint32, _P]),
    "pace_init": (ctypes.c_int, [ctypes.c_int]),
    "pace_device_status": (ctypes.c_int, [_P, _P, ctypes.c_int]),
    "pace_apc_params_default": (None, [ctypes.POINTER(ApcParams)]),
    "pace_apc_density_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, _P]),
    "pace_budget_vanilla": (ctypes.c_int32, [ctypes.c_int32, ctypes.c_int32, ctypes.c_double]),
    "pace_prune_index": (ctypes.c_int, [ctypes.c_int, _P, _P, _P, _P, _P, _P, _P]),
    "pace_gather_multi": (ctypes.c_int, [ctypes.POINTER(GatherTensor), ctypes.c_int, _P, ctypes.c_int64, _P]),
    "pace_apc_density_tokens_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, ctypes.c_int]),
    "pace_apc_density_tokens": (ctypes.c_int, [_P, _P, ctypes.c_int, ctypes.c_int, _P, _P,
                                               ctypes.POINTER(ApcParams), _P, _P, _P, ctypes.c_size_t, _P]),
    "pace_apc_density": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.POINTER(ApcParams), _P, _P,
                                        _P, ctypes.c_size_t, _P]),
    "pace_apc_pixel_features": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.c_int, _P, _P]),
    "pace_apc_density_pixel_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, _P]),
    "pace_apc_density_pixel": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.c_int,
                                              ctypes.POINTER(ApcParams), _P, _P, _P, ctypes.c_size_t, _P]),
    "pace_apc_density_static": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.POINTER(ApcParams),
                                               _P, _P, _P]),
    "pace_apc_resample": (ctypes.c_int, [_P, _P, _P, _P, _P, _P, _P, ctypes.c_int, _P]),
    "pace_apc_resample_to": (ctypes.c_int, [_P, _P, _P, _P, _P, _P, _P, _P, ctypes.c_int, _P]),
    "pace_vit_attn_importance_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, ctypes.c_int]),
    "pace_vit_attn_importance": (ctypes.c_int, [_P, _P, _P, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                                                ctypes.c_float, ctypes.c_int, _P, _P, ctypes.c_size_t, _P]),
    "pace_vit_attn_importance_chunked": (ctypes.c_int, [_P, _P, _P, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                                                        ctypes.c_float, ctypes.c_int, _P, _P, ctypes.c_size_t,
                                                        ctypes.c_int, _P, ctypes.POINTER(ctypes.c_void_p), _P]),
    "pace_llm_text_visual_importance_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, _P, ctypes.c_int,
                                                                         ctypes.c_int]),
    "pace_llm_text_visual_importance": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.c_int,
                                                       ctypes.c_int, ctypes.c_int, ctypes.c_float, _P, _P,
                                                       ctypes.c_size_t, _P]),
    "pace_llm_sequence_importance_workspace_size": (ctypes.c_size_t, [ctypes.c_int, _P, _P, _P,
                                                                      ctypes.c_int, ctypes.c_int, ctypes.c_int]),
    "pace_llm_sequence_importance": (ctypes.c_int, [_P, _P, _P, _P, _P, ctypes.c_int, ctypes.c_int,
                                                    ctypes.c_int, ctypes.c_int, ctypes.c_float, ctypes.c_int, _P,
                                                    _P, ctypes.c_size_t, _P]),
    "pace_ddae_params_default": (None, [ctypes.POINTER(DdaeParams)]),
    "pace_budget": (ctypes.c_int32, [ctypes.c_int32, ctypes.c_double]),
    "pace_ddae_select": (ctypes.c_int, [_P, _P, _P, _P, ctypes.c_int, ctypes.POINTER(DdaeParams), _P, _P,
                                        _P, _P]),
    "pace_gather": (ctypes.c_int, [_P, ctypes.c_int64, ctypes.c_int64, _P, ctypes.c_int64, _P, _P]),
}

_lib = None


def lib() -> ctypes.CDLL:
    """Opens libpace.so (once).  Raises if it is missing."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(f"{LIB_PATH} is not built; run paper_2608_27206_gb300.build.build() "
                               "(needs nvcc with sm_103a support)")
        L = ctypes.CDLL(LIB_PATH)
        for name, (res, args) in _SIGS.items():
            f = getattr(L, name)
            f.restype = res
            f.argtypes = args
        _lib = L
    return _lib


def status_string(status: int) -> str:
    return lib().pace_status_string(int(status)).decode()


def _check(fn: str, status: int):
    if status != PACE_OK:
        detail = f" (cudaError {lib().pace_last_cuda_error()})" if status == PACE_ERR_CUDA else ""
        raise PaceError(fn, status, detail)


# Host index arrays.  A call costs the GPU as little as 15 us, so what happens per argument counts:
# a list becomes an array.array (0.3 us; a numpy conversion with its ctypes pointer 3 us), a numpy
# array of the right type is passed as it is.  Each helper returns (owner, address, length); the
# owner has to outlive the call.
def _ints(a, code: str, dtype):
    if type(a) is list or type(a) is tuple:
        try:
            x = array(code, a)
            return x, x.buffer_info()[0], len(x)
        except (TypeError, OverflowError):
            pass    # nested, or not whole numbers: numpy decides
    elif type(a) is np.ndarray and a.dtype == dtype and a.flags.c_contiguous:
        return a, a.__array_interface__["data"][0], len(a)
    x = np.ascontiguousarray(np.asarray(a, dtype=dtype))
    return x, x.__array_interface__["data"][0], len(x)


_I32, _I64 = np.dtype(np.int32), np.dtype(np.int64)


def _i32(a):
    return _ints(a, "i", _I32)


def _i64(a):
    return _ints(a, "q", _I64)


def _n_patches(h, w) -> int:
    """Patches of the images whose sides the owners h and w hold."""
    if len(h) != len(w):
        raise ValueError("H and W differ in length")
    if len(h) == 1:
        return int(h[0]) // 14 * (int(w[0]) // 14)
    return sum(x // 14 * (y // 14) for x, y in zip(h.tolist(), w.tolist()))


def _first(t: torch.Tensor, n: int) -> torch.Tensor:
    return t if t.shape[0] == n else t[:n]


def _dev(t: Optional[torch.Tensor]):
    if t is None:
        return None
    if not t.is_cuda:
        raise ValueError("expected a CUDA tensor")
    if not t.is_contiguous():
        raise ValueError("expected a contiguous tensor")
    return t.data_ptr()


# The current stream's handle without a Stream object around it (0.1 us against 2.9), where torch has it.
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)


def _stream(stream):
    if stream is not None:
        return stream.cuda_stream
    if _raw_stream is not None:
        return _raw_stream(torch.cuda.current_device())
    return torch.cuda.current_stream().cuda_stream


def _workspace(size, args, ws: Optional[torch.Tensor], device):
    """The workspace tensor and its bytes: the caller's, or a new one of size(*args) bytes."""
    if ws is None:
        ws = torch.empty(max(int(size(*args)), 16), dtype=torch.uint8, device=device)
    return ws, ws.numel() * ws.element_size()


def _check_ws(fn: str, status: int, given):
    """_check; a caller's workspace that is too small is named as such."""
    if status != PACE_OK:
        _check("workspace" if status == PACE_ERR_WORKSPACE and given is not None else fn, status)


# ----------------------------------------------------------------------------------------------
# library state
# ----------------------------------------------------------------------------------------------
def pace_init(device: int = 0) -> None:
    _check("pace_init", lib().pace_init(int(device)))


def pace_device_status(clear: bool = True):
    """(code, kernel id) of the device status word; synchronises the device."""
    code, where = ctypes.c_int32(0), ctypes.c_int32(0)
    _check("pace_device_status", lib().pace_device_status(ctypes.byref(code), ctypes.byref(where), int(clear)))
    return code.value, where.value


def pace_selftest_wait_timeout(limit_us: int, stream=None) -> None:
    """Launches a kernel whose bounded wait must run out and report PACE_ERR_TIMEOUT."""
    _check("pace_selftest_wait_timeout", lib().pace_selftest_wait_timeout(int(limit_us), _stream(stream)))


def pace_kernel_launch_count() -> int:
    """Kernels launched by libpace so far in this process."""
    return int(lib().pace_kernel_launch_count())


def pace_budget(n_vis: int, frac: float) -> int:
    return int(lib().pace_budget(int(n_vis), float(frac)))


def apc_params(**kw) -> ApcParams:
    p = ApcParams()
    lib().pace_apc_params_default(ctypes.byref(p))
    for k, v in kw.items():
        setattr(p, k, v)
    return p


def ddae_params(**kw) -> DdaeParams:
    p = DdaeParams()
    lib().pace_ddae_params_default(ctypes.byref(p))
    for k, v in kw.items():
        setattr(p, k, v)
    return p


# ----------------------------------------------------------------------------------------------
# Condense
# ----------------------------------------------------------------------------------------------
def pace_apc_density_workspace_size(H: Sequence[int], W: Sequence[int]) -> int:
    (_h, hp, B), (_w, wp, _) = _i32(H), _i32(W)
    return int(lib().pace_apc_density_workspace_size(B, hp, wp))


def _density_outputs(n: int, B: int, dev, d_out, stats):
    if d_out is None:
        d_out = torch.empty(max(n, 1), dtype=torch.float32, device=dev)
    if stats is None:
        stats = torch.zeros((max(B, 1), 10), dtype=torch.int32, device=dev)
    return d_out, stats


def _params(params):
    return ctypes.byref(params) if params is not None else None


def pace_apc_density(img: torch.Tensor, img_off, H, W, params: Optional[ApcParams] = None,
                     d_out: Optional[torch.Tensor] = None, stats: Optional[torch.Tensor] = None,
                     ws: Optional[torch.Tensor] = None, stream=None):
    """APC density of B packed uint8 images.  Returns (d [sum N] float32, stats [B, 10] int32 view)."""
    (_o, op, _), (h, hp, B), (w, wp, _) = _i64(img_off), _i32(H), _i32(W)
    n = _n_patches(h, w)
    d_out, stats = _density_outputs(n, B, img.device, d_out, stats)
    L = lib()
    buf, nbytes = _workspace(L.pace_apc_density_workspace_size, (B, hp, wp), ws, img.device)
    _check_ws("pace_apc_density", L.pace_apc_density(_dev(img), op, hp, wp, B, _params(params), _dev(d_out), _dev(stats),
                                                     _dev(buf), nbytes, _stream(stream)), ws)
    return _first(d_out, n), _first(stats, B)


def _feature(feature) -> int:
    return PIXEL_FEATURES[feature] if isinstance(feature, str) else int(feature)


def pace_apc_pixel_features(img: torch.Tensor, img_off, H, W, feature, out: Optional[torch.Tensor] = None,
                            stream=None) -> torch.Tensor:
    """Pixel-statistic feature tokens float32 [sum N, 8] of B packed uint8 images; feature is
    "rgb_stats", "color_entropy", "edge_density", "laplacian" or a FEATURE_* code."""
    (_o, op, _), (h, hp, B), (w, wp, _) = _i64(img_off), _i32(H), _i32(W)
    n = _n_patches(h, w)
    if out is None:
        out = torch.empty((max(n, 1), PIXEL_FEATURE_DIM), dtype=torch.float32, device=img.device)
    _check("pace_apc_pixel_features", lib().pace_apc_pixel_features(_dev(img), op, hp, wp, B, _feature(feature), _dev(out),
                                                                    _stream(stream)))
    return _first(out, n)


def pace_apc_density_pixel_workspace_size(H, W) -> int:
    (_h, hp, B), (_w, wp, _) = _i32(H), _i32(W)
    return int(lib().pace_apc_density_pixel_workspace_size(B, hp, wp))


def pace_apc_density_pixel(img: torch.Tensor, img_off, H, W, feature, params: Optional[ApcParams] = None,
                           d_out: Optional[torch.Tensor] = None, stats: Optional[torch.Tensor] = None,
                           ws: Optional[torch.Tensor] = None, stream=None):
    """APC density with a pixel-statistic preview.  Returns (d [sum N], stats [B, 10])."""
    (_o, op, _), (h, hp, B), (w, wp, _) = _i64(img_off), _i32(H), _i32(W)
    n = _n_patches(h, w)
    d_out, stats = _density_outputs(n, B, img.device, d_out, stats)
    L = lib()
    buf, nbytes = _workspace(L.pace_apc_density_pixel_workspace_size, (B, hp, wp), ws, img.device)
    _check_ws("pace_apc_density_pixel",
              L.pace_apc_density_pixel(_dev(img), op, hp, wp, B, _feature(feature), _params(params), _dev(d_out), _dev(stats),
                                       _dev(buf), nbytes, _stream(stream)), ws)
    return _first(d_out, n), _first(stats, B)


PACE_APC_STATIC_MAX_IMAGES = 16
PACE_APC_STATIC_MAX_PATCHES = 65536


def pace_apc_density_static(img: torch.Tensor, img_off, H, W, params: Optional[ApcParams] = None,
                            d_out: Optional[torch.Tensor] = None, stats: Optional[torch.Tensor] = None,
                            stream=None):
    """pace_apc_density with the library's own static scratch: no workspace argument.

    For callers that cannot allocate device scratch.  Limited to PACE_APC_STATIC_MAX_IMAGES
    images and PACE_APC_STATIC_MAX_PATCHES patches per call; calls that overlap on the GPU
    share one scratch array and must be serialised.  Returns (d, stats) like pace_apc_density.
    """
    (_o, op, _), (h, hp, B), (w, wp, _) = _i64(img_off), _i32(H), _i32(W)
    n = _n_patches(h, w)
    d_out, stats = _density_outputs(n, B, img.device, d_out, stats)
    _check("pace_apc_density_static", lib().pace_apc_density_static(_dev(img), op, hp, wp, B, _params(params), _dev(d_out),
                                                                    _dev(stats), _stream(stream)))
    return _first(d_out, n), _first(stats, B)


def pace_apc_density_tokens_workspace_size(cu_tokens, D: int) -> int:
    _c, cp, n = _i32(cu_tokens)
    return int(lib().pace_apc_density_tokens_workspace_size(n - 1, cp, D))


def pace_apc_density_tokens(T: torch.Tensor, cu_tokens, H, W, params: Optional[ApcParams] = None,
                            d_out: Optional[torch.Tensor] = None, stats: Optional[torch.Tensor] = None,
                            ws: Optional[torch.Tensor] = None, stream=None):
    """APC density of B images' preview tokens T (bf16 [sum N, D]).  Returns (d [sum N], stats)."""
    (cu, cp, B), (_h, hp, _), (_w, wp, _) = _i32(cu_tokens), _i32(H), _i32(W)
    B -= 1
    n, D = int(cu[-1]), int(T.shape[-1])
    d_out, stats = _density_outputs(n, B, T.device, d_out, stats)
    L = lib()
    if ws is None:
        ws = torch.empty(max(int(L.pace_apc_density_tokens_workspace_size(B, cp, D)), 16), dtype=torch.uint8, device=T.device)
    _check("pace_apc_density_tokens", L.pace_apc_density_tokens(_dev(T), cp, B, D, hp, wp, _params(params), _dev(d_out),
                                                                _dev(stats), _dev(ws), ws.numel(), _stream(stream)))
    return _first(d_out, n), _first(stats, B)


def pace_budget_vanilla(n_vis_vanilla: int, n_vis_condensed: int, frac: float) -> int:
    return int(lib().pace_budget_vanilla(int(n_vis_vanilla), int(n_vis_condensed), float(frac)))


def pace_prune_index(cu_seq, vis_start, cu_vis, cu_keep, kept: torch.Tensor, out: Optional[torch.Tensor] = None,
                     stream=None):
    """Row list of the pruned sequences (global pre-prune rows), int32 on kept's device."""
    (sq, sp, B), (_vs, vsp, _), (v, vp, _), (kp, kpp, _) = _i32(cu_seq), _i32(vis_start), _i32(cu_vis), _i32(cu_keep)
    B -= 1
    n_out = int(sq[-1]) - int(sq[0]) - int(v[-1]) + int(kp[-1]) if B > 0 else 0
    if out is None:
        out = torch.empty(max(n_out, 1), dtype=torch.int32, device=kept.device)
    _check("pace_prune_index", lib().pace_prune_index(B, sp, vsp, vp, kpp, _dev(kept), _dev(out), _stream(stream)))
    return _first(out, n_out)


def gather_spec(src: torch.Tensor, dst: torch.Tensor, dim: int) -> GatherTensor:
    """Descriptor for gathering contiguous src along `dim` into contiguous dst: the dimensions
    before `dim` are slabs, the ones after it form a row."""
    if not (src.is_contiguous() and dst.is_contiguous()) or src.dtype != dst.dtype:
        raise ValueError("gather_spec needs contiguous src and dst of one dtype")
    if src.shape[:dim] != dst.shape[:dim] or src.shape[dim + 1:] != dst.shape[dim + 1:]:
        raise ValueError("src and dst may differ only along the gathered dimension")
    es = src.element_size()
    row = es * int(np.prod(src.shape[dim + 1:], dtype=np.int64))
    slabs = int(np.prod(src.shape[:dim], dtype=np.int64))
    return GatherTensor(src.data_ptr(), dst.data_ptr(), row, row, row, slabs, row * src.shape[dim],
                        row * dst.shape[dim], src.shape[dim])


def pace_gather_multi(specs, idx: torch.Tensor, stream=None):
    """Gathers every GatherTensor in `specs` with the same row list idx (device int32)."""
    arr = (GatherTensor * max(len(specs), 1))(*specs)
    st = lib().pace_gather_multi(arr, len(specs), _dev(idx), idx.numel(), _stream(stream))
    _check("pace_gather_multi", st)


def stats_dict(stats: torch.Tensor):
    """Decodes pace_apc_stats rows ([B, 10] int32) into a list of dicts."""
    a = stats.detach().cpu().numpy().astype(np.int32)
    f = a.view(np.float32)
    out = []
    for i in range(a.shape[0]):
        d = {k: float(f[i, j]) for j, k in enumerate(STATS_FIELDS[:6])}
        d.update({k: int(a[i, 6 + j]) for j, k in enumerate(STATS_FIELDS[6:])})
        out.append(d)
    return out


def pace_apc_resample(src: torch.Tensor, src_off, H, W, stats: torch.Tensor, dst: torch.Tensor, dst_off,
                      stream=None) -> None:
    (_o, op, _), (_h, hp, B), (_w, wp, _), (_d, dp, _) = _i64(src_off), _i32(H), _i32(W), _i64(dst_off)
    _check("pace_apc_resample", lib().pace_apc_resample(_dev(src), op, hp, wp, _dev(stats), _dev(dst), dp, B,
                                                        _stream(stream)))


def pace_apc_resample_to(src: torch.Tensor, src_off, H, W, H_out, W_out, dst: torch.Tensor, dst_off,
                         stream=None) -> None:
    (_o, op, _), (_h, hp, B), (_w, wp, _), (_d, dp, _) = _i64(src_off), _i32(H), _i32(W), _i64(dst_off)
    (_ho, hop, _), (_wo, wop, _) = _i32(H_out), _i32(W_out)
    _check("pace_apc_resample_to", lib().pace_apc_resample_to(_dev(src), op, hp, wp, hop, wop, _dev(dst), dp, B,
                                                              _stream(stream)))


# ----------------------------------------------------------------------------------------------
# Extract
# ----------------------------------------------------------------------------------------------
def pace_vit_attn_importance_workspace_size(cu_seqlens, n_heads: int) -> int:
    _c, cp, n = _i32(cu_seqlens)
    return int(lib().pace_vit_attn_importance_workspace_size(n - 1, cp, int(n_heads)))


def pace_vit_attn_importance(Q: torch.Tensor, K: torch.Tensor, cu_seqlens, scale: Optional[float] = None,
                             merge: int = 4, out: Optional[torch.Tensor] = None,
                             ws: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """S_vis_raw [total / merge] from bf16 Q, K [total, heads, head_dim]."""
    cu, cp, B = _i32(cu_seqlens)
    B -= 1
    total, Hh, D = Q.shape
    n = int(cu[-1]) // merge if merge else 0   # (refused by the library)
    if scale is None:
        scale = float(D) ** -0.5
    if out is None:
        out = torch.empty(max(n, 1), dtype=torch.float32, device=Q.device)
    L = lib()
    buf, nbytes = _workspace(L.pace_vit_attn_importance_workspace_size, (B, cp, Hh), ws, Q.device)
    _check_ws("pace_vit_attn_importance",
              L.pace_vit_attn_importance(_dev(Q), _dev(K), cp, B, Hh, D, float(scale), int(merge), _dev(out), _dev(buf),
                                         nbytes, _stream(stream)), ws)
    return _first(out, n)


def vit_chunk_rows(cu_seqlens, n_chunks: int, pair: int = 256) -> np.ndarray:
    """End rows of `n_chunks` near-equal pieces of Q, each end moved down to the end of a
    `pair`-row block of its image (or the image's end), so no block waits for a later piece."""
    cu = np.asarray(cu_seqlens, dtype=np.int64)
    total = int(cu[-1])
    ends = []
    for c in range(1, n_chunks):
        r = total * c // n_chunks
        b = int(np.searchsorted(cu, r, side="right")) - 1
        b = min(max(b, 0), len(cu) - 2)
        e = int(cu[b]) + (r - int(cu[b])) // pair * pair
        ends.append(max(e, ends[-1] if ends else 0))
    ends.append(total)
    return np.asarray(ends, dtype=np.int64)


def pace_vit_attn_importance_chunked(Q: torch.Tensor, K: torch.Tensor, cu_seqlens, chunk_end_rows,
                                     chunk_ready: Sequence[torch.cuda.Event], scale: Optional[float] = None,
                                     merge: int = 4, out: Optional[torch.Tensor] = None,
                                     ws: Optional[torch.Tensor] = None, stream=None) -> torch.Tensor:
    """pace_vit_attn_importance whose row log-sum-exp pass runs in pieces of query rows, piece c
    after the (already recorded) event chunk_ready[c]; bit-identical results."""
    cu, cp, B = _i32(cu_seqlens)
    B -= 1
    total, Hh, D = Q.shape
    n = int(cu[-1]) // merge if merge else 0   # (refused by the library)
    if scale is None:
        scale = float(D) ** -0.5
    if out is None:
        out = torch.empty(max(n, 1), dtype=torch.float32, device=Q.device)
    _e, ep, n_ends = _i64(chunk_end_rows)
    if len(chunk_ready) != n_ends:
        raise ValueError("one event per chunk")
    evs = (ctypes.c_void_p * max(n_ends, 1))(*[int(e.cuda_event) for e in chunk_ready])
    L = lib()
    buf, nbytes = _workspace(L.pace_vit_attn_importance_workspace_size, (B, cp, Hh), ws, Q.device)
    _check_ws("pace_vit_attn_importance_chunked",
              L.pace_vit_attn_importance_chunked(_dev(Q), _dev(K), cp, B, Hh, D, float(scale), int(merge), _dev(out),
                                                 _dev(buf), nbytes, n_ends, ep, evs, _stream(stream)), ws)
    return _first(out, n)


def pace_llm_text_visual_importance_workspace_size(cu_q, cu_k, n_q_heads: int, n_kv_heads: int) -> int:
    (_q, qp, n), (_k, kp, _) = _i32(cu_q), _i32(cu_k)
    return int(lib().pace_llm_text_visual_importance_workspace_size(n - 1, qp, kp, int(n_q_heads), int(n_kv_heads)))


def pace_llm_text_visual_importance(Q: torch.Tensor, K: torch.Tensor, cu_q, cu_k, scale: Optional[float] = None,
                                    out: Optional[torch.Tensor] = None, ws: Optional[torch.Tensor] = None,
                                    stream=None) -> torch.Tensor:
    """S_llm_raw [sum Nv] from bf16 Q [sum Tq, Hq, D] and K [sum Nv, Hkv, D]."""
    (_q, qp, B), (k, kp, _) = _i32(cu_q), _i32(cu_k)
    B -= 1
    _, Hq, D = Q.shape
    Hkv = K.shape[1]
    n = int(k[-1])
    if scale is None:
        scale = float(D) ** -0.5
    if out is None:
        out = torch.empty(max(n, 1), dtype=torch.float32, device=Q.device)
    L = lib()
    buf, nbytes = _workspace(L.pace_llm_text_visual_importance_workspace_size, (B, qp, kp, Hq, Hkv), ws, Q.device)
    _check_ws("pace_llm_text_visual_importance",
              L.pace_llm_text_visual_importance(_dev(Q), _dev(K), qp, kp, B, Hq, Hkv, D, float(scale), _dev(out), _dev(buf),
                                                nbytes, _stream(stream)), ws)
    return _first(out, n)


def _query_set(query_set) -> int:
    return QUERY_SETS[query_set] if isinstance(query_set, str) else int(query_set)


def pace_llm_sequence_importance_workspace_size(cu_seq, vis_start, n_vis, n_q_heads: int, n_kv_heads: int,
                                                query_set="vision_text") -> int:
    (_c, cp, B), (_v, vp, _), (_n, np_, _) = _i32(cu_seq), _i32(vis_start), _i32(n_vis)
    return int(lib().pace_llm_sequence_importance_workspace_size(B - 1, cp, vp, np_, int(n_q_heads), int(n_kv_heads),
                                                                 _query_set(query_set)))


def pace_llm_sequence_importance(Q: torch.Tensor, K: torch.Tensor, cu_seq, vis_start, n_vis,
                                 query_set="vision_text", scale: Optional[float] = None,
                                 out: Optional[torch.Tensor] = None, ws: Optional[torch.Tensor] = None,
                                 stream=None) -> torch.Tensor:
    """Full-sequence S_llm_raw [sum n_vis] from bf16 Q [sum S, Hq, D] and K [sum S, Hkv, D] of causal
    sequences; query_set is "vision_text", "text" or "last" (or a QUERY_* code)."""
    (_c, cp, B), (_v, vp, _), (n, np_, _) = _i32(cu_seq), _i32(vis_start), _i32(n_vis)
    B -= 1
    _, Hq, D = Q.shape
    Hkv = K.shape[1]
    qs = _query_set(query_set)
    if scale is None:
        scale = float(D) ** -0.5
    total = sum(n.tolist()) if B > 0 else 0
    if out is None:
        out = torch.empty(max(total, 1), dtype=torch.float32, device=Q.device)
    L = lib()
    buf, nbytes = _workspace(L.pace_llm_sequence_importance_workspace_size, (B, cp, vp, np_, Hq, Hkv, qs), ws, Q.device)
    _check_ws("pace_llm_sequence_importance",
              L.pace_llm_sequence_importance(_dev(Q), _dev(K), cp, vp, np_, B, Hq, Hkv, D, float(scale), qs, _dev(out),
                                             _dev(buf), nbytes, _stream(stream)), ws)
    return _first(out, total)


def pace_ddae_select(s_llm_raw: torch.Tensor, s_vis_raw: torch.Tensor, cu_v, cu_keep,
                     params: Optional[DdaeParams] = None, s_final: Optional[torch.Tensor] = None,
                     weights: Optional[torch.Tensor] = None, kept: Optional[torch.Tensor] = None, stream=None):
    """Returns (s_final [sum Nv], weights [B, 2], kept int32 [sum K])."""
    (v, vp, B), (kp, kpp, _) = _i32(cu_v), _i32(cu_keep)
    B -= 1
    n, k = int(v[-1]), int(kp[-1])
    dev = s_llm_raw.device
    if s_final is None:
        s_final = torch.empty(max(n, 1), dtype=torch.float32, device=dev)
    if weights is None:
        weights = torch.empty((max(B, 1), 2), dtype=torch.float32, device=dev)
    if kept is None:
        kept = torch.empty(max(k, 1), dtype=torch.int32, device=dev)
    _check("pace_ddae_select", lib().pace_ddae_select(_dev(s_llm_raw), _dev(s_vis_raw), vp, kpp, B, _params(params),
                                                      _dev(s_final), _dev(weights), _dev(kept), _stream(stream)))
    return _first(s_final, n), _first(weights, B), _first(kept, k)


def pace_gather(src: torch.Tensor, idx: torch.Tensor, dst: Optional[torch.Tensor] = None, stream=None):
    """dst[r] = src[idx[r]] row by row (byte copy); src is [rows, ...] contiguous."""
    n_src = src.shape[0]
    row_bytes = src.numel() // n_src * src.element_size() if n_src else 0
    n = idx.numel()
    if dst is None:
        dst = torch.empty((max(n, 1),) + tuple(src.shape[1:]), dtype=src.dtype, device=src.device)
    st = lib().pace_gather(_dev(src), n_src, row_bytes, _dev(idx), n, _dev(dst), _stream(stream))
    _check("pace_gather", st)
    return _first(dst, n)
