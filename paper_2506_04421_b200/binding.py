"""Binding of libhmar.so: argument marshalling only, for the hot calls in a compiled module, for the others by ctypes.

Every function here has the name and argument order of the C entry point it wraps (see
include/hmar.h). Tensors are torch CUDA tensors used purely as device buffers; all of the
arithmetic runs inside the library's kernels. There is no CPU fallback: the first call loads the
library, and the first hot call the compiled module, each compiled first where its file is missing
or older than its sources (nvcc, g++, and a package directory that can be written), and raises
where that fails. build.build() compiles both ahead of time.
"""
import ctypes
import functools
import importlib.machinery
import importlib.util
import os
import threading

import torch

from . import build as _build

_LIB = None
_HOST = None
_LOADING = threading.Lock()

HMAR_OK = 0
HMAR_ERR_BAD_ARG = -1
HMAR_ERR_UNSUPPORTED = -2
HMAR_ERR_CUDA = -3
HMAR_ERR_WORKSPACE = -4
HMAR_ERR_DEVICE_TIMEOUT = -5
HMAR_ERR_BOUNDS = -6

HMAR_WINDOW_MARKOV = 0      # scales k-1 and k (HMAR)
HMAR_WINDOW_CAUSAL = 1      # scales 1..k (VAR's block-causal mask)
HMAR_WINDOW_SELF = 2        # scale k only (block-diagonal)
HMAR_WINDOW_PREV = 3        # scale k-1 only; the first scale attends to itself

EXPORTED_SYMBOLS = (
    "hmar_attn_fwd", "hmar_attn_fwd_f32", "hmar_attn_fwd_window", "hmar_attn_fwd_window_f32", "hmar_attn_fwd_packed", "hmar_attn_bwd_packed",
    "hmar_attn_bwd_workspace_bytes", "hmar_attn_bwd", "hmar_attn_bwd_f32", "hmar_attn_bwd_window",
    "hmar_attn_bwd_window_f32", "hmar_schedule_tiles_window", "hmar_attn_bwd_noalloc", "hmar_attn_scale_step", "hmar_attn_scale_step_f32", "hmar_attn_scale_step_strided", "hmar_schedule_tiles", "hmar_schedule_bwd_full_tile_share", "hmar_schedule_bwd_items",
    "hmar_recon_accumulate", "hmar_recon_downsample", "hmar_device_status", "hmar_selftest_bounded_wait", "hmar_profile_begin", "hmar_profile_end", "hmar_debug_force_simt", "hmar_launch_count", "hmar_shutdown",
    "hmar_status_string",
)


class HmarError(RuntimeError):
    def __init__(self, status, where):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} ({status})")


def lib():
    """Load (building first if the sources are newer) the in-tree shared library."""
    global _LIB
    if _LIB is not None:
        return _LIB
    path = _build.LIB_PATH                 # libhmar.so, or the library named by the HMAR_LIBRARY environment variable
    if os.path.abspath(path) == os.path.abspath(_build.CHECKED_LIB_PATH):
        if _build.needs_build(path):
            path = _build.build(checked=True)
    elif "HMAR_LIBRARY" not in os.environ and _build.needs_build():
        path = _build.build()
    L = ctypes.CDLL(path)
    vp, ip, fp = ctypes.c_void_p, ctypes.POINTER(ctypes.c_int), ctypes.c_float
    i = ctypes.c_int
    L.hmar_attn_fwd.argtypes = [vp, vp, vp, vp, vp, i, i, i, i, ip, fp, vp]
    L.hmar_attn_fwd_f32.argtypes = L.hmar_attn_fwd.argtypes
    L.hmar_attn_fwd_window.argtypes = [vp, vp, vp, vp, vp, i, i, i, i, ip, i, fp, vp]
    L.hmar_attn_fwd_window_f32.argtypes = L.hmar_attn_fwd_window.argtypes
    L.hmar_attn_fwd_packed.argtypes = [vp, vp, vp, i, i, i, i, ip, fp, vp]
    L.hmar_attn_bwd_packed.argtypes = [vp] * 5 + [vp, ctypes.c_size_t, i, i, i, i, ip, fp, vp]
    L.hmar_attn_bwd_workspace_bytes.argtypes = [i, i, i, i, ip]
    L.hmar_attn_bwd_workspace_bytes.restype = ctypes.c_size_t
    L.hmar_attn_bwd.argtypes = [vp] * 9 + [vp, ctypes.c_size_t, i, i, i, i, ip, fp, vp]
    L.hmar_attn_bwd_f32.argtypes = L.hmar_attn_bwd.argtypes
    L.hmar_attn_bwd_window.argtypes = [vp] * 9 + [vp, ctypes.c_size_t, i, i, i, i, ip, i, fp, vp]
    L.hmar_attn_bwd_window_f32.argtypes = L.hmar_attn_bwd_window.argtypes
    L.hmar_schedule_tiles_window.argtypes = [i, ip, i, i, ctypes.POINTER(ctypes.c_int32), i]
    L.hmar_schedule_bwd_full_tile_share.argtypes = [i, ip, i]
    L.hmar_schedule_bwd_items.argtypes = [i, ip, i, i, i, ctypes.POINTER(ctypes.c_int32), i]
    L.hmar_attn_bwd_noalloc.argtypes = [vp] * 9 + [i, i, i, i, ip, fp, vp]
    L.hmar_attn_scale_step.argtypes = [vp] * 7 + [i, i, i, i, i, fp, vp]
    L.hmar_attn_scale_step_f32.argtypes = L.hmar_attn_scale_step.argtypes
    ll = ctypes.c_longlong
    L.hmar_attn_scale_step_strided.argtypes = [vp] * 7 + [i, i, i, i, i, ll, ll, ll, ll, fp, vp]
    L.hmar_schedule_tiles.argtypes = [i, ip, i, ctypes.POINTER(ctypes.c_int32), i]
    L.hmar_recon_accumulate.argtypes = [vp, vp, vp, vp, vp, vp, i, i, i, i, i, vp]
    L.hmar_recon_downsample.argtypes = [vp, vp, i, i, i, i, vp]
    L.hmar_device_status.argtypes = [ip]
    L.hmar_selftest_bounded_wait.argtypes = [vp]
    L.hmar_profile_begin.restype = None
    L.hmar_profile_end.argtypes = [ctypes.c_char_p, ctypes.c_size_t]
    L.hmar_debug_force_simt.argtypes = [i]
    L.hmar_launch_count.restype = ctypes.c_longlong
    L.hmar_shutdown.restype = None
    L.hmar_status_string.argtypes = [i]
    L.hmar_status_string.restype = ctypes.c_char_p
    for name in EXPORTED_SYMBOLS:
        getattr(L, name)                     # a missing symbol fails here, at load time
    _LIB = L
    return L


def status_string(status):
    return lib().hmar_status_string(int(status)).decode()


@functools.lru_cache(maxsize=256)
def _sides_array(sides):
    return (ctypes.c_int * len(sides))(*sides), len(sides)


def _sides(side_lens):
    """(C array, length) of a side list; the arrays are read-only and shared by all calls with equal lists."""
    len(side_lens)                         # a generator has none, and is refused: a second call would find it used up
    return _sides_array(tuple(map(int, side_lens)))


def _ptr(t):
    return None if t is None else t.data_ptr()


_current_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)


def _stream(stream):
    if stream is not None:
        return stream.cuda_stream
    if _current_raw_stream is not None:
        return _current_raw_stream(torch.cuda.current_device())
    return torch.cuda.current_stream().cuda_stream


def _host():
    """The compiled module that checks the tensors, allocates the results and makes the call (csrc/host_binding.cpp)."""
    return _HOST if _HOST is not None else _load_host()


def _load_host():
    with _LOADING:                         # threads whose first calls meet compile and load the module once
        return _HOST if _HOST is not None else _load_host_locked()


def _load_host_locked():
    global _HOST
    library = lib()
    loader = importlib.machinery.ExtensionFileLoader("_hmar_host", _build.build_host())
    module = importlib.util.module_from_spec(importlib.util.spec_from_loader("_hmar_host", loader))
    loader.exec_module(module)
    module.bind(library._handle)
    _HOST = module
    return module


def _handle(stream):
    return None if stream is None else stream.cuda_stream


def _done(result, where, window=HMAR_WINDOW_MARKOV):
    """What a function of the compiled module returned: its results, or the library's status."""
    if result.__class__ is int:
        raise HmarError(result, where if window == HMAR_WINDOW_MARKOV else where + "_window")
    return result


def _check(status, where):
    if status != HMAR_OK:
        raise HmarError(status, where)


def _is_f32(t):
    if t.dtype == torch.float32:
        return True
    if t.dtype == torch.bfloat16:
        return False
    raise TypeError("tensors must be bfloat16 or float32")


def _need(*tensors):
    for t in tensors:
        if t is not None and not (t.is_cuda and t.is_contiguous()):
            raise ValueError("tensors must be contiguous CUDA tensors")


def hmar_attn_fwd(q, k, v, side_lens, softmax_scale, out=None, lse=None, stream=None, window=HMAR_WINDOW_MARKOV):
    """Training forward. q, k, v: [B,H,L,D]. Returns (out [B,H,L,D], lse [B,H,L] fp32).
    `window` other than HMAR_WINDOW_MARKOV goes through hmar_attn_fwd_window."""
    return _done(_host().fwd(q, k, v, out, lse, side_lens, softmax_scale, _handle(stream), window), "hmar_attn_fwd", window)


def hmar_attn_fwd_packed(qkv, side_lens, softmax_scale, out=None, lse=None, stream=None):
    """Training forward on the packed projection output. qkv: [B,L,3,H,D] bf16.
    Returns (out [B,L,H,D], lse [B,H,L] fp32)."""
    return _done(_host().fwd_packed(qkv, out, lse, side_lens, softmax_scale, _handle(stream)), "hmar_attn_fwd_packed")


def hmar_attn_bwd_packed(qkv, out, lse, dout, side_lens, softmax_scale, dqkv=None, workspace=None, stream=None):
    """Training backward on the packed layouts. qkv [B,L,3,H,D], out and dout [B,L,H,D], lse [B,H,L].
    Returns dqkv [B,L,3,H,D]."""
    return _done(_host().bwd_packed(qkv, out, lse, dout, side_lens, softmax_scale, dqkv, workspace, _handle(stream)), "hmar_attn_bwd_packed")


def hmar_attn_bwd_workspace_bytes(B, H, D, side_lens):
    sides, n = _sides(side_lens)
    return int(lib().hmar_attn_bwd_workspace_bytes(B, H, D, n, sides))


def hmar_attn_bwd(q, k, v, out, lse, dout, side_lens, softmax_scale, dq=None, dk=None, dv=None,
                  workspace=None, stream=None, window=HMAR_WINDOW_MARKOV):
    """Training backward. Returns (dq, dk, dv), each [B,H,L,D].
    `window` other than HMAR_WINDOW_MARKOV goes through hmar_attn_bwd_window."""
    return _done(_host().bwd(q, k, v, out, lse, dout, side_lens, softmax_scale, dq, dk, dv, workspace, _handle(stream), window), "hmar_attn_bwd", window)


HMAR_NOALLOC_MAX_ROWS = 32768


def hmar_attn_bwd_noalloc(q, k, v, out, lse, dout, side_lens, softmax_scale, dq, dk, dv, stream=None):
    """Backward through the entry point that allocates nothing: for callers that may not touch the
    device allocator (memory owned by someone else's pool, no growth after start-up, no call that may
    synchronise). The caller passes every output tensor; neither this wrapper nor the library
    allocates. B*H*L must not exceed HMAR_NOALLOC_MAX_ROWS, and calls must not overlap on the GPU."""
    _need(q, k, v, out, lse, dout, dq, dk, dv)
    if _is_f32(q):
        raise TypeError("hmar_attn_bwd_noalloc takes bfloat16 tensors")
    B, H, L, D = q.shape
    sides, n = _sides(side_lens)
    _check(lib().hmar_attn_bwd_noalloc(_ptr(q), _ptr(k), _ptr(v), _ptr(out), _ptr(lse), _ptr(dout), _ptr(dq),
                                       _ptr(dk), _ptr(dv), B, H, D, n, sides, float(softmax_scale),
                                       _stream(stream)), "hmar_attn_bwd_noalloc")
    return dq, dk, dv


def hmar_attn_scale_step(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale,
                         out=None, lse=None, want_lse=True, stream=None):
    """Inference step of one scale. q, k_cur, v_cur: [B,H,side_cur^2,D]; k_prev, v_prev:
    [B,H,side_prev^2,D] or None when side_prev == 0. Returns (out, lse or None)."""
    return _done(_host().scale_step(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale, out, lse, want_lse,
                                    _handle(stream)), "hmar_attn_scale_step")


def hmar_attn_scale_step_strided(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale,
                                 out=None, lse=None, want_lse=True, stream=None):
    """Inference step on views whose heads are not packed back to back, e.g. slices of one K/V ring
    [B,H,ring_rows,D] (k_prev = ring[:, :, a:a+n_prev], k_cur = ring[:, :, a+n_prev:a+n_prev+n_cur]).
    Every tensor is a [B,H,rows,D] view with contiguous rows and heads a constant stride apart."""
    return _done(_host().scale_step_strided(q, k_prev, v_prev, k_cur, v_cur, side_prev, side_cur, softmax_scale, out, lse, want_lse,
                                            _handle(stream)), "hmar_attn_scale_step_strided")


def hmar_recon_accumulate(xhat, codebook, tokens_new, tokens_old=None, mask=None, tokens_out=None, stream=None):
    """xhat [B,C,S,S] fp32 += bicubic(lookup(codebook [V,C], selected tokens [B,s,s])); returns xhat.
    `mask` (uint8 [B,s,s]) chooses tokens_new over tokens_old per position; `tokens_out` receives the selection."""
    return _done(_host().recon_accumulate(xhat, codebook, tokens_new, tokens_old, mask, tokens_out, _handle(stream)),
                 "hmar_recon_accumulate")


def hmar_recon_downsample(xhat, out_side, out=None, stream=None):
    """Area interpolation of xhat [B,C,S,S] fp32 down to [B,C,out_side,out_side]; returns the result."""
    return _done(_host().recon_downsample(xhat, out_side, out, _handle(stream)), "hmar_recon_downsample")


def hmar_schedule_tiles(side_lens, direction, window=HMAR_WINDOW_MARKOV):
    """Work list of one head as a list of dicts (host only; needs no GPU)."""
    sides, n = _sides(side_lens)
    count = lib().hmar_schedule_tiles_window(n, sides, int(window), int(direction), None, 0)
    if count < 0:
        raise HmarError(count, "hmar_schedule_tiles")
    buf = (ctypes.c_int32 * (6 * count))()
    lib().hmar_schedule_tiles_window(n, sides, int(window), int(direction), buf, count)
    keys = ("row_begin", "row_count", "partner_begin", "partner_end", "uniform", "cost")
    return [dict(zip(keys, buf[6 * t:6 * t + 6])) for t in range(count)]


def hmar_schedule_bwd_items(side_lens, n_heads, n_blocks, window=HMAR_WINDOW_MARKOV):
    """The backward's items as (block, head, first key row, steps), block by block in the order in which the blocks take
    them (host only; needs no GPU)."""
    sides, n = _sides(side_lens)
    count = lib().hmar_schedule_bwd_items(n, sides, int(window), int(n_heads), int(n_blocks), None, 0)
    if count < 0:
        raise HmarError(count, "hmar_schedule_bwd_items")
    buf = (ctypes.c_int32 * (4 * count))()
    lib().hmar_schedule_bwd_items(n, sides, int(window), int(n_heads), int(n_blocks), buf, count)
    flat = list(buf)
    return [tuple(flat[4 * t:4 * t + 4]) for t in range(count)]


def hmar_schedule_bwd_full_tile_share(side_lens, window=HMAR_WINDOW_MARKOV):
    """Thousandths of a head's backward steps that lie in full tiles (host only; needs no GPU)."""
    sides, n = _sides(side_lens)
    share = lib().hmar_schedule_bwd_full_tile_share(n, sides, int(window))
    if share < 0:
        raise HmarError(share, "hmar_schedule_bwd_full_tile_share")
    return share


def hmar_device_status():
    """(status, detail) recorded by the kernels since the last call; synchronises the device."""
    detail = ctypes.c_int(0)
    status = lib().hmar_device_status(ctypes.byref(detail))
    return status, detail.value


def hmar_selftest_bounded_wait(stream=None):
    """Launches the one-block kernel whose bounded wait must run out (see include/hmar.h)."""
    _check(lib().hmar_selftest_bounded_wait(_stream(stream)), "hmar_selftest_bounded_wait")


def hmar_profile_begin():
    lib().hmar_profile_begin()


def hmar_profile_end():
    """{kernel name: (launches, total_ms)} for the kernels launched since hmar_profile_begin()."""
    buf = ctypes.create_string_buffer(8192)
    _check(lib().hmar_profile_end(buf, len(buf)), "hmar_profile_end")
    out = {}
    for line in buf.value.decode().splitlines():
        name, count, ms = line.split()
        out[name] = (int(count), float(ms))
    return out


def hmar_debug_force_simt(enable):
    return lib().hmar_debug_force_simt(1 if enable else 0)


def hmar_launch_count():
    return int(lib().hmar_launch_count())


def hmar_shutdown():
    lib().hmar_shutdown()
