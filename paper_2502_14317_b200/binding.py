"""ctypes binding for libpc.so.  Same names as the C entry points, minus the ``pc_`` prefix.

Tensors are torch CUDA tensors; bf16 data is ``torch.bfloat16``.  Outputs and
workspaces are allocated here with torch (device memory only) unless passed in.
All calls enqueue on torch's current stream and do not synchronise.
"""
from __future__ import annotations

import ctypes
import functools
import importlib.util
import math
import os
from ctypes import c_float, c_int32, c_int64, c_size_t, c_void_p, c_char_p, POINTER, Structure

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
_LIB = None


class PcError(RuntimeError):
    pass


class _PrefillDesc(Structure):
    _fields_ = [("C", c_int32), ("L", c_int32), ("w", c_int32), ("Hq", c_int32), ("Hkv", c_int32), ("d", c_int32),
                ("rope_theta", c_float), ("softmax_scale", c_float),
                ("q_stride", c_int64 * 3), ("k_stride", c_int64 * 3), ("v_stride", c_int64 * 3),
                ("o_stride", c_int64 * 3)]


class _HotPathArgs(Structure):                             # pc_hot_path_args for callers through ctypes; hot_path fills it in csrc/pc_host.cpp
    _fields_ = [(n, c_void_p) for n in ("q", "k", "v", "q_win", "o", "k_rot", "win_score", "win_lse", "given_score", "chunk_score",
                                        "kept", "idx", "kc", "vc", "pos", "fg", "status_word", "ws_prefill")] + \
               [("ws_prefill_bytes", c_size_t), ("ws_parallel", c_void_p), ("ws_parallel_bytes", c_size_t),
                ("m", c_int32), ("k_keep", c_int32), ("n_score", c_int32), ("clear_status", c_int32)]


# outputs and workspaces of hot_path, in the order of csrc/pc_host.cpp
_HOT_PATH_BUFFERS = ("o", "k_rot", "win_score", "win_lse", "chunk_score", "kept", "idx", "kc", "vc", "pos", "fg", "status", "ws_prefill",
                     "ws_par")
_BAD_INPUT = "q, k and v must be bfloat16, k and v [C, L, Hkv, d] with the C, L and d of q, everything on one device"
_Strides = c_int64 * 3
_STAGES = (None, "pc_chunk_prefill_attn", "pc_select_chunks", "pc_score_select_chunks", "pc_select_tokens", "pc_gather_kv",
           "pc_parallel_attn")


def lib_path() -> str:
    return os.path.join(_HERE, "libpc.so")


def load_library():
    """Load libpc.so (built in-tree by ``python -m paper_2502_14317_b200.build``).  Fails loudly if absent."""
    global _LIB
    if _LIB is not None:
        return _LIB
    path = lib_path()
    if not os.path.exists(path):
        raise PcError(f"{path} not found: build it with `python -m paper_2502_14317_b200.build` "
                      "(there is no fallback path)")
    lib = ctypes.CDLL(path)
    lib.pc_status_string.restype = c_char_p
    lib.pc_status_string.argtypes = [c_int32]
    lib.pc_version.restype = c_int32
    lib.pc_chunk_prefill_attn_workspace_bytes.restype = c_size_t
    lib.pc_chunk_prefill_attn_workspace_bytes.argtypes = [POINTER(_PrefillDesc)]
    lib.pc_chunk_prefill_attn.restype = c_int32
    lib.pc_chunk_prefill_attn.argtypes = [POINTER(_PrefillDesc)] + [c_void_p] * 11 + [c_size_t, c_void_p]
    lib.pc_rope_position_reuse_workspace_bytes.restype = c_size_t
    lib.pc_rope_position_reuse_workspace_bytes.argtypes = [c_int32, c_int32]
    lib.pc_rope_position_reuse.restype = c_int32
    lib.pc_rope_position_reuse.argtypes = [c_void_p] + [c_int32] * 4 + [c_float, c_void_p, c_void_p, c_size_t, c_void_p]
    lib.pc_debug_bounded_wait_test.restype = c_int32
    lib.pc_debug_bounded_wait_test.argtypes = [c_int64, c_int32]
    lib.pc_launch_count.restype = ctypes.c_uint64
    lib.pc_launch_count.argtypes = []
    lib.pc_chunk_score_from_lse.restype = c_int32
    lib.pc_chunk_score_from_lse.argtypes = [c_void_p, c_int32, c_int32, c_int32, c_void_p, c_void_p]
    lib.pc_score_select_chunks.restype = c_int32
    lib.pc_score_select_chunks.argtypes = [c_void_p] + [c_int32] * 5 + [c_void_p, c_void_p, c_void_p]
    lib.pc_select_chunks.restype = c_int32
    lib.pc_select_chunks.argtypes = [c_void_p, c_int32, c_int32, c_int32, c_void_p, c_void_p]
    lib.pc_select_tokens.restype = c_int32
    lib.pc_select_tokens.argtypes = [c_void_p, c_void_p] + [c_int32] * 6 + [c_void_p, c_void_p]
    lib.pc_select_tokens_calibrated.restype = c_int32
    lib.pc_select_tokens_calibrated.argtypes = [c_void_p, c_void_p] + [c_int32] * 8 + [c_float] * 3 + [c_void_p, c_void_p]
    lib.pc_gather_kv.restype = c_int32
    lib.pc_gather_kv.argtypes = [c_void_p, c_void_p, POINTER(c_int64), c_void_p, c_void_p] + [c_int32] * 4 + \
                                [c_void_p, c_void_p, c_void_p, c_void_p]
    lib.pc_queue_init.restype = c_int32
    lib.pc_queue_init.argtypes = [c_int32, c_void_p, c_void_p, c_void_p]
    lib.pc_queue_update.restype = c_int32
    lib.pc_queue_update.argtypes = [c_void_p] + [c_int32] * 4 + [c_void_p] * 4
    lib.pc_queue_gather.restype = c_int32
    lib.pc_queue_gather.argtypes = [c_void_p, c_void_p, POINTER(c_int64), c_void_p, c_void_p] + [c_int32] * 4 + \
        [c_void_p] * 4
    lib.pc_queue_select_gather.restype = c_int32
    lib.pc_queue_select_gather.argtypes = [c_void_p, c_void_p, c_void_p, POINTER(c_int64), c_void_p] + [c_int32] * 6 + [c_void_p] * 4
    lib.pc_queue_emit.restype = c_int32
    lib.pc_queue_emit.argtypes = [c_void_p] + [c_int32] * 4 + [c_void_p] * 9
    lib.pc_parallel_attn_workspace_bytes.restype = c_size_t
    lib.pc_parallel_attn_workspace_bytes.argtypes = [c_int32] * 6
    lib.pc_parallel_attn.restype = c_int32
    lib.pc_parallel_attn.argtypes = [c_int32] * 6 + [c_void_p, c_int32, c_float, c_float] + [c_void_p] * 8 + \
                                    [c_size_t, c_void_p]
    lib.pc_parallel_attn_append.restype = c_int32
    lib.pc_parallel_attn_append.argtypes = [c_int32] * 7 + [c_void_p, c_int32, c_float, c_float] + [c_void_p] * 8 + \
                                           [c_size_t, c_void_p]
    lib.pc_hot_path_workspace_bytes.restype = c_size_t
    lib.pc_hot_path_workspace_bytes.argtypes = [POINTER(_PrefillDesc), c_int32, c_int32, POINTER(c_size_t)]
    lib.pc_hot_path.restype = c_int32
    lib.pc_hot_path.argtypes = [POINTER(_PrefillDesc), POINTER(_HotPathArgs), POINTER(c_int32), c_void_p]
    lib.pc_parallel_attn_static_scratch_bytes.restype = c_size_t
    lib.pc_parallel_attn_static_scratch_bytes.argtypes = []
    lib.pc_parallel_attn_static.restype = c_int32
    lib.pc_parallel_attn_static.argtypes = [c_int32] * 6 + [c_void_p, c_int32, c_float, c_float] + [c_void_p] * 8
    _LIB = lib
    return lib


def _host_hot_path(lib):
    """hot_path of csrc/pc_host.cpp on this library's entry points."""
    call = getattr(lib, "_host_hot_path", None)
    if call is None:
        from .build import host_path
        path = host_path(torch.__version__)
        try:
            spec = importlib.util.spec_from_file_location(__package__ + "._pc_host", path)
            module = importlib.util.module_from_spec(spec)
            spec.loader.exec_module(module)
        except ImportError as e:
            raise PcError("%s cannot be loaded: build it with `python -m paper_2502_14317_b200.build` (%s)" % (path, e)) from e
        address = lambda f: ctypes.cast(f, c_void_p).value
        call = lib._host_hot_path = functools.partial(module.hot_path, address(lib.pc_hot_path_workspace_bytes), address(lib.pc_hot_path))
    return call


def version() -> int:
    return int(load_library().pc_version())


def launch_count() -> int:
    """pc_launch_count: kernels launched by the library in this process so far."""
    return int(load_library().pc_launch_count())


def status_string(code: int) -> str:
    return load_library().pc_status_string(int(code)).decode()


def _check(rc: int, what: str):
    if rc != 0:
        raise PcError(f"{what} failed: {status_string(rc)} ({rc})")


def _ptr(t):
    return None if t is None else t.data_ptr()


def _stream():
    """The current stream of the current device as an integer.  (torch.cuda.current_stream() builds a Stream object and looks
    the device up again: 7 us a call, a quarter of the host time of a short prompt through the whole path.)"""
    return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())


def _like(t, shape):
    """New contiguous bf16 tensor on t's device (empty_like is the cheapest way to get one).  Its strides are those of its
    shape: t may count as contiguous with any stride in a dimension of one entry."""
    if t.dtype is torch.bfloat16 and t.shape == shape and t.is_contiguous():
        return torch.empty_like(t, memory_format=torch.contiguous_format)
    return t.new_empty(shape, dtype=torch.bfloat16)


def _same_rows(a, b):
    """Whether the strides of a serve b too: equal wherever a dimension has more than one entry, the innermost contiguous."""
    sa, sb = a.stride(), b.stride()
    return sa[3] == 1 and (sa == sb or (sb[3] == 1 and all(x == y or n == 1 for x, y, n in zip(sa, sb, a.shape))))


def _window(t, L, w):
    """The window rows of chunk 0, [1,w,H,d], contiguous: a view where the storage allows it."""
    s = t.stride()
    v = t.as_strided((1, w, t.shape[2], t.shape[3]), s, t.storage_offset() + (L - w) * s[1])
    return v if v.is_contiguous() else v.contiguous()


def _need_cuda(*tensors):
    for t in tensors:
        if t is not None and not t.is_cuda:
            raise PcError("tensors must live on a CUDA device")


def _let_go(t, stream=None):
    """A kept tensor is about to be dropped.  Its memory belongs to the stream it was made on; the calls that used it may have been on the
    present one, and it is not given out again before that has come here."""
    if t is not None and t.is_cuda:
        t.record_stream(torch.cuda.current_stream(t.device) if stream is None else stream)


def _kept(b, name, shape, dtype, device):
    """Tensor ``name`` of the buffers b for an output of this shape, as csrc/pc_host.cpp takes it: as it is, or a view of its first elements
    where it has enough of them (an earlier call had other sizes); None (make a new one) where it is absent or too small."""
    t = b.get(name)
    if t is None:
        return None
    if t.dtype is not dtype or t.device != device or not (t.is_contiguous() or (name == "o" and t.shape == shape)):
        raise PcError("buffers[%r] is of another type or device, or not contiguous" % name)
    if t.shape == shape:
        return t
    n = math.prod(shape)
    if t.numel() >= n:
        return t.view(-1)[:n].view(shape)
    _let_go(t)
    return None


def _check_inputs(q, k, v, dev):
    """The launches go by q's sizes: keys and values of others would be read out of range."""
    C, L, _, d = q.shape
    rows = (L, k.shape[2], d)
    if not (k.shape[1:] == v.shape[1:] == rows and k.shape[0] >= C and v.shape[0] >= C and
            q.dtype is k.dtype is v.dtype is torch.bfloat16 and q.device == k.device == v.device == dev):
        raise PcError(_BAD_INPUT)


def _make_desc(q, k, v, o, w, rope_theta, softmax_scale):
    C, L, Hq, d = q.shape
    Hkv = k.shape[2]
    sq, sk, sv, so = q.stride(), k.stride(), v.stride(), o.stride()
    if not sq[3] == sk[3] == sv[3] == so[3] == 1:
        raise PcError("head dimension must be contiguous")
    return _PrefillDesc(C, L, w, Hq, Hkv, d, float(rope_theta), float(softmax_scale), sq[:3], sk[:3], sv[:3], so[:3])


def chunk_prefill_attn_workspace_bytes(C, L, w, Hq, Hkv, d, k_rot_in_workspace=False) -> int:
    desc = _PrefillDesc(C, L, w, Hq, Hkv, d, 10000.0, 0.0)
    need = int(load_library().pc_chunk_prefill_attn_workspace_bytes(ctypes.byref(desc)))
    if need and k_rot_in_workspace:                           # rotated keys in the workspace (k_rot = NULL in the call)
        need += (C * L * Hkv * d * 2 + 255) // 256 * 256
    return need


def chunk_prefill_attn(q, k, v, *, w, rope_theta, softmax_scale=0.0, want_lse=False, out=None, k_rot=None,
                       win_score=None, win_lse=None, lse=None, status=None, workspace=None, chunk_len=None):
    """pc_chunk_prefill_attn: q [C,L,Hq,d], k/v [C,L,Hkv,d] bf16 (pre-RoPE); chunk_len: int32 [C] device tensor
    (tokens per chunk, window included) or None for full chunks.

    Returns dict(o, k_rot, win_score, win_lse, lse, status, workspace).
    """
    lib = load_library()
    _need_cuda(q, k, v)
    C, L, Hq, d = q.shape
    Hkv = k.shape[2]
    dev = q.device
    o = _like(q, q.shape) if out is None else out
    if k_rot is None:
        k_rot = _like(k, k.shape)
    if win_score is None:
        win_score = torch.empty((C, Hkv, L), dtype=torch.float32, device=dev)
    if win_lse is None:
        win_lse = torch.empty((C, Hq, w), dtype=torch.float32, device=dev)
    if lse is None and want_lse:
        lse = torch.empty((C, Hq, L), dtype=torch.float32, device=dev)
    if status is None:
        status = torch.zeros(1, dtype=torch.int32, device=dev)
    desc = _make_desc(q, k, v, o, w, rope_theta, softmax_scale)
    need = int(lib.pc_chunk_prefill_attn_workspace_bytes(ctypes.byref(desc)))
    if workspace is None or workspace.numel() < need:          # need == 0: a bad descriptor, which the call below names
        _let_go(workspace)
        workspace = torch.empty(max(need, 16), dtype=torch.uint8, device=dev)
    if chunk_len is not None and (chunk_len.dtype != torch.int32 or chunk_len.numel() != C or not chunk_len.is_cuda):
        raise PcError("chunk_len must be an int32 CUDA tensor with one entry per chunk")
    rc = lib.pc_chunk_prefill_attn(ctypes.byref(desc), q.data_ptr(), k.data_ptr(), v.data_ptr(), _ptr(chunk_len), o.data_ptr(),
                                   k_rot.data_ptr(), _ptr(lse), win_score.data_ptr(), win_lse.data_ptr(), status.data_ptr(),
                                   workspace.data_ptr(), workspace.numel(), _stream())
    _check(rc, "pc_chunk_prefill_attn")
    return {"o": o, "k_rot": k_rot, "win_score": win_score, "win_lse": win_lse, "lse": lse, "status": status,
            "workspace": workspace}


def rope_position_reuse(x, *, rope_theta, out=None, workspace=None):
    """pc_rope_position_reuse: x [C,L,H,d] bf16 contiguous -> the rotated tensor (positions 0..L-1 in every chunk)."""
    lib = load_library()
    _need_cuda(x)
    if not x.is_contiguous():
        raise PcError("pc_rope_position_reuse takes a contiguous tensor")
    C, L, H, d = x.shape
    out = torch.empty_like(x) if out is None else out
    need = int(lib.pc_rope_position_reuse_workspace_bytes(L, d))
    if workspace is None or workspace.numel() < need:
        workspace = torch.empty(max(need, 16), dtype=torch.uint8, device=x.device)
    _check(lib.pc_rope_position_reuse(_ptr(x), C, L, H, d, float(rope_theta), _ptr(out), _ptr(workspace), workspace.numel(),
                                      _stream()), "pc_rope_position_reuse")
    return out


def chunk_score_from_lse(win_lse, out=None):
    """pc_chunk_score_from_lse: win_lse [C,Hq,w] fp32 -> [C] fp32."""
    lib = load_library()
    _need_cuda(win_lse)
    C, Hq, w = win_lse.shape
    out = torch.empty(C, dtype=torch.float32, device=win_lse.device) if out is None else out
    _check(lib.pc_chunk_score_from_lse(_ptr(win_lse), C, Hq, w, _ptr(out), _stream()), "pc_chunk_score_from_lse")
    return out


def select_chunks(chunk_score, m, lower_is_better=True, out=None):
    """pc_select_chunks: chunk_score [C] fp32 -> kept [m] int32 (ascending ids)."""
    lib = load_library()
    _need_cuda(chunk_score)
    C = chunk_score.numel()
    out = torch.empty(m, dtype=torch.int32, device=chunk_score.device) if out is None else out
    _check(lib.pc_select_chunks(_ptr(chunk_score), C, int(m), int(bool(lower_is_better)), _ptr(out), _stream()),
           "pc_select_chunks")
    return out


def score_select_chunks(win_lse, m, lower_is_better=True, score_out=None, kept_out=None):
    """pc_score_select_chunks: win_lse [C,Hq,w] fp32 -> (chunk_score [C] fp32, kept [m] int32), one launch for C <= 64."""
    lib = load_library()
    _need_cuda(win_lse)
    C, Hq, w = win_lse.shape
    score = torch.empty(C, dtype=torch.float32, device=win_lse.device) if score_out is None else score_out
    kept = torch.empty(m, dtype=torch.int32, device=win_lse.device) if kept_out is None else kept_out
    _check(lib.pc_score_select_chunks(_ptr(win_lse), C, Hq, w, int(m), int(bool(lower_is_better)), _ptr(score), _ptr(kept),
                                      _stream()), "pc_score_select_chunks")
    return score, kept


def select_tokens(win_score, kept, n_cand, k, out=None):
    """pc_select_tokens: win_score [C,Hkv,L] fp32, kept [m] int32 -> idx [m,Hkv,k] int32."""
    lib = load_library()
    _need_cuda(win_score, kept)
    C, Hkv, L = win_score.shape
    m = kept.numel()
    out = torch.empty((m, Hkv, k), dtype=torch.int32, device=win_score.device) if out is None else out
    _check(lib.pc_select_tokens(_ptr(win_score), _ptr(kept), C, m, Hkv, L, int(n_cand), int(k), _ptr(out), _stream()),
           "pc_select_tokens")
    return out


def select_tokens_calibrated(win_score, kept, n_cand, k, *, n_s=100, n_r=100, lambda_s=float("inf"),
                             lambda_m=float("inf"), lambda_r=float("inf"), out=None):
    """pc_select_tokens_calibrated: Eq. 8 eviction of over-attended tokens per region, then the top-k of Eq. 7."""
    lib = load_library()
    _need_cuda(win_score, kept)
    C, Hkv, L = win_score.shape
    m = kept.numel()
    out = torch.empty((m, Hkv, k), dtype=torch.int32, device=win_score.device) if out is None else out
    _check(lib.pc_select_tokens_calibrated(_ptr(win_score), _ptr(kept), C, m, Hkv, L, int(n_cand), int(k), int(n_s),
                                           int(n_r), float(lambda_s), float(lambda_m), float(lambda_r), _ptr(out),
                                           _stream()), "pc_select_tokens_calibrated")
    return out


def gather_kv(k_src, v_src, kept, idx, k_out=None, v_out=None, pos_out=None, want_pos=True):
    """pc_gather_kv: k_src/v_src [C,L,Hkv,d] bf16 -> (k_out, v_out [Hkv, m*k, d], pos [Hkv, m*k])."""
    lib = load_library()
    _need_cuda(k_src, v_src, kept, idx)
    C, L, Hkv, d = k_src.shape
    m, _, k = idx.shape
    dev = k_src.device
    if not _same_rows(k_src, v_src):
        raise PcError("k_src and v_src must share strides with a contiguous head dimension")
    k_out = _like(k_src, (Hkv, m * k, d)) if k_out is None else k_out
    v_out = _like(k_out, (Hkv, m * k, d)) if v_out is None else v_out
    if pos_out is None and want_pos:
        pos_out = torch.empty((Hkv, m * k), dtype=torch.int32, device=dev)
    strides = _Strides(*k_src.stride()[:3])
    _check(lib.pc_gather_kv(_ptr(k_src), _ptr(v_src), strides, _ptr(kept), _ptr(idx), m, Hkv, k, d, _ptr(k_out),
                            _ptr(v_out), _ptr(pos_out), _stream()), "pc_gather_kv")
    return k_out, v_out, pos_out


def queue_init(m, Hkv, k, d, device):
    """pc_queue_init: an empty online chunk queue of m slots with its slot storage.

    Returns the state dict {q_score [m] f32, q_chunk [m] i32, q_k, q_v [Hkv, m*k, d] bf16, q_pos [Hkv, m*k] i32,
    slot_src [m] i32}."""
    lib = load_library()
    st = {"q_score": torch.empty(m, dtype=torch.float32, device=device),
          "q_chunk": torch.empty(m, dtype=torch.int32, device=device),
          "q_k": torch.empty((Hkv, m * k, d), dtype=torch.bfloat16, device=device),
          "q_v": torch.empty((Hkv, m * k, d), dtype=torch.bfloat16, device=device),
          "q_pos": torch.empty((Hkv, m * k), dtype=torch.int32, device=device),
          "slot_src": torch.empty(m, dtype=torch.int32, device=device),
          "m": m, "Hkv": Hkv, "k": k, "d": d}
    _need_cuda(st["q_score"])
    _check(lib.pc_queue_init(m, _ptr(st["q_score"]), _ptr(st["q_chunk"]), _stream()), "pc_queue_init")
    return st


def queue_update(state, chunk_score, chunk_id0, lower_is_better=True):
    """pc_queue_update: push the scores of a batch of chunks (ids chunk_id0, chunk_id0 + 1, ...); fills state['slot_src']."""
    lib = load_library()
    _need_cuda(chunk_score)
    if chunk_score.dtype != torch.float32 or not chunk_score.is_contiguous():
        raise PcError("chunk_score must be contiguous float32")
    _check(lib.pc_queue_update(chunk_score.data_ptr(), chunk_score.numel(), int(chunk_id0), 1 if lower_is_better else 0, state["m"],
                               state["q_score"].data_ptr(), state["q_chunk"].data_ptr(), state["slot_src"].data_ptr(), _stream()),
           "pc_queue_update")
    return state["slot_src"]


def queue_gather(state, k_src, v_src, idx):
    """pc_queue_gather: move the compressed caches of the chunks that entered the queue into their slots.

    k_src/v_src [Cb,L,Hkv,d] bf16 (rotated keys, values of the batch), idx [Cb,Hkv,k] from select_tokens on all chunks."""
    lib = load_library()
    _need_cuda(k_src, v_src, idx)
    Cb, L, Hkv, d = k_src.shape
    if idx.shape != (Cb, Hkv, state["k"]) or Hkv != state["Hkv"] or d != state["d"]:
        raise PcError("idx must be [Cb, Hkv, k] for the queue's k; Hkv and d must match the queue")
    if not _same_rows(k_src, v_src):
        raise PcError("k_src and v_src must share strides with a contiguous head dimension")
    strides = _Strides(*k_src.stride()[:3])
    _check(lib.pc_queue_gather(_ptr(k_src), _ptr(v_src), strides, _ptr(state["slot_src"]), _ptr(idx), state["m"], Hkv,
                               state["k"], d, _ptr(state["q_k"]), _ptr(state["q_v"]), _ptr(state["q_pos"]), _stream()),
           "pc_queue_gather")


def queue_select_gather(state, win_score, k_src, v_src, n_cand):
    """pc_queue_select_gather: rank the tokens of the chunks that entered the queue and move their kept rows into
    their slots, one launch.  win_score [Cb,Hkv,L] fp32, k_src/v_src [Cb,L,Hkv,d] bf16 of the batch."""
    lib = load_library()
    _need_cuda(win_score, k_src, v_src)
    Cb, L, Hkv, d = k_src.shape
    if Hkv != state["Hkv"] or d != state["d"] or win_score.shape != (Cb, Hkv, L) or not win_score.is_contiguous():
        raise PcError("win_score must be contiguous [Cb, Hkv, L]; Hkv and d must match the queue")
    if not _same_rows(k_src, v_src):
        raise PcError("k_src and v_src must share strides with a contiguous head dimension")
    strides = _Strides(*k_src.stride()[:3])
    _check(lib.pc_queue_select_gather(win_score.data_ptr(), k_src.data_ptr(), v_src.data_ptr(), strides, state["slot_src"].data_ptr(),
                                      state["m"], Hkv, L, int(n_cand), state["k"], d, state["q_k"].data_ptr(), state["q_v"].data_ptr(),
                                      state["q_pos"].data_ptr(), _stream()), "pc_queue_select_gather")


def queue_emit(state, k_out=None, v_out=None, pos_out=None, kept_out=None):
    """pc_queue_emit: the surviving chunks in ascending id order -> (kept [m], k_out, v_out [Hkv, m*k, d], pos [Hkv, m*k])."""
    lib = load_library()
    m, Hkv, k, d = state["m"], state["Hkv"], state["k"], state["d"]
    dev = state["q_k"].device
    k_out = torch.empty((Hkv, m * k, d), dtype=torch.bfloat16, device=dev) if k_out is None else k_out
    v_out = torch.empty((Hkv, m * k, d), dtype=torch.bfloat16, device=dev) if v_out is None else v_out
    pos_out = torch.empty((Hkv, m * k), dtype=torch.int32, device=dev) if pos_out is None else pos_out
    kept_out = torch.empty(m, dtype=torch.int32, device=dev) if kept_out is None else kept_out
    order = state.get("slot_order")
    if order is None:
        order = state["slot_order"] = torch.empty(m, dtype=torch.int32, device=dev)
    _check(lib.pc_queue_emit(state["q_chunk"].data_ptr(), m, Hkv, k, d, state["q_k"].data_ptr(), state["q_v"].data_ptr(),
                             state["q_pos"].data_ptr(), kept_out.data_ptr(), order.data_ptr(), k_out.data_ptr(), v_out.data_ptr(),
                             pos_out.data_ptr(), _stream()), "pc_queue_emit")
    return kept_out, k_out, v_out, pos_out


def parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, Nk) -> int:
    return int(load_library().pc_parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, Nk))


def parallel_attn(q_win, k_cache, v_cache, k_win, v_win, *, q_pos0, rope_theta, softmax_scale=0.0, out=None,
                  lse_out=None, want_lse=False, status=None, workspace=None):
    """pc_parallel_attn: q_win [B,w,Hq,d] (pre-RoPE), k_cache/v_cache [B,Hkv,Nk,d], k_win/v_win [B,w,Hkv,d]."""
    lib = load_library()
    _need_cuda(q_win, k_cache, v_cache, k_win, v_win)
    B, w, Hq, d = q_win.shape
    Hkv, Nk = k_cache.shape[1], k_cache.shape[2]
    dev = q_win.device
    for t in (q_win, k_cache, v_cache, k_win, v_win):
        if not t.is_contiguous():
            raise PcError("pc_parallel_attn takes contiguous tensors")
    out = _like(q_win, q_win.shape) if out is None else out
    if lse_out is None and want_lse:
        lse_out = torch.empty((B, Hq, w), dtype=torch.float32, device=dev)
    if status is None:
        status = torch.zeros(1, dtype=torch.int32, device=dev)
    need = parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, Nk)
    if workspace is None or workspace.numel() < need:
        _let_go(workspace)
        workspace = torch.empty(max(need, 16), dtype=torch.uint8, device=dev)
    rc = lib.pc_parallel_attn(B, w, Hq, Hkv, d, Nk, q_win.data_ptr(), int(q_pos0), float(rope_theta), float(softmax_scale),
                              k_cache.data_ptr(), v_cache.data_ptr(), k_win.data_ptr(), v_win.data_ptr(), out.data_ptr(), _ptr(lse_out),
                              status.data_ptr(), workspace.data_ptr(), workspace.numel(), _stream())
    _check(rc, "pc_parallel_attn")
    return {"out": out, "lse": lse_out, "status": status, "workspace": workspace}


def parallel_attn_append(q_win, k_cache, v_cache, n_valid, k_win, v_win, *, q_pos0, rope_theta, softmax_scale=0.0,
                         out=None, lse_out=None, want_lse=False, status=None, workspace=None):
    """pc_parallel_attn_append: as parallel_attn over the first ``n_valid`` entries of k_cache / v_cache
    [B,Hkv,Nk_cap,d]; afterwards k_win, v_win are written to entries n_valid .. n_valid + w - 1 of the caches."""
    lib = load_library()
    _need_cuda(q_win, k_cache, v_cache, k_win, v_win)
    B, w, Hq, d = q_win.shape
    Hkv, cap = k_cache.shape[1], k_cache.shape[2]
    dev = q_win.device
    for t in (q_win, k_cache, v_cache, k_win, v_win):
        if not t.is_contiguous():
            raise PcError("pc_parallel_attn_append takes contiguous tensors")
    out = _like(q_win, q_win.shape) if out is None else out
    if lse_out is None and want_lse:
        lse_out = torch.empty((B, Hq, w), dtype=torch.float32, device=dev)
    if status is None:
        status = torch.zeros(1, dtype=torch.int32, device=dev)
    need = parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, int(n_valid))
    if workspace is None or workspace.numel() < need:
        workspace = torch.empty(max(need, 16), dtype=torch.uint8, device=dev)
    rc = lib.pc_parallel_attn_append(B, w, Hq, Hkv, d, int(n_valid), cap, _ptr(q_win), int(q_pos0), float(rope_theta),
                                     float(softmax_scale), _ptr(k_cache), _ptr(v_cache), _ptr(k_win), _ptr(v_win),
                                     _ptr(out), _ptr(lse_out), _ptr(status), _ptr(workspace), workspace.numel(), _stream())
    _check(rc, "pc_parallel_attn_append")
    return {"out": out, "lse": lse_out, "status": status, "workspace": workspace}


def parallel_attn_static_scratch_bytes() -> int:
    return int(load_library().pc_parallel_attn_static_scratch_bytes())


def parallel_attn_static(q_win, k_cache, v_cache, k_win, v_win, out, *, q_pos0, rope_theta, softmax_scale=0.0,
                         lse_out=None, status=None):
    """pc_parallel_attn_static: pc_parallel_attn for callers that may not allocate device memory.

    Nothing is allocated here either: ``out`` (and ``lse_out`` / ``status`` if wanted) must be passed in, and
    the scratch is the fixed array inside the library.  Shapes that need more scratch than that array
    holds are refused.  Calls on one device share the array, so keep them on one stream.
    """
    lib = load_library()
    _need_cuda(q_win, k_cache, v_cache, k_win, v_win, out)
    B, w, Hq, d = q_win.shape
    Hkv, Nk = k_cache.shape[1], k_cache.shape[2]
    for t in (q_win, k_cache, v_cache, k_win, v_win, out):
        if not t.is_contiguous():
            raise PcError("pc_parallel_attn_static takes contiguous tensors")
    need, have = parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, Nk), parallel_attn_static_scratch_bytes()
    if need > have:
        raise PcError(f"pc_parallel_attn_static: this shape needs {need} bytes of scratch, the built-in array holds "
                      f"{have}; use pc_parallel_attn with a workspace instead")
    rc = lib.pc_parallel_attn_static(B, w, Hq, Hkv, d, Nk, _ptr(q_win), int(q_pos0), float(rope_theta),
                                     float(softmax_scale), _ptr(k_cache), _ptr(v_cache), _ptr(k_win), _ptr(v_win),
                                     _ptr(out), _ptr(lse_out), _ptr(status), _stream())
    _check(rc, "pc_parallel_attn_static")
    return out


def hot_path(q, k, v, *, w, rope_theta, m, k_keep, softmax_scale=0.0, chunk_score=None, buffers=None):
    """pc_hot_path: one pass of the whole path on the current stream, no host sync.

    ``chunk_score`` (device fp32 [C]) stands for the self-information of Eq. 3; if None the
    single-layer stand-in computed from the window log-sum-exp is used.
    ``buffers`` (dict) lets repeated calls reuse outputs and workspaces; what is too small for this call is replaced in it.
    """
    b = {} if buffers is None else buffers
    lib = load_library()
    _need_cuda(q, k, v, chunk_score)
    if chunk_score is not None and (chunk_score.dtype != torch.float32 or not chunk_score.is_contiguous()):
        raise PcError("chunk_score must be contiguous float32")
    C, L, Hq, d = q.shape
    Hkv = k.shape[2]
    m, k_keep = int(m), int(k_keep)
    get = b.get
    # new tensors in the place of those that are not there, workspaces, descriptor and call: csrc/pc_host.cpp
    rc, stage, out = _host_hot_path(lib)(_stream(), q, k, v, chunk_score, tuple([get(n) for n in _HOT_PATH_BUFFERS]),
                                         (C, L, Hq, Hkv, d, w, m, k_keep), float(rope_theta), float(softmax_scale))
    if rc != 0:
        if rc == 1:
            raise PcError("head dimension must be contiguous")
        if rc == 2:
            raise PcError("k_src and v_src must share strides with a contiguous head dimension")
        if rc == 3:
            raise PcError(_BAD_INPUT)
        if rc == 4:
            raise PcError("buffers[%r] is of another type or device, or not contiguous" % _HOT_PATH_BUFFERS[stage])
        _check(rc, _STAGES[stage])
    score = out[4]
    res = dict(zip(_HOT_PATH_BUFFERS, out))
    if buffers is not None:
        given = get("chunk_score") if chunk_score is not None else score
        buffers.update(res)
        buffers["chunk_score"] = given                         # a caller's scores are not a buffer
    return res


def hot_path_streaming(q, k, v, *, w, rope_theta, m, k_keep, batch=None, softmax_scale=0.0, chunk_score=None,
                       buffers=None):
    """The whole path with the chunks taken one batch at a time through the online chunk queue.

    Per batch: chunk-local attention, queue update, then the chunks that entered the queue are ranked per kv-head
    and their kept rows copied into their slots (one launch; a chunk that does not enter is dropped whole); the batch's outputs
    (attention output, rotated keys, window scores) live in buffers of batch size that the next batch
    overwrites, so device memory beyond the inputs is O(batch + m) chunks whatever C is.  After the last batch
    the queue is emitted in chunk order and the window attends over it.  Same results as :func:`hot_path`
    (kept chunks, indices and compressed cache bit for bit).

    q, k, v are either whole device tensors [C,L,*,d], cut into batches of ``batch`` chunks, or lists of
    per-batch tensors [Cb,L_b,*,d].  In a list the chunk length may differ from batch to batch (a shorter
    last chunk is a batch of its own: its window directly follows its context, and only the k_keep tokens it
    contributes persist); every L_b - w must be at least k_keep.  The query window of the global attention is
    taken from the first chunk of the first batch.  A caller that streams from elsewhere makes the same calls
    on its own batches.
    """
    b = {} if buffers is None else buffers
    if isinstance(q, (list, tuple)):
        batches = list(zip(q, k, v))
        for of_batch in batches:
            _check_inputs(*of_batch, batches[0][0].device)
    else:
        if batch is None:
            raise PcError("hot_path_streaming needs a batch size for whole tensors")
        _check_inputs(q, k, v, q.device)
        if batch >= q.shape[0] == k.shape[0] == v.shape[0] > 0:
            batches = [(q, k, v)]
        else:
            batches = [(q[c0:c0 + batch], k[c0:c0 + batch], v[c0:c0 + batch]) for c0 in range(0, q.shape[0], batch)]
    q0, k0, v0 = batches[0]
    _, L0, Hq, d = q0.shape
    Hkv = k0.shape[2]
    dev = q0.device
    f32, i32, bf16 = torch.float32, torch.int32, torch.bfloat16
    qu = b.get("queue")
    if qu is None or (qu["m"], qu["Hkv"], qu["k"], qu["d"], qu["q_k"].device) != (m, Hkv, k_keep, d, dev):
        for t in () if qu is None else qu.values():
            if torch.is_tensor(t):
                _let_go(t)
        b["queue"] = queue_init(m, Hkv, k_keep, d, dev)
    else:
        lib = load_library()
        _check(lib.pc_queue_init(m, _ptr(qu["q_score"]), _ptr(qu["q_chunk"]), _stream()), "pc_queue_init")
    qu = b["queue"]
    b["status"] = _kept(b, "status", (1,), i32, dev)
    c0 = 0
    k_win, fitted = None, {}
    for bq, bk, bv in batches:
        n, L, hq, dq = bq.shape
        hkv = bk.shape[2]
        if L - w < k_keep:
            raise PcError("a chunk of %d tokens has fewer than k_keep = %d context tokens" % (L, k_keep))
        pb = b.setdefault("pre_%dx%d" % (n, L), {})            # buffers per batch shape
        if fitted.get((n, L)) != (hq, hkv, dq):                # to this call's other sizes, with its first batch of the shape
            fitted[n, L] = hq, hkv, dq
            for name, shape, dtype in (("o", (n, L, hq, dq), bf16), ("k_rot", (n, L, hkv, dq), bf16), ("win_score", (n, hkv, L), f32),
                                       ("win_lse", (n, hq, w), f32), ("score", (n,), f32), ("idx", (n, hkv, k_keep), i32)):
                if name in pb:
                    pb[name] = _kept(pb, name, shape, dtype, dev)
        pre = chunk_prefill_attn(bq, bk, bv, w=w, rope_theta=rope_theta, softmax_scale=softmax_scale,
                                 out=pb.get("o"), k_rot=pb.get("k_rot"), win_score=pb.get("win_score"),
                                 win_lse=pb.get("win_lse"), status=b["status"], workspace=pb.get("workspace"))
        b["status"] = pre["status"]
        pb.update({"o": pre["o"], "k_rot": pre["k_rot"], "win_score": pre["win_score"], "win_lse": pre["win_lse"],
                   "workspace": pre["workspace"]})
        if chunk_score is not None:
            score = chunk_score[c0:c0 + n]
        else:
            score = chunk_score_from_lse(pre["win_lse"], out=pb.get("score"))
            pb["score"] = score
        queue_update(qu, score, c0, True)
        if k_keep <= 10240:                                    # rank and compact the chunks that entered, one launch
            queue_select_gather(qu, pre["win_score"], pre["k_rot"], bv, L - w)
        else:
            if "ids" not in b or b["ids"].numel() < n:
                _let_go(b.get("ids"))
                b["ids"] = torch.arange(n, dtype=torch.int32, device=dev)
            idx = select_tokens(pre["win_score"], b["ids"][:n], L - w, k_keep, out=pb.get("idx"))
            pb["idx"] = idx
            queue_gather(qu, pre["k_rot"], bv, idx)
        if k_win is None:                                      # the window is the same in every chunk: keep the first
            k_win = _kept(b, "k_win", (1, w, Hkv, d), bf16, dev)
            if k_win is None:
                k_win = torch.empty((1, w, Hkv, d), dtype=torch.bfloat16, device=dev)
            k_win.copy_(_window(pre["k_rot"], L, w))
            b["k_win"] = k_win
        c0 += n
    rows = (Hkv, m * k_keep)
    kept, kc, vc, pos = queue_emit(qu, k_out=_kept(b, "kc", (*rows, d), bf16, dev), v_out=_kept(b, "vc", (*rows, d), bf16, dev),
                                   pos_out=_kept(b, "pos", rows, i32, dev), kept_out=_kept(b, "kept", (m,), i32, dev))
    b.update({"kc": kc, "vc": vc, "pos": pos, "kept": kept})
    q_win, v_win = _window(q0, L0, w), _window(v0, L0, w)
    pa = parallel_attn(q_win, kc.unsqueeze(0), vc.unsqueeze(0), k_win, v_win, q_pos0=L0 - w, rope_theta=rope_theta,
                       softmax_scale=softmax_scale, out=_kept(b, "fg", (1, w, Hq, d), bf16, dev), status=b["status"], workspace=b.get("ws_par"))
    b.update({"fg": pa["out"], "ws_par": pa["workspace"]})
    return {"kept": kept, "kc": kc, "vc": vc, "pos": pos, "fg": pa["out"], "status": b["status"]}


def hot_path_from_host(hq, hk, hv, *, w, rope_theta, m, k_keep, softmax_scale=0.0, n_groups=4, buffers=None):
    """The whole path for inputs that live in pinned HOST memory (hq [C,L,Hq,d], hk/hv [C,L,Hkv,d], bf16).

    Chunks are independent until the chunk ranking, so they are uploaded in ``n_groups`` groups on a copy
    stream while the attention of the previous group runs on the current stream; the ranking, gather and
    parallel attention follow once all groups are done.  ``buffers`` (dict) keeps the device tensors,
    streams and events between calls.  Returns the same dict as :func:`hot_path` (device tensors).
    """
    b = {} if buffers is None else buffers
    C, L, Hq, d = hq.shape
    Hkv = hk.shape[2]
    dev = torch.device("cuda", torch.cuda.current_device())
    if not (hk.shape[1:] == hv.shape[1:] == (L, Hkv, d) and hk.shape[0] >= C and hv.shape[0] >= C):
        raise PcError("hk and hv must be [C, L, Hkv, d] with the C, L and d of hq")
    f32, i32, bf16 = torch.float32, torch.int32, torch.bfloat16
    for name, shape, dtype in (("q", hq.shape, bf16), ("k", hk.shape, bf16), ("v", hv.shape, bf16), ("o", hq.shape, bf16), ("k_rot", hk.shape, bf16),
                               ("win_score", (C, Hkv, L), f32), ("win_lse", (C, Hq, w), f32)):
        t = _kept(b, name, shape, dtype, dev)
        if t is None:
            if "copy_stream" in b:                              # a call that failed half-way may have left uploads into it
                _let_go(b.get(name), b["copy_stream"])
            t = torch.empty(shape, dtype=dtype, device=dev)
        b[name] = t
    t = _kept(b, "status", (1,), i32, dev)
    b["status"] = torch.zeros(1, dtype=i32, device=dev) if t is None else t
    if "copy_stream" not in b:
        b["copy_stream"], b["uploaded"] = torch.cuda.Stream(device=dev), []
    b["uploaded"] += [torch.cuda.Event() for _ in range(n_groups - len(b["uploaded"]))]
    q, k, v = b["q"], b["k"], b["v"]
    main, copy = torch.cuda.current_stream(), b["copy_stream"]
    copy.wait_stream(main)                       # the previous call may still read q, k, v
    bounds = [(g * C) // n_groups for g in range(n_groups + 1)]
    for g in range(n_groups):
        c0, c1 = bounds[g], bounds[g + 1]
        if c1 == c0:
            continue
        qg, kg, vg = q[c0:c1], k[c0:c1], v[c0:c1]
        with torch.cuda.stream(copy):
            qg.copy_(hq[c0:c1], non_blocking=True)
            kg.copy_(hk[c0:c1], non_blocking=True)
            vg.copy_(hv[c0:c1], non_blocking=True)
            b["uploaded"][g].record(copy)
        main.wait_event(b["uploaded"][g])
        pre = chunk_prefill_attn(qg, kg, vg, w=w, rope_theta=rope_theta, softmax_scale=softmax_scale,
                                 out=b["o"][c0:c1], k_rot=b["k_rot"][c0:c1], win_score=b["win_score"][c0:c1],
                                 win_lse=b["win_lse"][c0:c1], status=b["status"], workspace=b.get("ws_prefill"))
        b["ws_prefill"] = pre["workspace"]
    score, kept = score_select_chunks(b["win_lse"], m, True, score_out=_kept(b, "chunk_score", (C,), f32, dev),
                                      kept_out=_kept(b, "kept", (m,), i32, dev))
    idx = select_tokens(b["win_score"], kept, L - w, k_keep, out=_kept(b, "idx", (m, Hkv, k_keep), i32, dev))
    rows = (Hkv, m * k_keep)
    kc, vc, pos = gather_kv(b["k_rot"], v, kept, idx, k_out=_kept(b, "kc", (*rows, d), bf16, dev), v_out=_kept(b, "vc", (*rows, d), bf16, dev),
                            pos_out=_kept(b, "pos", rows, i32, dev))
    pa = parallel_attn(_window(q, L, w), kc.unsqueeze(0), vc.unsqueeze(0), _window(b["k_rot"], L, w), _window(v, L, w),
                       q_pos0=L - w, rope_theta=rope_theta, softmax_scale=softmax_scale, out=_kept(b, "fg", (1, w, Hq, d), bf16, dev),
                       status=b["status"], workspace=b.get("ws_par"))
    b.update(chunk_score=score, kept=kept, idx=idx, kc=kc, vc=vc, pos=pos, fg=pa["out"], ws_par=pa["workspace"])
    return {"o": b["o"], "k_rot": b["k_rot"], "win_score": b["win_score"], "win_lse": b["win_lse"], "chunk_score": score,
            "kept": kept, "idx": idx, "kc": kc, "vc": vc, "pos": pos, "fg": pa["out"], "status": b["status"]}
