"""CPU checks of what the C ABI does around its launches: its host code and the rotation's linked with a fake CUDA runtime
(fake_runtime.cpp), in which a chosen launch fails."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _fake(tmp_path_factory, *more):
    """libpc on the fake runtime: the entry points, the rotation and further source files."""
    from paper_2502_14317_b200 import binding, build
    csrc, out = build.CSRC, str(tmp_path_factory.mktemp("fake") / "libpc_fake.so")
    subprocess.run([build._nvcc(), "-shared", "-cudart", "none", "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17",
                    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", csrc, "-Xlinker", "-Bsymbolic", "-Xlinker", "--no-undefined",
                    os.path.join(ROOT, "tests", "fake_runtime.cpp"), "-o", out] +
                   [os.path.join(csrc, f) for f in ("pc_api.cu", "pc_rope.cu", "pc_static_scratch.cu", *more)],
                   check=True, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    with pytest.MonkeyPatch.context() as mp:
        mp.setattr(binding, "_LIB", None)
        mp.setattr(binding, "lib_path", lambda: out)
        return binding.load_library()


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return _fake(tmp_path_factory)


P = 1 << 20                                                       # a device address that nothing follows


def _desc(C=2, L=300, w=16, Hq=4, Hkv=2, d=128, v_stride=(0, 0, 0)):
    from paper_2502_14317_b200.binding import _PrefillDesc
    return _PrefillDesc(C, L, w, Hq, Hkv, d, 1e4, 0.0, (0, 0, 0), (0, 0, 0), v_stride, (0, 0, 0))


def _calls(lib):
    """name, call, launches of the rotation ahead of the attention"""
    big = 1 << 40
    desc = lambda **kw: ctypes.byref(_desc(**kw))
    prefill = lambda **kw: lib.pc_chunk_prefill_attn(desc(**kw), P, P, P, None, P, P, None, P, P, None, P, big, None)
    parallel = lambda B, w: lib.pc_parallel_attn(B, w, 8, 2, 128, 3000, P, 0, 1e4, 0.0, P, P, P, P, P, None, None, P, big, None)
    return [("rope, own tables", lambda: lib.pc_rope_position_reuse(P, 1, 100, 4, 64, 1e4, P, P, big, None), 1),
            ("rope, table kernel", lambda: lib.pc_rope_position_reuse(P, 4, 4096, 8, 128, 1e4, P, P, big, None), 2),
            ("prefill, own tables", lambda: prefill(), 1), ("prefill, table kernel", lambda: prefill(C=8, L=2000), 2),
            ("window", lambda: parallel(1, 64), 1), ("window, table kernel", lambda: parallel(64, 64), 2), ("few rows", lambda: parallel(1, 1), 0)]


@pytest.mark.parametrize("which", range(7))
def test_a_failed_launch_is_reported_by_the_call_that_made_it(fake, which):
    name, call, rotation = _calls(fake)[which]
    fake.fake_reset(-1)
    assert call() == 0
    n_attention = fake.fake_attention_launches()
    for at in range(rotation + n_attention):
        fake.fake_reset(at)
        assert call() == -4, f"{name}: launch {at} failed"
        if at < rotation:
            assert fake.fake_attention_launches() == 0, f"{name}: the attention ran on what a failed rotation left"
        assert fake.fake_last_error() == 0, f"{name}: the error is left to a later call"
        assert call() == 0


def _hot_path(lib, desc, n_score=None):
    from paper_2502_14317_b200.binding import _HotPathArgs
    a = _HotPathArgs(**{n: P for n, t in _HotPathArgs._fields_ if t is ctypes.c_void_p}, ws_prefill_bytes=1 << 40, ws_parallel_bytes=1 << 40,
                     m=1, k_keep=64, n_score=n_score or 0, clear_status=0)
    if n_score is None:
        a.given_score = None
    failed = ctypes.c_int32(-1)
    lib.fake_reset(-1)
    return lib.pc_hot_path(ctypes.byref(desc), ctypes.byref(a), ctypes.byref(failed), None), failed.value, lib.fake_attention_launches()


def test_whole_path_refuses_scores_of_chunks_that_do_not_exist(fake):
    """Before anything is launched; fewer scores than chunks rank the first chunks, as pc_select_chunks does."""
    assert _hot_path(fake, _desc(C=3), n_score=4) == (-1, 2, 0)
    for n in (1, 3, None):
        assert _hot_path(fake, _desc(C=3), n_score=n) == (0, 0, 2)


def test_whole_path_refuses_values_that_are_not_contiguous(fake):
    """The prefill takes strides of v, the stages behind it do not."""
    for v_stride in ((2 * 300 * 256, 256, 128), (300 * 256, 128, 300 * 128), (300 * 512, 512, 128)):
        assert _hot_path(fake, _desc(v_stride=v_stride)) == (-1, 1, 0), v_stride
    for C, Hkv, v_stride in ((2, 2, (0, 0, 0)), (2, 2, (300 * 256, 256, 128)), (1, 2, (900 * 256, 256, 128)), (2, 1, (300 * 128, 128, 38400))):
        assert _hot_path(fake, _desc(C=C, Hkv=Hkv, v_stride=v_stride)) == (0, 0, 2), v_stride


@pytest.mark.parametrize("B,w,Hq,Hkv,Nk,items", [
    (8, 32, 64, 4, 3000, 64), (16, 64, 16, 1, 4096, 64), (12, 128, 32, 8, 8192, 192),    # 512 rows a kv-head: one item of 512 would idle pairs
    (16, 128, 32, 8, 4096, 128), (64, 64, 64, 4, 8192, 512),                               # here it does not
])
def test_row_groups_that_fill_the_gpu(fake, B, w, Hq, Hkv, Nk, items):
    fake.fake_reset(-1)
    assert fake.pc_parallel_attn(B, w, Hq, Hkv, 128, Nk, P, 0, 1e4, 0.0, P, P, P, P, P, None, None, P, 1 << 40, None) == 0
    assert fake.fake_window_items() == items


def _host_call(lib, q, k, v, given=None, buffers={}, m=2, k_keep=64, w=16):
    from paper_2502_14317_b200.binding import _HOT_PATH_BUFFERS, _host_hot_path
    (C, L, Hq, d), Hkv = q.shape, k.shape[2]
    lib.fake_reset(-1)
    rc, stage, out = _host_hot_path(lib)(0, q, k, v, given, tuple([buffers.get(n) for n in _HOT_PATH_BUFFERS]), (C, L, Hq, Hkv, d, w, m, k_keep),
                                         1e4, 0.0)
    return rc, stage, dict(zip(_HOT_PATH_BUFFERS, out))


@pytest.mark.parametrize("d,Hq,Hkv,w", [(64, 4, 2, 16), (128, 6, 2, 1), (128, 4, 4, 128)])
def test_host_side_of_the_whole_path(fake, d, Hq, Hkv, w):
    """Tensors that are made, kept and replaced, on host memory and the fake runtime."""
    torch = pytest.importorskip("torch")
    from paper_2502_14317_b200 import build
    build.build_library()
    C, L, m, kk = 3, 300, 2, 64
    q, k, v = (torch.zeros((C, L, H, d), dtype=torch.bfloat16) for H in (Hq, Hkv, Hkv))
    shapes = {"o": q.shape, "k_rot": k.shape, "win_score": (C, Hkv, L), "win_lse": (C, Hq, w), "chunk_score": (C,), "kept": (m,),
              "idx": (m, Hkv, kk), "kc": (Hkv, m * kk, d), "vc": (Hkv, m * kk, d), "pos": (Hkv, m * kk), "fg": (1, w, Hq, d), "status": (1,)}
    types = {n: torch.bfloat16 if n in ("o", "k_rot", "kc", "vc", "fg") else torch.int32 if n in ("kept", "idx", "pos", "status") else torch.float32
             for n in shapes}
    rc, _, a = _host_call(fake, q, k, v, w=w)
    assert rc == 0 and fake.fake_attention_launches() == 2
    for n, s in shapes.items():
        assert a[n].shape == tuple(s) and a[n].dtype == types[n] and a[n].is_contiguous(), n
    assert a["ws_par"] is a["ws_prefill"] or a["ws_par"].numel() > a["ws_prefill"].numel()
    # everything is kept, a score of the caller's is passed on, a workspace that is too small is replaced
    score = torch.zeros(C)
    rc, _, b = _host_call(fake, q, k, v, given=score, buffers=a, w=w)
    assert rc == 0 and b["chunk_score"] is score and all(b[n] is a[n] for n in a if n != "chunk_score")
    small = torch.empty(16, dtype=torch.uint8)
    rc, _, b = _host_call(fake, q, k, v, buffers=dict(a, ws_prefill=small, ws_par=small, pos=None), w=w)
    assert rc == 0 and b["ws_prefill"].numel() == a["ws_prefill"].numel() and b["ws_par"].numel() >= 16 and b["pos"] is not a["pos"]
    assert all(b[n] is a[n] for n in shapes if n != "pos")
    # head-major queries go through a copy of the window; other strides of v are refused, as is a head dimension that is not innermost
    heads = torch.zeros((C, Hq, L, d), dtype=torch.bfloat16).transpose(1, 2)
    assert _host_call(fake, heads, k, v, w=w)[0] == 0
    assert _host_call(fake, q, k, torch.zeros((C, Hkv, L, d), dtype=torch.bfloat16).transpose(1, 2), w=w)[0] == (2 if Hkv > 1 else 0)
    assert _host_call(fake, torch.zeros((C, L, d, Hq), dtype=torch.bfloat16).transpose(2, 3), k, v, w=w)[0] == 1
    # the library's own refusals come back with their stage, arguments that are none as exceptions
    assert _host_call(fake, q, k, v, given=torch.zeros(C + 1), w=w)[:2] == (-1, 2)
    assert _host_call(fake, q, k, v, w=w, m=C + 1)[0] == -1
    with pytest.raises(TypeError):
        _host_call(fake, q, k, v, given=3.0, w=w)
    with pytest.raises(RuntimeError):
        _host_call(fake, q, k, v, w=w, k_keep=-1)


@pytest.mark.parametrize("d,Hq,Hkv,w", [(64, 4, 2, 16), (128, 6, 2, 1), (128, 4, 4, 128), (64, 4, 1, 16)])
def test_small_workspaces_and_strides_of_the_values(fake, d, Hq, Hkv, w):
    torch = pytest.importorskip("torch")
    C, L, m, kk = 3, 300, 2, 64
    q, k, v = (torch.zeros((C, L, H, d), dtype=torch.bfloat16) for H in (Hq, Hkv, Hkv))
    small, need_par = torch.empty(16, dtype=torch.uint8), ctypes.c_size_t()
    need = fake.pc_hot_path_workspace_bytes(ctypes.byref(_desc(C, L, w, Hq, Hkv, d)), m, kk, ctypes.byref(need_par))
    rc, _, out = _host_call(fake, q, k, v, buffers={"ws_prefill": small, "ws_par": small}, w=w)
    assert rc == 0 and out["ws_prefill"].numel() >= need > small.numel() and out["ws_par"].numel() >= need_par.value > small.numel()
    # head-major values are packed with one kv-head, and refused with more
    heads = torch.zeros((C, Hkv, L, d), dtype=torch.bfloat16).transpose(1, 2)
    assert _host_call(fake, q, k, heads, w=w)[0] == (2 if Hkv > 1 else 0)


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("packed", [False, True])
def test_arguments_of_the_whole_path(fake, packed, given):
    """What pc_hot_path is called with: pointers and strides of the tensors that come back, sizes and flags."""
    torch = pytest.importorskip("torch")
    from paper_2502_14317_b200 import binding
    C, L, Hq, Hkv, d, w, m, kk = 3, 300, 6, 2, 64, 16, 2, 70
    got = {}

    @ctypes.CFUNCTYPE(ctypes.c_int32, ctypes.POINTER(binding._PrefillDesc), ctypes.POINTER(binding._HotPathArgs), ctypes.POINTER(ctypes.c_int32), ctypes.c_void_p)
    def run(desc, args, failed, stream):
        read = lambda s: {n: list(x) if isinstance(x, ctypes.Array) else x for n, x in ((n, getattr(s, n)) for n, _ in s._fields_)}
        got.update(read(args[0]), desc=read(desc[0]), stream=stream)
        if got["q_win"] != q[0, L - w:].data_ptr():
            got["window"] = ctypes.string_at(got["q_win"], w * Hq * d * 2)
        return 0
    ints = lambda *size: torch.randint(-32768, 32767, size, dtype=torch.int16).view(torch.bfloat16)
    q, k, v, o = ints(C, L, Hq, d), ints(C, L, Hkv, d), ints(C, L, Hkv, d), ints(C, L, Hq, d)
    if not packed:                                                # head-major, and keys between others
        q, o, k = ints(C, Hq, L, d).transpose(1, 2), ints(C, Hq, L, d).transpose(1, 2), ints(C, L, 3 * Hkv, d)[:, :, Hkv:2 * Hkv]
    score = torch.zeros(C - 1) if given else None
    buffers = {"o": o} if packed else {"o": o, "status": torch.zeros(1, dtype=torch.int32)}
    call = binding._host_hot_path(fake)
    rc, _, out = call.func(call.args[0], ctypes.cast(run, ctypes.c_void_p).value, 77, q, k, v, score,
                           tuple([buffers.get(n) for n in binding._HOT_PATH_BUFFERS]), (C, L, Hq, Hkv, d, w, m, kk), 5e5, 0.25)
    out = dict(zip(binding._HOT_PATH_BUFFERS, out))
    assert rc == 0 and out["o"] is o
    for n, t in dict(out, q=q, k=k, v=v).items():
        field = {"status": "status_word", "ws_par": "ws_parallel"}.get(n, n)
        assert got[field] == t.data_ptr(), n
    assert got["given_score"] == (score.data_ptr() if given else None) and got["n_score"] == (C - 1 if given else C)
    assert (got["m"], got["k_keep"], got["clear_status"], got["stream"]) == (m, kk, packed, 77)
    assert (got["ws_prefill_bytes"], got["ws_parallel_bytes"]) == (out["ws_prefill"].numel(), out["ws_par"].numel())
    assert got["desc"] == dict(C=C, L=L, w=w, Hq=Hq, Hkv=Hkv, d=d, rope_theta=5e5, softmax_scale=0.25,
                               **{n + "_stride": list(t.stride()[:3]) for n, t in (("q", q), ("k", k), ("v", v), ("o", o))})
    if packed:
        assert got["q_win"] == q[0, L - w:].data_ptr()
    else:
        assert got["window"] == q[0, L - w:].contiguous().view(torch.int16).numpy().tobytes()


def _path_shapes(C, L, Hq, Hkv, d, w, m, k_keep):
    return {"o": (C, L, Hq, d), "k_rot": (C, L, Hkv, d), "win_score": (C, Hkv, L), "win_lse": (C, Hq, w), "chunk_score": (C,), "kept": (m,),
            "idx": (m, Hkv, k_keep), "kc": (Hkv, m * k_keep, d), "vc": (Hkv, m * k_keep, d), "pos": (Hkv, m * k_keep), "fg": (1, w, Hq, d),
            "status": (1,)}


def _zeros(torch, C, L, Hq, Hkv, d):
    return tuple(torch.zeros((C, L, H, d), dtype=torch.bfloat16) for H in (Hq, Hkv, Hkv))


def test_whole_path_with_buffers_of_another_call(fake):
    """The launches go by the sizes of this call: what an earlier call of other sizes left is big enough, or replaced, and has this call's shape."""
    torch = pytest.importorskip("torch")
    sizes = [(3, 300, 4, 2, 64, 16, 2, 64), (6, 900, 8, 2, 128, 16, 4, 128), (2, 200, 4, 4, 64, 8, 1, 64), (3, 300, 4, 2, 64, 64, 2, 65), (3, 300, 4, 1, 64, 64, 3, 64)]
    kept = {}
    for C, L, Hq, Hkv, d, w, m, kk in sizes:
        rc, _, kept = _host_call(fake, *_zeros(torch, C, L, Hq, Hkv, d), buffers=kept, w=w, m=m, k_keep=kk)
        assert rc == 0
        for n, s in _path_shapes(C, L, Hq, Hkv, d, w, m, kk).items():
            assert kept[n].shape == s and kept[n].is_contiguous(), n
    # the caller's own memory is written wherever it is big enough
    C, L, Hq, Hkv, d, w, m, kk = sizes[0]
    flat = torch.empty(Hkv * m * kk * d + 8, dtype=torch.bfloat16)
    strided = torch.empty((C, Hq, L, d), dtype=torch.bfloat16).transpose(1, 2)
    rc, _, out = _host_call(fake, *_zeros(torch, C, L, Hq, Hkv, d), buffers={"kc": flat, "vc": flat[8:].view(-1, d), "o": strided}, w=w, m=m, k_keep=kk)
    assert rc == 0 and out["kc"].data_ptr() == flat.data_ptr() and out["vc"].data_ptr() == flat[8:].data_ptr() and out["o"] is strided
    assert out["kc"].shape == out["vc"].shape == (Hkv, m * kk, d)


def test_whole_path_refuses_tensors_that_do_not_go_together(fake):
    torch = pytest.importorskip("torch")
    from paper_2502_14317_b200.binding import _HOT_PATH_BUFFERS
    q, k, v = _zeros(torch, 6, 900, 4, 2, 64)
    assert _host_call(fake, q, k, v)[0] == 0
    for wrong in (k[:3], k[:, :300], k[..., :32], k.float(), k.half()):
        assert _host_call(fake, q, wrong, v)[0] == 3 and fake.fake_attention_launches() == 0
        assert _host_call(fake, q, k, wrong)[0] == 3 and fake.fake_attention_launches() == 0
    assert _host_call(fake, q, k, v[:, :, :1])[0] == 3 and _host_call(fake, q.float(), k, v)[0] == 3
    assert _host_call(fake, q, k.to("meta"), v)[0] == 3 and _host_call(fake, q, k, v, given=torch.zeros(6, device="meta"))[0] == 3
    assert _host_call(fake, q[:5], k, v)[0] == _host_call(fake, q[:5], k[:5], v)[0] == 0       # chunks that no query asks for
    good = _host_call(fake, q, k, v)[2]
    for n, t in good.items():
        wrong = [t.to("meta")] + ([t.new_empty(t.numel() * 2)[::2]] if t.numel() > 1 else []) + ([] if n.startswith("ws") else [t.double()])
        for bad in wrong:
            assert _host_call(fake, q, k, v, buffers=dict(good, **{n: bad}))[:2] == (4, _HOT_PATH_BUFFERS.index(n)), n
            assert fake.fake_attention_launches() == 0


@pytest.fixture
def on_host(fake, monkeypatch):
    """The binding's calls on host memory and the fake runtime."""
    from paper_2502_14317_b200 import binding
    monkeypatch.setattr(binding, "_LIB", fake)
    monkeypatch.setattr(binding, "_need_cuda", lambda *tensors: None)
    monkeypatch.setattr(binding, "_stream", lambda: 0)
    return binding


def _stream_sizes():
    """C, L, Hq, Hkv, d, w, m, k_keep: larger, smaller and other heads; the batches have the same chunks and tokens throughout"""
    return [(4, 300, 4, 2, 64, 16, 2, 64), (4, 300, 8, 4, 128, 32, 4, 128), (4, 300, 2, 1, 64, 8, 1, 32), (4, 300, 4, 1, 128, 64, 3, 100)]


def _written(binding, monkeypatch):
    """Tensors that the streamed path's calls are given to write, with the sizes that the library writes."""
    seen = []
    prefill, emit, parallel, score = binding.chunk_prefill_attn, binding.queue_emit, binding.parallel_attn, binding.chunk_score_from_lse

    def spy_prefill(q, k, v, *, w, **kw):
        (C, L, Hq, d), Hkv = q.shape, k.shape[2]
        seen.extend((n, kw.get(n), s) for n, s in (("out", (C, L, Hq, d)), ("k_rot", (C, L, Hkv, d)), ("win_score", (C, Hkv, L)), ("win_lse", (C, Hq, w))))
        return prefill(q, k, v, w=w, **kw)

    def spy_emit(state, **kw):
        rows = (state["Hkv"], state["m"] * state["k"])
        seen.extend((n, kw.get(n), s) for n, s in (("k_out", (*rows, state["d"])), ("v_out", (*rows, state["d"])), ("pos_out", rows), ("kept_out", (state["m"],))))
        return emit(state, **kw)

    def spy_parallel(q_win, *args, **kw):
        seen.append(("out", kw.get("out"), tuple(q_win.shape)))
        return parallel(q_win, *args, **kw)

    def spy_score(win_lse, out=None):
        seen.append(("score", out, (win_lse.shape[0],)))
        return score(win_lse, out=out)
    for n, f in (("chunk_prefill_attn", spy_prefill), ("queue_emit", spy_emit), ("parallel_attn", spy_parallel), ("chunk_score_from_lse", spy_score)):
        monkeypatch.setattr(binding, n, f)
    return seen


def test_streamed_path_with_buffers_of_another_call(on_host, monkeypatch):
    torch = pytest.importorskip("torch")
    seen, b = _written(on_host, monkeypatch), {}
    for C, L, Hq, Hkv, d, w, m, kk in _stream_sizes():
        for _ in range(2):
            seen.clear()
            got = on_host.hot_path_streaming(*_zeros(torch, C, L, Hq, Hkv, d), w=w, rope_theta=1e4, m=m, k_keep=kk, batch=2, buffers=b)
            assert all(t is None or t.shape == s for _, t, s in seen), [(n, t.shape, s) for n, t, s in seen if t is not None and t.shape != s]
        assert all(t is not None for n, t, _ in seen), "everything is reused by a call of the same sizes"
        shapes = _path_shapes(C, L, Hq, Hkv, d, w, m, kk)
        assert all(got[n].shape == shapes[n] for n in ("kept", "kc", "vc", "pos", "fg", "status"))
        assert (b["queue"]["q_k"].shape, b["queue"]["q_score"].shape) == (shapes["kc"], (m,))
    q, k, v = _zeros(torch, 4, 300, 4, 2, 64)
    args = dict(w=16, rope_theta=1e4, m=2, k_keep=64, batch=2)
    for wrong in ((q, k[:, :200], v), (q, k, v[:, :, :1]), (q.float(), k, v), (q, k[:2], v[:2])):
        with pytest.raises(on_host.PcError, match="bfloat16|C, L"):
            on_host.hot_path_streaming(*wrong, **args)
        if wrong[0].shape[0] == 4:                                # in a list, where only the second batch is wrong
            parts = [(t[:2], t[2:]) for t in (q, k, v)]
            with pytest.raises(on_host.PcError, match="C, L"):
                on_host.hot_path_streaming(*([a, t[2:]] for (a, _), t in zip(parts, wrong)), **args)
    with pytest.raises(on_host.PcError, match="'kc'"):
        on_host.hot_path_streaming(q, k, v, buffers={"kc": torch.empty(2, 128, 64)}, **args)


def test_path_from_host_memory_with_buffers_of_another_call(on_host, monkeypatch):
    import contextlib
    import types
    torch = pytest.importorskip("torch")
    stream = types.SimpleNamespace(wait_stream=lambda other: None, wait_event=lambda event: None)
    cuda = types.SimpleNamespace(current_device=lambda: 0, current_stream=lambda: stream, Stream=lambda device: stream,
                                 stream=lambda s: contextlib.nullcontext(), Event=lambda: types.SimpleNamespace(record=lambda s: None))

    class OnHost:                                                 # torch with its GPU calls on host memory
        device = staticmethod(lambda *a: torch.device("cpu"))

        def __getattr__(self, name):
            return cuda if name == "cuda" else getattr(torch, name)
    monkeypatch.setattr(on_host, "torch", OnHost())
    b = {}
    for n_groups, (C, L, Hq, Hkv, d, w, m, kk) in zip((1, 3, 2, 4), _stream_sizes()):
        for extra in (0, 3):
            q, k, v = _zeros(torch, C + extra, L, Hq, Hkv, d)
            got = on_host.hot_path_from_host(q, k, v, w=w, rope_theta=1e4, m=m, k_keep=kk, n_groups=n_groups, buffers=b)
            assert all(got[n].shape == s for n, s in _path_shapes(C + extra, L, Hq, Hkv, d, w, m, kk).items())
    for wrong in ((q, k[:, :200], v), (q, k[:2], v), (q, k, v[:, :, :, :64])):
        with pytest.raises(on_host.PcError, match="C, L"):
            on_host.hot_path_from_host(*wrong, w=64, rope_theta=1e4, m=2, k_keep=64)


def test_grid_of_the_gather(tmp_path_factory):
    """More blocks than the SMs hold only where all the rows move: slots of the queue may keep theirs, which the host cannot see."""
    lib = _fake(tmp_path_factory, "pc_select_gather.cu")
    strides = (ctypes.c_int64 * 3)(8 << 20, 1024, 128)
    for m, Hkv, k, d, blocks in [(1, 1, 1, 64, 1), (1, 2, 100, 128, 13), (8, 8, 2048, 128, 1184), (8, 8, 2400, 128, 1184),
                                 (8, 8, 2401, 128, 9472), (8, 8, 10241, 128, 9472), (8, 16, 10241, 64, 9472)]:
        assert lib.pc_gather_kv(P, P, strides, P, P, m, Hkv, k, d, P, P, P, None) == 0 and lib.fake_last_grid() == blocks
        assert lib.pc_queue_gather(P, P, strides, P, P, m, Hkv, k, d, P, P, P, None) == 0 and lib.fake_last_grid() == min(blocks, 1184)
