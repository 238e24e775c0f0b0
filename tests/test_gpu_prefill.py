"""GPU parity: pc_chunk_prefill_attn against the CPU oracle, element by element (through the C ABI)."""
import numpy as np
import pytest
import torch

import pc_inputs
from oracle import parallelcomp_oracle as orc
from tests.gpu_util import to_dev, to_bits, to_f64, check_attention_output, check_scores

pytestmark = pytest.mark.gpu


def _run_and_compare(q, k, v, w, theta, want_lse=True, sharp=False):
    import paper_2502_14317_b200 as pc
    C, L, Hq, d = q.shape
    Hkv = k.shape[2]
    G = Hq // Hkv
    res = pc.chunk_prefill_attn(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=theta, want_lse=want_lse)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0, f"device wait ran out, code {int(res['status'].item())}"
    O, LSE, k_rot = orc.local_attention(q, k, v, theta)
    scale = 1.0 / np.sqrt(d)
    S, O_win, LSE_win = orc.window_scores(orc.rope_bf16(q, theta), k_rot, v, w, scale)
    # rotated keys: the rotation is evaluated in fp64 on both sides -> same bits
    assert np.array_equal(to_bits(res["k_rot"]), k_rot), "k_rot differs from the oracle"
    check_attention_output(to_f64(res["o"]), O, sharp=sharp)
    lse = res["lse"].cpu().numpy().astype(np.float64)
    assert np.abs(lse - LSE).max() <= 2e-3, f"LSE max err {np.abs(lse - LSE).max():.3e}"
    win_lse = res["win_lse"].cpu().numpy().astype(np.float64)
    assert np.abs(win_lse - LSE_win).max() <= 2e-3
    got_S = res["win_score"].cpu().numpy()
    check_scores(got_S, S, G, w, L)
    assert np.allclose(got_S.sum(-1), G * w, rtol=1e-4)        # Eq. 6: G*w softmax rows, each summing to 1
    return res


def test_cfg0_full(cfg0_inputs):
    cfg, inp = cfg0_inputs
    _run_and_compare(inp["q"], inp["k"], inp["v"], cfg.w, cfg.rope_theta)


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,theta", [
    (2, 384, 64, 4, 1, 128, 500000.0),     # GQA G=4 (two head pairs), d=128, three query tiles
    (2, 300, 16, 2, 2, 64, 10000.0),       # MHA (tile-pair mode), ragged last tile (300 = 2*128 + 44)
    (1, 200, 128, 2, 1, 64, 10000.0),      # window spans two tiles, ragged
    (3, 520, 8, 3, 3, 128, 10000.0),       # MHA, odd tile count (5 tiles), smallest window
    (1, 100, 32, 8, 1, 64, 10000.0),       # single ragged tile, G*w = 256 window rows
    (1, 640, 64, 8, 1, 128, 500000.0),     # G*w = 512 window rows: two score passes
    (1, 130, 64, 1, 1, 64, 10000.0),       # single head, MHA, two tiles with a 2-token tail
    # head size 128 runs on CTA pairs: four (q-head, query tile) blocks per pair
    (2, 300, 16, 2, 1, 128, 10000.0),      # G=2: two heads, two tiles a unit, ragged last tile
    (1, 100, 32, 1, 1, 128, 10000.0),      # MHA, a single ragged tile: one of the four blocks is there
    (1, 256, 128, 4, 2, 128, 500000.0),    # widest window = exactly the last tile, two kv-heads
    (2, 1100, 64, 6, 2, 128, 10000.0),     # G=3 (odd): units of four tiles of a head, 9 tiles, ragged
    (1, 1024, 8, 2, 2, 128, 10000.0),      # MHA, even tile count, smallest window
    (1, 200, 128, 8, 1, 128, 10000.0),     # G*w = 1024 window rows: four score passes, window over two tiles
    # windows that are no power of two (the sweep pads a head's rows to a multiple of 8 and leaves the pad out)
    (2, 400, 24, 4, 2, 128, 10000.0),      # CTA pairs, w = 24
    (1, 700, 100, 4, 1, 128, 500000.0),    # CTA pairs, w = 100 (the region size of App. C), window over two tiles
    (1, 300, 5, 2, 1, 128, 10000.0),       # CTA pairs, w = 5 < 8
    (1, 260, 1, 4, 2, 128, 10000.0),       # CTA pairs, a single query token
    (2, 400, 24, 3, 3, 128, 10000.0),      # multi-head, units of four tiles, w = 24
    (1, 520, 100, 6, 2, 128, 10000.0),     # G = 3, w = 100
    (2, 300, 24, 4, 2, 64, 10000.0),       # head size 64, w = 24
    (1, 333, 100, 2, 1, 64, 10000.0),      # head size 64, w = 100
    (1, 140, 3, 8, 2, 64, 10000.0),        # head size 64, w = 3
])
def test_shapes(C, L, w, Hq, Hkv, d, theta):
    rng = np.random.default_rng(L * 7 + Hq)
    q = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hq, d)).astype(np.float32))
    k = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hkv, d)).astype(np.float32))
    v = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hkv, d)).astype(np.float32))
    k[:, 0] = pc_inputs.f32_to_bf16_bits(pc_inputs.bf16_bits_to_f32(k[:, 0]) * np.float32(4.0))
    _run_and_compare(q, k, v, w, theta)


@pytest.mark.parametrize("L,Hq,Hkv,chunk_len", [
    (128, 1, 1, None), (129, 1, 1, None), (384, 3, 1, None), (512, 2, 2, None), (513, 1, 1, None), (770, 7, 1, None),   # G odd: units of 4 tiles
    (127, 2, 1, None), (256, 6, 1, None), (640, 4, 2, None),                     # G = 2 mod 4: units of 2 tiles, odd and even counts
    (385, 8, 1, None), (260, 12, 1, None),                                       # G = 0 mod 4: two and three sets of 4 heads
    (700, 5, 1, [700, 41, 129, 512]), (700, 2, 1, [257, 700]), (513, 4, 1, [384, 513, 41]),   # shorter chunks: absent blocks
])
def test_units_of_a_cta_pair(L, Hq, Hkv, chunk_len):
    """Head size 128: a pair of CTAs takes four (q-head, query tile) blocks at a time, which blocks depends on the
    group size; the edges are tile counts that do not fill a unit, windows that cross tiles and shorter chunks."""
    import paper_2502_14317_b200 as pc
    w, d, theta = 40, 128, 10000.0
    C = len(chunk_len) if chunk_len else 2
    rng = np.random.default_rng(L + 31 * Hq)
    q, k, v = (pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, h, d)).astype(np.float32)) for h in (Hq, Hkv, Hkv))
    if chunk_len is None:
        _run_and_compare(q, k, v, w, theta)
        return
    cl = torch.tensor(chunk_len, dtype=torch.int32, device="cuda")
    res = pc.chunk_prefill_attn(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=theta, want_lse=True, chunk_len=cl)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    for c, n in enumerate(chunk_len):
        O, LSE, k_rot = orc.local_attention(q[c:c + 1, :n], k[c:c + 1, :n], v[c:c + 1, :n], theta)
        S, _, _ = orc.window_scores(orc.rope_bf16(q[c:c + 1, :n], theta), k_rot, v[c:c + 1, :n], w, 1.0 / np.sqrt(d))
        check_attention_output(to_f64(res["o"][c:c + 1, :n]), O)
        assert np.abs(res["lse"][c:c + 1, :, :n].cpu().numpy() - LSE).max() <= 2e-3
        check_scores(res["win_score"][c:c + 1, :, :n].cpu().numpy(), S, Hq // Hkv, w, n)
        assert not res["o"][c, n:].any() and not res["win_score"][c, :, n:].any()


@pytest.mark.parametrize("C,L,w,Hq,Hkv,chunk_len", [
    (3, 100, 8, 32, 32, None), (10, 129, 100, 24, 8, None), (40, 256, 16, 6, 2, None), (20, 300, 24, 20, 4, None), (25, 384, 128, 9, 3, None),
    (38, 128, 1, 2, 2, None), (5, 384, 40, 16, 16, [384, 41, 129, 256, 300]), (3, 260, 64, 75, 25, [65, 260, 128]),
])
def test_short_chunks_of_odd_groups(C, L, w, Hq, Hkv, chunk_len):
    """Head size 128 on single CTAs: up to three query tiles, an odd number of q-heads per kv-head, more groups than CTA pairs."""
    if chunk_len is None:
        test_shapes(C, L, w, Hq, Hkv, 128, 10000.0)
    else:
        test_score_sweeps_as_items_of_their_own(C, L, w, Hq, Hkv, 128, chunk_len)


@pytest.mark.parametrize("d", [64, 128])
def test_growing_logits_rescale_path(d):
    """Keys whose norm grows along the chunk make the running row maximum jump by more than the lazy
    threshold again and again, so the accumulator is rescaled in most tiles (rare otherwise)."""
    rng = np.random.default_rng(99 + d)
    C, L, Hq, Hkv, w = 1, 700, 4, 2, 32
    q = rng.standard_normal((C, L, Hq, d)).astype(np.float32)
    k = rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    v = rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    k *= np.linspace(1.0, 40.0, L, dtype=np.float32)[None, :, None, None]
    bits = [pc_inputs.f32_to_bf16_bits(x) for x in (q, k, v)]
    _run_and_compare(bits[0], bits[1], bits[2], w, 10000.0, sharp=True)


@pytest.mark.parametrize("d,rise", [(64, 2.0), (64, 6.0), (128, 4.0), (128, 6.0)])
def test_logits_that_rise_less_than_the_threshold_a_tile(d, rise):
    """Every key tile lies `rise` (in log2) above the one before: no logit exceeds the reference maximum by 2^8, but 64
    probabilities of 2^rise sum up to more than 2^8 (rise = 2: about as much, so that some rows of a warp are raised and others are
    not).  The rise goes through the slowest pair, which the rotation leaves as it is.  (What is tested is the repeated half; that a
    logit is noticed in either half: the next test.)"""
    rng = np.random.default_rng(31 + d)
    C, L, Hq, Hkv, w = 1, 900, 4, 2, 32
    q = 0.3 * rng.standard_normal((C, L, Hq, d)).astype(np.float32)
    k = 0.3 * rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    v = rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    q[..., d // 2 - 1] = 8.0
    k[..., d // 2 - 1] = (np.arange(L) // 128 * rise * np.sqrt(d) / (8.0 * np.log2(np.e)))[None, :, None]
    bits = [pc_inputs.f32_to_bf16_bits(x) for x in (q, k, v)]
    _run_and_compare(bits[0], bits[1], bits[2], w, 1.0e9, sharp=True)


@pytest.mark.parametrize("d,Hq,Hkv", [(64, 4, 2), (128, 8, 2), (128, 4, 2), (128, 3, 1)])
@pytest.mark.parametrize("at", [266, 356])                 # in the first / in the second half of a key tile
def test_one_logit_far_above_the_others(d, Hq, Hkv, at):
    """A single key lies more than 2^130 above all the others: taken against the maximum of the tiles before, its probability is beyond
    fp32, so it has to be noticed in whichever half of a tile it stands, also by rows whose second half is masked (query rows 266 to
    319 for the key at 266).  It goes through the slowest pair, which the rotation leaves as it is."""
    rng = np.random.default_rng(at + d)
    C, L, w = 1, 700, 32
    q, k, v = (rng.standard_normal((C, L, h, d)).astype(np.float32) * g for h, g in ((Hq, 0.3), (Hkv, 0.3), (Hkv, 1.0)))
    q[..., d // 2 - 1], k[..., d // 2 - 1] = 8.0, 0.0
    k[:, at, :, d // 2 - 1] = 150.0 * np.sqrt(d) / (8.0 * np.log2(np.e))
    s = np.einsum("ihd,jd->hij", q[0, :, :Hq // Hkv], k[0, :, 0]) * (np.log2(np.e) / np.sqrt(d))
    with np.errstate(over="ignore"):
        assert np.isinf(np.exp2(s[:, at:, at] - s[:, at:, :at].max(-1)).astype(np.float32)).all()
    bits = [pc_inputs.f32_to_bf16_bits(x) for x in (q, k, v)]
    _run_and_compare(bits[0], bits[1], bits[2], w, 1.0e9, sharp=True)


@pytest.mark.parametrize("Hq,Hkv", [(4, 2), (2, 2), (6, 2)])
def test_growing_logits_many_tiles(Hq, Hkv):
    """The same stress over 13 key tiles, two chunks, even and odd group sizes: the softmax warpgroups and the TMEM
    buffers go through many rounds in which a warpgroup stalls in the rescale path while the other runs ahead,
    including across query blocks and the score sweep."""
    rng = np.random.default_rng(7 + Hq)
    C, L, w, d = 2, 1600, 64, 128
    q = rng.standard_normal((C, L, Hq, d)).astype(np.float32)
    k = rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    v = rng.standard_normal((C, L, Hkv, d)).astype(np.float32)
    k *= np.linspace(1.0, 60.0, L, dtype=np.float32)[None, :, None, None]
    bits = [pc_inputs.f32_to_bf16_bits(x) for x in (q, k, v)]
    _run_and_compare(bits[0], bits[1], bits[2], w, 10000.0, sharp=True)


def test_deterministic_and_strided(cfg0_inputs):
    import paper_2502_14317_b200 as pc
    cfg, inp = cfg0_inputs
    q, k, v = to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"])
    a = pc.chunk_prefill_attn(q, k, v, w=cfg.w, rope_theta=cfg.rope_theta)
    b = pc.chunk_prefill_attn(q, k, v, w=cfg.w, rope_theta=cfg.rope_theta)
    # head-major storage viewed token-major: same numbers through explicit strides
    qh = q.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    kh = k.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    vh = v.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    c = pc.chunk_prefill_attn(qh, kh, vh, w=cfg.w, rope_theta=cfg.rope_theta)
    torch.cuda.synchronize()
    for key in ("o", "k_rot", "win_score", "win_lse"):
        assert torch.equal(a[key], b[key]), f"{key} not reproducible run to run"
        assert torch.equal(a[key], c[key]), f"{key} differs for strided inputs"


def test_deterministic_head_size_128():
    """The kernel on CTA pairs (work dealt out by a counter, a softmax warpgroup per query block) must give the same
    bits run to run: accumulation order and score sums are fixed by construction."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(5)
    q = to_dev(pc_inputs.f32_to_bf16_bits(rng.standard_normal((2, 900, 8, 128)).astype(np.float32)))
    k = to_dev(pc_inputs.f32_to_bf16_bits(rng.standard_normal((2, 900, 2, 128)).astype(np.float32)))
    v = to_dev(pc_inputs.f32_to_bf16_bits(rng.standard_normal((2, 900, 2, 128)).astype(np.float32)))
    runs = [pc.chunk_prefill_attn(q, k, v, w=64, rope_theta=5e5, want_lse=True) for _ in range(3)]
    torch.cuda.synchronize()
    for key in ("o", "win_score", "win_lse", "lse"):
        assert torch.equal(runs[0][key], runs[1][key]) and torch.equal(runs[0][key], runs[2][key]), key


def test_argument_errors():
    import paper_2502_14317_b200 as pc
    q = torch.zeros((1, 256, 4, 64), dtype=torch.bfloat16, device="cuda")
    k = torch.zeros((1, 256, 2, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(pc.PcError, match="unsupported"):
        pc.chunk_prefill_attn(q, k, k, w=129, rope_theta=1e4)          # window wider than a tile
    with pytest.raises(pc.PcError, match="invalid"):
        pc.chunk_prefill_attn(q, k, k, w=256, rope_theta=1e4)          # window >= L
    q96 = torch.zeros((1, 256, 4, 96), dtype=torch.bfloat16, device="cuda")
    k96 = torch.zeros((1, 256, 2, 96), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(pc.PcError, match="unsupported"):
        pc.chunk_prefill_attn(q96, k96, k96, w=16, rope_theta=1e4)     # head size
    small = torch.empty(16, dtype=torch.uint8, device="cuda")
    lib = pc.load_library()
    import ctypes
    from paper_2502_14317_b200.binding import _make_desc, _ptr
    o = torch.empty_like(q)
    desc = _make_desc(q, k, k, o, 16, 1e4, 0.0)
    ws = torch.empty(64, dtype=torch.uint8, device="cuda")
    S = torch.empty((1, 2, 256), dtype=torch.float32, device="cuda")
    Lw = torch.empty((1, 4, 16), dtype=torch.float32, device="cuda")
    rc = lib.pc_chunk_prefill_attn(ctypes.byref(desc), _ptr(q), _ptr(k), _ptr(k), None, _ptr(o), None, None, _ptr(S), _ptr(Lw),
                                   None, _ptr(ws), ws.numel(), None)
    assert rc == -3                                                     # PC_ERR_WORKSPACE
    rc = lib.pc_chunk_prefill_attn(ctypes.byref(desc), None, _ptr(k), _ptr(k), None, _ptr(o), None, None, _ptr(S), _ptr(Lw),
                                   None, _ptr(ws), ws.numel(), None)
    assert rc == -1                                                     # PC_ERR_INVALID_ARG


@pytest.mark.parametrize("C,L,H,d,theta", [
    (2, 8192, 4, 128, 500000.0),           # positions up to 8191 (angles up to 8191 rad)
    (1, 4096, 8, 128, 10000.0),
    (3, 333, 2, 128, 10000.0),             # ragged last tile
    (2, 1000, 3, 64, 10000.0),             # head size 64
])
def test_rope_position_reuse_equals_fp64_rotation_rounded_once(C, L, H, d, theta):
    """The rotation is fp32 with two exact fallbacks; its bits must be those of the oracle's fp64 rotation.  Mixed
    magnitudes so that many outputs sit near a bf16 rounding boundary; with millions of outputs the second level
    (about 1 in 1300) runs thousands of times."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(5 + L + d)
    x = rng.standard_normal((C, L, H, d)).astype(np.float32) * np.exp2(rng.integers(-6, 7, size=(C, L, H, 1))).astype(np.float32)
    x[0, :, 0, : d // 2] = np.float32(1.0)                    # exact cosines / sines of the table reach the output
    x[0, :, 0, d // 2:] = np.float32(0.0)
    bits = pc_inputs.f32_to_bf16_bits(x)
    got = to_bits(pc.rope_position_reuse(to_dev(bits), rope_theta=theta))
    torch.cuda.synchronize()
    ref = orc.rope_bf16(bits, theta)
    bad = np.argwhere(got != ref)
    assert bad.shape[0] == 0, f"{bad.shape[0]} of {ref.size} rotated values differ from the fp64 rotation, first at {bad[0]}"


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,chunk_len", [
    (1, 700, 32, 8, 2, 64, None), (1, 1500, 100, 8, 2, 128, None), (2, 900, 64, 3, 1, 128, None), (1, 1100, 40, 6, 3, 64, None),
    (3, 1000, 24, 4, 1, 128, [1000, 129, 41]), (2, 1030, 128, 5, 1, 64, [200, 1030]),
])
def test_score_sweeps_as_items_of_their_own(C, L, w, Hq, Hkv, d, chunk_len):
    """Few (chunk, kv-head) groups: units and slices of the score sweep are dealt out one by one and a sweep waits for the group's
    window rows; windows over one and two tiles, short chunks with fewer steps than slices."""
    import paper_2502_14317_b200 as pc
    theta = 10000.0
    rng = np.random.default_rng(L + w)
    q, k, v = (pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, h, d)).astype(np.float32)) for h in (Hq, Hkv, Hkv))
    if chunk_len is None:
        _run_and_compare(q, k, v, w, theta)
        return
    cl = torch.tensor(chunk_len, dtype=torch.int32, device="cuda")
    res = pc.chunk_prefill_attn(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=theta, want_lse=True, chunk_len=cl)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    for c, n in enumerate(chunk_len):
        O, LSE, k_rot = orc.local_attention(q[c:c + 1, :n], k[c:c + 1, :n], v[c:c + 1, :n], theta)
        S, _, _ = orc.window_scores(orc.rope_bf16(q[c:c + 1, :n], theta), k_rot, v[c:c + 1, :n], w, 1.0 / np.sqrt(d))
        check_attention_output(to_f64(res["o"][c:c + 1, :n]), O)
        check_scores(res["win_score"][c:c + 1, :, :n].cpu().numpy(), S, Hq // Hkv, w, n)
        assert not res["o"][c, n:].any() and not res["win_score"][c, :, n:].any()


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,chunk_len", [
    (1, 206, 37, 14, 2, 64, None), (2, 129, 1, 6, 2, 64, None), (1, 256, 128, 8, 1, 64, None), (1, 640, 64, 32, 8, 64, None),
    (2, 300, 50, 6, 2, 128, None), (1, 512, 128, 7, 1, 128, None), (3, 640, 16, 12, 2, 128, [640, 17, 400]), (3, 260, 24, 14, 2, 64, [25, 260, 128]),
])
def test_short_chunks_with_several_units_of_heads(C, L, w, Hq, Hkv, d, chunk_len):
    """Few groups of two to five tiles whose heads are several units: dealt out one by one as well; score sweeps of several passes."""
    test_score_sweeps_as_items_of_their_own(C, L, w, Hq, Hkv, d, chunk_len)


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,chunk_len", [
    (1, 2048, 128, 24, 8, 128, None),                         # 64 sweeps of one step and two passes each
    (4, 1500, 50, 5, 1, 128, [1500, 100, 900, 1300]),         # sweeps of one step or none
    (4, 1536, 50, 8, 8, 64, [1536, 100, 900, 1300]), (1, 2304, 8, 16, 8, 64, None), (1, 900, 16, 62, 62, 64, None),
])
def test_several_short_score_sweeps_on_one_cta(C, L, w, Hq, Hkv, d, chunk_len):
    """Sweeps of a few steps: the CTA that is through its units first takes several of them, whose descriptors its warps reach
    well apart; a warp that could be a whole sweep ahead of another must not signal it through a barrier's parity."""
    test_score_sweeps_as_items_of_their_own(C, L, w, Hq, Hkv, d, chunk_len)


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,gain", [
    (1, 2048, 64, 8, 2, 128, 40.0), (1, 1500, 50, 6, 2, 64, 20.0),
    (20, 130, 128, 16, 8, 64, 20.0), (30, 200, 64, 60, 20, 128, 30.0),      # more window rows than the rotation's tables have room for
])
def test_window_scores_are_as_precise_as_their_log_sum_exp(C, L, w, Hq, Hkv, d, gain):
    """Large logits: what limits a score is the log-sum-exp of its rows, rounded once to fp32 in log2 units.  The 2-norm of the error may
    exceed what that rounding alone gives (evaluated here in fp64) by a quarter, for the fp32 logits; a second rounding, of the natural
    logarithm, would double it."""
    import paper_2502_14317_b200 as pc
    theta, G, log2e = 10000.0, Hq // Hkv, np.log2(np.e)
    rng = np.random.default_rng(3)
    q, k, v = (pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, h, d)).astype(np.float32) * g) for h, g in ((Hq, 1.0), (Hkv, gain), (Hkv, 1.0)))
    res = pc.chunk_prefill_attn(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=theta)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    qr, kr = orc.bf16_to_f64(orc.rope_bf16(q, theta)), orc.bf16_to_f64(orc.rope_bf16(k, theta))
    s = np.einsum("cigd,cjgd->cgij", qr[:, L - w:], np.repeat(kr, G, axis=2)) * (log2e / np.sqrt(d))
    s[:, :, np.arange(L)[None] > (L - w + np.arange(w))[:, None]] = -np.inf
    m = s.max(-1, keepdims=True)
    lse = m + np.log2(np.exp2(s - m).sum(-1, keepdims=True))
    score = lambda l: np.exp2(s - l).sum(2).reshape(C, Hkv, G, L).sum(2)
    S = score(lse)
    one_rounding = np.linalg.norm(score(lse.astype(np.float32)) - S)
    assert np.linalg.norm(res["win_score"].cpu().numpy() - S) <= 1.25 * one_rounding
    assert np.abs(res["win_lse"].cpu().numpy() - lse[..., 0] / log2e).max() <= 2e-3


@pytest.mark.parametrize("C,L,H,d", [(1, 1, 1, 64), (1, 1, 1, 128), (5, 9, 3, 64), (2, 512, 8, 128), (1, 1025, 8, 128), (1, 2049, 8, 64), (3, 700, 37, 128)])
def test_rope_with_and_without_a_table_kernel(C, L, H, d):
    """Up to 2^20 values the warps of the rotation pass compute their own table rows, above that a kernel of its own does: the
    smallest inputs, the last size of the first kind and the first two above it give the oracle's bits."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(L + d)
    bits = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, H, d)).astype(np.float32))
    got = to_bits(pc.rope_position_reuse(to_dev(bits), rope_theta=10000.0))
    torch.cuda.synchronize()
    assert np.array_equal(got, orc.rope_bf16(bits, 10000.0))


@pytest.mark.parametrize("C,L", [(1, 40), (4, 2500)])             # with and without a table kernel
def test_rope_of_infinities_and_nans(C, L):
    """As the fp64 formula gives them: infinities keep their sign, inf - inf and 0 * inf are NaN."""
    import paper_2502_14317_b200 as pc
    H, d, inf = 2, 128, np.inf
    x = np.random.default_rng(L).standard_normal((C, L, H, d)).astype(np.float32)
    x[..., 0, 5], x[..., 0, 6 + d // 2], x[..., 1, 9], x[..., 1, 9 + d // 2] = inf, -inf, inf, -inf
    bits = pc_inputs.f32_to_bf16_bits(x)
    bits[..., 1, 7] = 0x7FC0                                       # NaN
    got = to_f64(pc.rope_position_reuse(to_dev(bits), rope_theta=1e4))
    torch.cuda.synchronize()
    a = np.arange(L)[:, None] * 1e4 ** (-2.0 * np.arange(d // 2) / d)
    c, s = np.cos(a)[None, :, None], np.sin(a)[None, :, None]
    u = orc.bf16_to_f64(bits)
    with np.errstate(invalid="ignore"):
        ref = np.concatenate([u[..., : d // 2] * c - u[..., d // 2:] * s, u[..., d // 2:] * c + u[..., : d // 2] * s], axis=-1)
    odd = ~np.isfinite(ref)
    assert np.array_equal(got[odd], ref[odd], equal_nan=True) and np.isfinite(got[~odd]).all()


@pytest.mark.parametrize("L,w,Hq,Hkv,d,lens", [
    (640, 64, 4, 2, 128, [640, 500, 129, 65, 384]),      # CTA pairs: full, ragged, two tiles, one tile, tile-aligned
    (520, 24, 4, 1, 128, [300, 520, 25, 256]),           # w = 24, the shortest chunk has a single context token
    (640, 64, 3, 3, 128, [640, 333, 130, 65]),           # multi-head: units of four tiles, fewer in the shorter chunks
    (400, 16, 4, 2, 64, [400, 17, 250, 128]),            # head size 64
    (300, 100, 2, 2, 64, [101, 300, 229]),               # head size 64, multi-head, w = 100
])
def test_chunks_of_different_lengths_in_one_call(L, w, Hq, Hkv, d, lens):
    """Sec. 3.1: chunks of AT MOST the trained length.  chunk_len[c] tokens of chunk c count (window included, the
    window directly behind the context); every chunk must equal the oracle run on that chunk alone, and everything
    at or behind its end reads as zero."""
    import paper_2502_14317_b200 as pc
    C = len(lens)
    rng = np.random.default_rng(L + w + Hq + d)
    q = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hq, d)).astype(np.float32))
    k = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hkv, d)).astype(np.float32))
    v = pc_inputs.f32_to_bf16_bits(rng.standard_normal((C, L, Hkv, d)).astype(np.float32))
    k[:, 0] = pc_inputs.f32_to_bf16_bits(pc_inputs.bf16_bits_to_f32(k[:, 0]) * np.float32(4.0))
    theta, G = 10000.0, Hq // Hkv
    cl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    nan = float("nan")
    res = pc.chunk_prefill_attn(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=theta, want_lse=True, chunk_len=cl,
                                out=torch.full((C, L, Hq, d), nan, dtype=torch.bfloat16, device="cuda"),
                                win_score=torch.full((C, Hkv, L), nan, dtype=torch.float32, device="cuda"),
                                lse=torch.full((C, Hq, L), nan, dtype=torch.float32, device="cuda"))
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    got_o, got_S = to_f64(res["o"]), res["win_score"].cpu().numpy()
    got_lse, got_wl = res["lse"].cpu().numpy().astype(np.float64), res["win_lse"].cpu().numpy().astype(np.float64)
    assert np.array_equal(to_bits(res["k_rot"]), orc.rope_bf16(k, theta))
    scale = 1.0 / np.sqrt(d)
    for c, n in enumerate(lens):
        qc, kc, vc = q[c:c + 1, :n], k[c:c + 1, :n], v[c:c + 1, :n]
        O, LSE, k_rot = orc.local_attention(qc, kc, vc, theta)
        S, _, LSE_win = orc.window_scores(orc.rope_bf16(qc, theta), k_rot, vc, w, scale)
        check_attention_output(got_o[c:c + 1, :n], O, f"O of chunk {c} ({n} tokens)")
        assert np.abs(got_lse[c:c + 1, :, :n] - LSE).max() <= 2e-3
        assert np.abs(got_wl[c:c + 1] - LSE_win).max() <= 2e-3
        check_scores(got_S[c:c + 1, :, :n], S, G, w, n)
        assert np.allclose(got_S[c, :, :n].sum(-1), G * w, rtol=1e-4)
        assert np.all(got_o[c, n:] == 0.0) and np.all(got_S[c, :, n:] == 0.0) and np.all(got_lse[c, :, n:] == 0.0)


def test_a_wait_that_runs_out_returns_a_status_and_leaves_the_device_usable(cfg0_inputs):
    """Every device-side wait is bounded.  Here one is made to run out without faulting anything: the producer
    warp of the single-CTA kernel (head size 64) leaves out the data-free "no more work" signal after the last
    work item, when no copy and no tensor-core operation is in flight; the consumer warps wait for it for about a
    millisecond (limit set through the test hook), store the code of that wait in the status word, drain and
    return.  The outputs of that call are complete, and the next call on the same stream is bit-identical to a
    clean run."""
    import paper_2502_14317_b200 as pc
    cfg, inp = cfg0_inputs
    q, k, v = to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"])
    lib = pc.load_library()

    def run():
        r = pc.chunk_prefill_attn(q, k, v, w=cfg.w, rope_theta=cfg.rope_theta, want_lse=True)
        torch.cuda.synchronize()
        return r

    clean = run()
    assert int(clean["status"].item()) == 0
    assert lib.pc_debug_bounded_wait_test(2_000_000, 1) == 0          # waits give up after 2e6 cycles (about 1 ms)
    try:
        hit = run()
    finally:
        assert lib.pc_debug_bounded_wait_test(0, 0) == 0
    code = int(hit["status"].item())
    assert code == 101, f"expected the code of the work-item wait in the status word, got {code}"
    for key in ("o", "win_score", "win_lse", "lse", "k_rot"):
        assert torch.equal(hit[key], clean[key]), key                 # all work was done before the missing signal
    again = run()
    assert int(again["status"].item()) == 0
    for key in ("o", "win_score", "win_lse", "lse", "k_rot"):
        assert torch.equal(again[key], clean[key]), key
