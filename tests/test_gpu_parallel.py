"""GPU parity: pc_parallel_attn (Eq. 9-11) and the chained five-call path against the oracle."""
import numpy as np
import pytest
import torch

import pc_inputs
from oracle import parallelcomp_oracle as orc
from tests.gpu_util import to_dev, to_bits, to_f64, check_attention_output, check_scores

pytestmark = pytest.mark.gpu


def _bits(rng, shape):
    return pc_inputs.f32_to_bf16_bits(rng.standard_normal(shape).astype(np.float32))


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk,q_pos0,theta", [
    (2, 16, 4, 2, 64, 128, 240, 1e4),         # cfg0-like compressed cache
    (1, 64, 8, 2, 128, 1000, 8128, 5e5),      # ragged last cache tile, G*w = 256 rows: a CTA pair, both blocks of each CTA on alternate tiles
    (1, 64, 32, 8, 128, 4096, 8128, 5e5),     # B = 1: keys split, partial results merged
    (3, 8, 2, 2, 64, 300, 4088, 1e4),         # MHA, 8 rows: the kernel for few rows
    (1, 64, 8, 1, 128, 700, 8128, 5e5),       # G*w = 512 rows: two row groups of 256 per kv-head
    (2, 128, 2, 1, 64, 77, 0, 1e4),           # cache shorter than one tile, widest window
    (1, 32, 6, 2, 128, 2049, 100, 1e4),       # G = 3, one key past a tile boundary
    (2, 1, 8, 2, 128, 3000, 8191, 5e5),       # decoding step: one query token over the cache (+ its own key)
    (3, 2, 4, 4, 64, 500, 4094, 1e4),         # two query tokens, MHA
    (1, 4, 32, 8, 128, 16384, 8188, 5e5),     # four query tokens over a 16K cache, Llama-3 heads
    (2, 4, 8, 2, 128, 50, 77, 1e4),           # 16 rows, a cache of one tile and the window's
    (5, 1, 4, 4, 64, 128, 4095, 1e4),         # decoding, MHA, head size 64, cache of exactly one tile
    (1, 16, 8, 2, 128, 5000, 300, 5e5),       # 64 rows per kv-head, 40 cache tiles split over the CTAs, two streams each
    # batches that fill the CTA pairs
    (8, 64, 32, 8, 128, 300, 8128, 5e5),      # 64 groups, ragged last cache tile
    (15, 64, 32, 8, 128, 256, 8128, 5e5),     # 120 groups: two rounds per pair, cache of whole tiles
    (28, 32, 16, 2, 128, 520, 100, 1e4),      # G = 8, w = 32: four heads per block
    (16, 128, 8, 2, 128, 130, 0, 1e4),        # G*w = 512 rows on shared tiles, one head per block, two keys in the last tile
    (60, 8, 32, 1, 128, 129, 5, 1e4),         # window of 8: sixteen heads per block
])
def test_parallel_attn_shapes(B, w, Hq, Hkv, d, Nk, q_pos0, theta):
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + w)
    qw = _bits(rng, (B, w, Hq, d))
    kc, vc = _bits(rng, (B, Hkv, Nk, d)), _bits(rng, (B, Hkv, Nk, d))
    kw, vw = _bits(rng, (B, w, Hkv, d)), _bits(rng, (B, w, Hkv, d))
    kc[:, :, 0] = pc_inputs.f32_to_bf16_bits(pc_inputs.bf16_bits_to_f32(kc[:, :, 0]) * np.float32(4.0))
    res = pc.parallel_attn(to_dev(qw), to_dev(kc), to_dev(vc), to_dev(kw), to_dev(vw), q_pos0=q_pos0,
                           rope_theta=theta, want_lse=True)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    Fg, LSE = orc.parallel_attention(qw, q_pos0, theta, None, kc, vc, kw, vw)
    check_attention_output(to_f64(res["out"]), Fg, "Fg")
    assert np.abs(res["lse"].cpu().numpy() - LSE).max() <= 2e-3


@pytest.mark.parametrize("B", [1, 64])                            # keys split; whole items, blocks of different rows where that fills the GPU
@pytest.mark.parametrize("w,G,Hkv,d,Nk", [
    (64, 3, 2, 128, 1700), (64, 7, 1, 128, 1500), (128, 5, 1, 128, 2300), (16, 9, 2, 128, 2500),   # pairs: 2 + 1 heads; second block 2 + 1; three row groups, the last of one head
    (64, 7, 1, 64, 1600), (64, 3, 2, 64, 2500), (128, 2, 2, 64, 2000), (64, 4, 2, 64, 1900), (128, 4, 1, 64, 1500),
])
def test_row_blocks_that_are_not_full(B, w, G, Hkv, d, Nk):
    """Wide windows whose rows do not fill their blocks, on CTA pairs and single CTAs, with enough key tiles for the rings to go round."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + w + B)
    Hq = G * Hkv
    qw, kw, vw = (_bits(rng, (B, w, h, d)) for h in (Hq, Hkv, Hkv))
    kc, vc = _bits(rng, (B, Hkv, Nk, d)), _bits(rng, (B, Hkv, Nk, d))
    res = pc.parallel_attn(to_dev(qw), to_dev(kc), to_dev(vc), to_dev(kw), to_dev(vw), q_pos0=333, rope_theta=1e4, want_lse=True)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    for b in sorted({0, B // 2, B - 1}):
        Fg, LSE = orc.parallel_attention(qw[b:b + 1], 333, 1e4, None, *(x[b:b + 1] for x in (kc, vc, kw, vw)))
        check_attention_output(to_f64(res["out"][b:b + 1]), Fg, "Fg")
        assert np.abs(res["lse"][b:b + 1].cpu().numpy() - LSE).max() <= 2e-3


WIDE = [                                                                     # both ways to fill the blocks, keys split and whole, rings that go round
    (1, 64, 8, 2, 128, 1700), (40, 64, 8, 2, 128, 900),                      # pairs, alternate tiles
    (6, 128, 16, 4, 128, 1800), (74, 64, 8, 1, 128, 2000),                   # pairs, shared tiles
    (3, 16, 8, 2, 128, 1700), (80, 16, 8, 2, 128, 900),                      # single CTAs, alternate tiles
    (1, 64, 4, 2, 64, 1700), (80, 32, 8, 2, 64, 900),                        # head size 64, alternate tiles
    (12, 64, 16, 4, 64, 2600), (74, 64, 8, 2, 64, 1700),                     # head size 64, shared tiles
]


def _check_some_sequences(res, q, kc, vc, kw, vw, q_pos0, theta):
    assert int(res["status"].item()) == 0
    for b in sorted({0, q.shape[0] // 2, q.shape[0] - 1}):
        Fg, LSE = orc.parallel_attention(q[b:b + 1], q_pos0, theta, None, *(x[b:b + 1] for x in (kc, vc, kw, vw)))
        check_attention_output(to_f64(res["out"][b:b + 1]), Fg, "Fg", sharp=True)
        assert np.abs(res["lse"][b:b + 1].cpu().numpy() - LSE).max() <= 2e-3


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk", WIDE)
def test_many_query_rows_over_growing_keys(B, w, Hq, Hkv, d, Nk):
    """More than 32 query rows: the reference maxima are raised by factors other than zero in most tiles, in streams that hold
    different maxima, and the accumulators rescaled."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + w + d)
    grow = np.linspace(1.0, 40.0, Nk, dtype=np.float32)[None, None, :, None]
    kc = pc_inputs.f32_to_bf16_bits(rng.standard_normal((B, Hkv, Nk, d)).astype(np.float32) * grow)
    q, kw, vw, vc = (_bits(rng, s) for s in ((B, w, Hq, d), (B, w, Hkv, d), (B, w, Hkv, d), (B, Hkv, Nk, d)))
    res = pc.parallel_attn(*(to_dev(x) for x in (q, kc, vc, kw, vw)), q_pos0=500, rope_theta=1e4, want_lse=True)
    torch.cuda.synchronize()
    _check_some_sequences(res, q, kc, vc, kw, vw, 500, 1e4)


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk", WIDE[1::2])          # keys whole: the tile is no stream's first
@pytest.mark.parametrize("at", [522, 612])                        # in the first / in the second half of a key tile
def test_many_query_rows_and_one_logit_far_above_the_others(B, w, Hq, Hkv, d, Nk, at):
    """A single key whose probability, against the maximum of the tiles before, is beyond fp32: it has to be noticed in either half of
    a tile.  (Through the slowest pair, which the rotation leaves as it is.)"""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + at)
    q, kc, vc, kw, vw = (rng.standard_normal(s).astype(np.float32) * g for s, g in (
        ((B, w, Hq, d), 0.3), ((B, Hkv, Nk, d), 0.3), ((B, Hkv, Nk, d), 1.0), ((B, w, Hkv, d), 0.3), ((B, w, Hkv, d), 1.0)))
    q[..., d // 2 - 1], kc[..., d // 2 - 1], kw[..., d // 2 - 1] = 8.0, 0.0, 0.0
    kc[:, :, at, d // 2 - 1] = 150.0 * np.sqrt(d) / (8.0 * np.log2(np.e))
    q, kc, vc, kw, vw = (pc_inputs.f32_to_bf16_bits(x) for x in (q, kc, vc, kw, vw))
    res = pc.parallel_attn(*(to_dev(x) for x in (q, kc, vc, kw, vw)), q_pos0=500, rope_theta=1e9, want_lse=True)
    torch.cuda.synchronize()
    _check_some_sequences(res, q, kc, vc, kw, vw, 500, 1e9)


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk,code", [
    (1, 64, 8, 2, 128, 1700, 201), (74, 64, 8, 1, 128, 2000, 201), (3, 16, 8, 2, 128, 1700, 101), (80, 32, 8, 2, 64, 900, 101),
])
def test_a_wait_that_runs_out_in_the_wide_kernel(B, w, Hq, Hkv, d, Nk, code):
    """CTA pairs and single CTAs: the producers leave out the data-free "no more work" signal after the last work item, when no copy
    and no product is in flight.  The waits for it give up after about a millisecond, the status word holds their code, the producer
    drains its copies, both CTAs of a pair return, the outputs are complete and the next call gives the bits of a clean run."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk)
    t = [to_dev(_bits(rng, s)) for s in ((B, w, Hq, d), (B, Hkv, Nk, d), (B, Hkv, Nk, d), (B, w, Hkv, d), (B, w, Hkv, d))]
    lib = pc.load_library()

    def run():
        r = pc.parallel_attn(*t, q_pos0=300, rope_theta=1e4, want_lse=True)
        torch.cuda.synchronize()
        return r

    clean = run()
    assert int(clean["status"].item()) == 0
    assert lib.pc_debug_bounded_wait_test(2_000_000, 1) == 0          # waits give up after 2e6 cycles (about 1 ms)
    try:
        hit = run()
    finally:
        assert lib.pc_debug_bounded_wait_test(0, 0) == 0
    assert int(hit["status"].item()) == code
    again = run()
    assert int(again["status"].item()) == 0
    for r in (hit, again):
        assert torch.equal(r["out"], clean["out"]) and torch.equal(r["lse"], clean["lse"])


@pytest.mark.parametrize("Hq,Hkv,d", [(8, 2, 128), (4, 2, 128), (4, 2, 64)])
@pytest.mark.parametrize("shift", [16, 32, 48])
def test_workspace_at_any_multiple_of_16_bytes(Hq, Hkv, d, shift):
    """Keys split, so that partial results go through the workspace: its address needs 16 bytes of alignment, no more (pairs,
    single CTAs, head size 64)."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(shift + d)
    B, w, Nk = 1, 64, 2500
    t = [to_dev(_bits(rng, s)) for s in ((B, w, Hq, d), (B, Hkv, Nk, d), (B, Hkv, Nk, d), (B, w, Hkv, d), (B, w, Hkv, d))]
    need = pc.parallel_attn_workspace_bytes(B, w, Hq, Hkv, d, Nk)
    assert need > B * Hq * w * d * 4                                          # room for partial results: the keys are split
    room = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    at = -room.data_ptr() % 64 + shift
    want = pc.parallel_attn(*t, q_pos0=100, rope_theta=1e4, want_lse=True)
    got = pc.parallel_attn(*t, q_pos0=100, rope_theta=1e4, want_lse=True, workspace=room[at:at + need])
    torch.cuda.synchronize()
    assert int(got["status"].item()) == 0
    assert torch.equal(got["out"], want["out"]) and torch.equal(got["lse"], want["lse"])


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk,grow", [
    (1, 1, 1, 1, 128, 1, 0), (1, 1, 3, 1, 64, 127, 0), (2, 1, 2, 2, 128, 129, 0),    # one and two tiles: fewer than key splits
    (1, 2, 8, 1, 128, 2050, 0), (1, 1, 17, 1, 128, 700, 0), (2, 4, 8, 1, 64, 640, 0),   # 16, 17 and 32 rows per kv-head
    (1, 1, 33, 1, 64, 513, 0), (3, 8, 4, 1, 128, 1500, 0), (1, 32, 2, 2, 64, 900, 0),   # 33 rows (the row-major kernel), 32 rows
    (150, 1, 8, 2, 128, 140, 0), (40, 16, 16, 8, 64, 260, 0),                     # more items than CTAs fit
    (1, 4, 8, 2, 128, 3000, 1), (30, 8, 4, 1, 64, 600, 1),                            # growing keys: the reference maxima are raised in most tiles
])
def test_few_query_rows(B, w, Hq, Hkv, d, Nk, grow):
    """Up to 32 query rows per (sequence, kv-head): the transposed kernel, its row paddings, key splits and merge."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + 3 * w + Hq)
    qw = _bits(rng, (B, w, Hq, d))
    kc, vc = rng.standard_normal((B, Hkv, Nk, d)).astype(np.float32), _bits(rng, (B, Hkv, Nk, d))
    if grow:
        kc *= np.linspace(1.0, 40.0, Nk, dtype=np.float32)[None, None, :, None]
    kc = pc_inputs.f32_to_bf16_bits(kc)
    kw, vw = _bits(rng, (B, w, Hkv, d)), _bits(rng, (B, w, Hkv, d))
    res = pc.parallel_attn(to_dev(qw), to_dev(kc), to_dev(vc), to_dev(kw), to_dev(vw), q_pos0=500, rope_theta=1e4,
                           want_lse=True)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    Fg, LSE = orc.parallel_attention(qw, 500, 1e4, None, kc, vc, kw, vw)
    check_attention_output(to_f64(res["out"]), Fg, "Fg", sharp=bool(grow))
    assert np.abs(res["lse"].cpu().numpy() - LSE).max() <= 2e-3


@pytest.mark.parametrize("B,w,Hq,Hkv,d,Nk", [
    (1, 1, 4, 1, 128, 20000), (1, 1, 10, 10, 128, 5000), (3, 1, 12, 6, 128, 3000),   # deep ring, 16, 9 or 10 and fewer CTAs; stages reused
    (1, 16, 4, 2, 128, 300), (80, 8, 8, 2, 128, 300),                            # 16 tokens: angles found in the loop; three stages, 32 rows
    (75, 1, 4, 2, 128, 1000), (2, 32, 1, 1, 64, 2500),
])
def test_few_query_rows_deep_and_shallow_rings(B, w, Hq, Hkv, d, Nk):
    """The two builds of the transposed kernel (few items: six stages; many: three), odd cluster sizes and long token loops."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + B)
    qw, kw, vw = (_bits(rng, (B, w, h, d)) for h in (Hq, Hkv, Hkv))
    kc, vc = _bits(rng, (B, Hkv, Nk, d)), _bits(rng, (B, Hkv, Nk, d))
    res = pc.parallel_attn(to_dev(qw), to_dev(kc), to_dev(vc), to_dev(kw), to_dev(vw), q_pos0=777, rope_theta=1e4, want_lse=True)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    for b in sorted({0, B // 2, B - 1}):
        Fg, LSE = orc.parallel_attention(qw[b:b + 1], 777, 1e4, None, *(x[b:b + 1] for x in (kc, vc, kw, vw)))
        check_attention_output(to_f64(res["out"][b:b + 1]), Fg, "Fg")
        assert np.abs(res["lse"][b:b + 1].cpu().numpy() - LSE).max() <= 2e-3


@pytest.mark.parametrize("w,Hq,Hkv,d", [(1, 8, 2, 128), (8, 4, 1, 64), (4, 8, 1, 128), (64, 4, 2, 128)])      # 4, 32, 32 and 128 rows
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_queries_that_are_no_numbers(w, Hq, Hkv, d, bad):
    """A NaN (or an infinity: a logit of inf - inf) in one query makes that row NaN and no other."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(w)
    t = [to_dev(_bits(rng, s)) for s in ((1, w, Hq, d), (1, Hkv, 900, d), (1, Hkv, 900, d), (1, w, Hkv, d), (1, w, Hkv, d))]
    want = pc.parallel_attn(*t, q_pos0=70, rope_theta=1e4, want_lse=True)
    t[0] = t[0].clone()
    t[0][0, w - 1, Hq - 1, [3, 3 + d // 2]] = bad
    got = pc.parallel_attn(*t, q_pos0=70, rope_theta=1e4, want_lse=True)
    torch.cuda.synchronize()
    assert int(got["status"].item()) == 0
    assert got["out"][0, w - 1, Hq - 1].isnan().all() and got["lse"][0, Hq - 1, w - 1].isnan()
    got["out"][0, w - 1, Hq - 1] = want["out"][0, w - 1, Hq - 1]
    got["lse"][0, Hq - 1, w - 1] = want["lse"][0, Hq - 1, w - 1]
    # two bf16 roundings of P and of the result: the row's neighbours may be taken against another reference maximum
    assert (got["out"].float() - want["out"].float()).abs().max() <= 1e-2 and (got["lse"] - want["lse"]).abs().max() <= 2e-3


@pytest.mark.parametrize("G,d,Nk", [(8, 64, 50), (8, 64, 128), (4, 128, 3000), (17, 128, 700), (40, 64, 1500), (130, 128, 700)])
@pytest.mark.parametrize("where", ["window", "first tile", "every key"])
def test_logits_of_minus_infinity(G, d, Nk, where):
    """Keys whose logits are -inf for every query count nothing, also where they are all that a key split or a row's first tile holds;
    with no other key a row is NaN, as a softmax over nothing is.  (One token at position 0: its queries are not turned.)"""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(Nk + G)
    q, kc, vc, kw, vw = (to_dev(_bits(rng, s)) for s in ((1, 1, G, d), (1, 1, Nk, d), (1, 1, Nk, d), (1, 1, 1, d), (1, 1, 1, d)))
    q[..., 0], kc[..., 0], kw[..., 0] = 1.0, 0.0, 0.0
    if where != "first tile":
        kw[..., 0] = float("-inf")
    if where != "window":
        kc[:, :, :128 if where == "first tile" else Nk, 0] = float("-inf")
    res = pc.parallel_attn(q, kc, vc, kw, vw, q_pos0=0, rope_theta=1e4)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    s = torch.cat([kc, kw.transpose(1, 2)], dim=2)[0, 0].double() @ q[0, 0].double().T / d ** 0.5
    ref = torch.softmax(s, dim=0).T @ torch.cat([vc, vw.transpose(1, 2)], dim=2)[0, 0].double()
    if where == "every key":
        assert res["out"].isnan().all()
    else:
        check_attention_output(to_f64(res["out"])[0, 0], ref.cpu().numpy(), "Fg", sharp=True)


@pytest.mark.parametrize("w,Hq,Hkv,d,Nk,one_launch", [
    (8, 4, 1, 64, 511 * 128, True), (8, 4, 1, 64, 511 * 128 + 1, False), (1, 17, 1, 128, 1023 * 128 + 5, False),
    (1, 2, 1, 128, 1023 * 128, True), (1, 2, 1, 128, 1024 * 128, False), (2, 1, 1, 64, 1023 * 128 + 70, False),
])
def test_few_query_rows_over_long_caches(w, Hq, Hkv, d, Nk, one_launch):
    """At both sides of the cache lengths from which the wide kernel, which splits keys further, takes few rows too."""
    import paper_2502_14317_b200 as pc
    g = torch.Generator(device="cuda").manual_seed(Nk)
    t = [torch.randn(s, generator=g, device="cuda").bfloat16() for s in ((1, w, Hq, d), (1, Hkv, Nk, d), (1, Hkv, Nk, d), (1, w, Hkv, d), (1, w, Hkv, d))]
    n = pc.launch_count()
    res = pc.parallel_attn(*t, q_pos0=500, rope_theta=1e4, want_lse=True)
    assert (pc.launch_count() - n == 1) == one_launch
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    q, kc, vc, kw, vw = (to_bits(x) for x in t)
    Fg, LSE = orc.parallel_attention(q, 500, 1e4, None, kc, vc, kw, vw)
    check_attention_output(to_f64(res["out"]), Fg, "Fg")
    assert np.abs(res["lse"].cpu().numpy() - LSE).max() <= 2e-3


@pytest.mark.parametrize("B,Hq,Hkv,d,Nk0,cap,steps", [
    (2, 8, 2, 128, 250, 260, (1, 1, 4, 1)),   # crosses a tile boundary of the cache (256) while generating
    (3, 4, 4, 64, 40, 48, (1, 2, 1)),         # MHA, head size 64
])
def test_generation_steps_append_to_the_cache(B, Hq, Hkv, d, Nk0, cap, steps):
    """pc_parallel_attn_append in a loop: every step attends over the entries valid so far (oracle on the same prefix)
    and leaves its new keys / values behind them; entries further back stay as they were."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(cap)
    kc, vc = _bits(rng, (B, Hkv, cap, d)), _bits(rng, (B, Hkv, cap, d))    # entries >= Nk0: junk that must never be read
    k_dev, v_dev = to_dev(kc), to_dev(vc)
    n, pos, theta = Nk0, 1000, 1e4
    for w in steps:
        qw = _bits(rng, (B, w, Hq, d))
        kw, vw = _bits(rng, (B, w, Hkv, d)), _bits(rng, (B, w, Hkv, d))
        res = pc.parallel_attn_append(to_dev(qw), k_dev, v_dev, n, to_dev(kw), to_dev(vw), q_pos0=pos, rope_theta=theta,
                                      want_lse=True)
        torch.cuda.synchronize()
        assert int(res["status"].item()) == 0
        Fg, LSE = orc.parallel_attention(qw, pos, theta, None, np.ascontiguousarray(kc[:, :, :n]),
                                         np.ascontiguousarray(vc[:, :, :n]), kw, vw)
        check_attention_output(to_f64(res["out"]), Fg, f"Fg over {n} entries, {w} new")
        assert np.abs(res["lse"].cpu().numpy() - LSE).max() <= 2e-3
        kc[:, :, n:n + w] = kw.transpose(0, 2, 1, 3)
        vc[:, :, n:n + w] = vw.transpose(0, 2, 1, 3)
        assert np.array_equal(to_bits(k_dev), kc) and np.array_equal(to_bits(v_dev), vc), "cache after the append"
        n += w
        pos += w
    # a step that does not fit is refused before anything is launched
    lib = pc.load_library()
    assert lib.pc_parallel_attn_append(B, 1, Hq, Hkv, d, cap, cap, None, 0, 1e4, 0.0, None, None, None, None, None, None,
                                       None, None, 0, None) == -1


def test_cfg4_slice():
    """The batch-of-compressed-caches workload at a size the oracle finishes in seconds: 2 of the 64
    sequences, full Nk = 16384 (128 key tiles), same generator."""
    import paper_2502_14317_b200 as pc
    cfg = pc_inputs.get_config("cfg4")
    inp = pc_inputs.make_parallel_attn_inputs(cfg, B=2)
    res = pc.parallel_attn(to_dev(inp["q_win"]), to_dev(inp["k_cache"]), to_dev(inp["v_cache"]), to_dev(inp["k_win"]),
                           to_dev(inp["v_win"]), q_pos0=cfg.q_pos0, rope_theta=cfg.rope_theta, want_lse=True)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    Fg, LSE = orc.parallel_attention(inp["q_win"], cfg.q_pos0, cfg.rope_theta, None, inp["k_cache"], inp["v_cache"],
                                     inp["k_win"], inp["v_win"])
    check_attention_output(to_f64(res["out"]), Fg, "Fg")
    assert np.abs(res["lse"].cpu().numpy() - LSE).max() <= 2e-3


def test_cfg0_whole_path(cfg0_inputs, cfg0_oracle):
    """All five calls chained on one stream; every stage compared with the oracle."""
    import paper_2502_14317_b200 as pc
    cfg, inp = cfg0_inputs
    ref = cfg0_oracle
    q, k, v = to_dev(inp["q"]), to_dev(inp["k"]), to_dev(inp["v"])
    res = pc.hot_path(q, k, v, w=cfg.w, rope_theta=cfg.rope_theta, m=cfg.m, k_keep=cfg.k)
    torch.cuda.synchronize()
    assert int(res["status"].item()) == 0
    check_attention_output(to_f64(res["o"]), ref["O"])
    S_gpu = res["win_score"].cpu().numpy()
    check_scores(S_gpu, ref["S"], cfg.G, cfg.w, cfg.L)
    assert np.array_equal(to_bits(res["k_rot"]), ref["k_rot"])
    score_gpu = res["chunk_score"].cpu().numpy()
    assert np.allclose(score_gpu, ref["chunk_score"], atol=2e-3)
    # ranking and gather: bit-exact given the tensors the GPU ranked
    kept = orc.select_chunks(score_gpu, cfg.m)
    assert np.array_equal(res["kept"].cpu().numpy(), kept)
    idx = orc.select_tokens(S_gpu, kept, cfg.ctx, cfg.k)
    assert np.array_equal(res["idx"].cpu().numpy(), idx)
    Kc, Vc, pos = orc.gather_kv(ref["k_rot"], inp["v"], kept, idx)
    assert np.array_equal(to_bits(res["kc"]), Kc) and np.array_equal(to_bits(res["vc"]), Vc)
    assert np.array_equal(res["pos"].cpu().numpy(), pos)
    # global attention over the cache the GPU built
    L, w = cfg.L, cfg.w
    Fg, _ = orc.parallel_attention(inp["q"][0:1, L - w:], L - w, cfg.rope_theta, None, Kc[None], Vc[None],
                                   ref["k_rot"][0:1, L - w:], inp["v"][0:1, L - w:])
    check_attention_output(to_f64(res["fg"])[0], Fg[0], "Fg")
    # end to end the oracle made the same eviction decisions on this input
    assert np.array_equal(kept, ref["kept"])
    assert np.array_equal(idx, ref["idx"])
    check_attention_output(to_f64(res["fg"])[0], ref["Fg"], "Fg end-to-end")
    # planted keys survive (generator property)
    r = kept.tolist().index(2)
    for hk in range(cfg.Hkv):
        assert set(inp["planted_pos"][0, hk].tolist()) <= set(idx[r, hk].tolist())


def test_single_chunk_keep_all_equals_local_attention():
    """C = 1, keep everything: the global output equals the window rows of the local attention."""
    import paper_2502_14317_b200 as pc
    rng = np.random.default_rng(11)
    C, L, Hq, Hkv, d, w = 1, 400, 4, 2, 64, 16
    q, k, v = _bits(rng, (C, L, Hq, d)), _bits(rng, (C, L, Hkv, d)), _bits(rng, (C, L, Hkv, d))
    res = pc.hot_path(to_dev(q), to_dev(k), to_dev(v), w=w, rope_theta=1e4, m=1, k_keep=L - w)
    torch.cuda.synchronize()
    o_win = to_f64(res["o"])[0, L - w:]
    fg = to_f64(res["fg"])[0]
    assert np.abs(o_win - fg).max() <= 1e-2          # two bf16 roundings of the same quantity
    O, _, _ = orc.local_attention(q, k, v, 1e4)
    check_attention_output(fg, O[0, L - w:], "Fg vs full causal attention")


@pytest.mark.parametrize("C,L,w,Hq,Hkv,d,m,k,given,strided", [
    (4, 256, 16, 4, 2, 64, 2, 64, False, False), (3, 200, 32, 6, 3, 128, 2, 100, True, False),
    (1, 129, 8, 2, 1, 128, 1, 121, False, True), (5, 300, 64, 4, 4, 64, 3, 77, True, True),
])
def test_hot_path_equals_its_stages(C, L, w, Hq, Hkv, d, m, k, given, strided):
    """The whole path as one call gives the bits of the five calls made one by one, with fresh outputs (the status word
    starts from whatever was in memory) and with kept ones, and names the stage that refuses its arguments."""
    import paper_2502_14317_b200 as pc
    g = torch.Generator(device="cuda").manual_seed(C + L)
    q, kk, v = (torch.randn((C, L, h, d), generator=g, device="cuda").bfloat16() for h in (Hq, Hkv, Hkv))
    if strided:
        q = torch.cat([q, q], dim=2)[:, :, :Hq]
    score = torch.randn(C, generator=g, device="cuda") if given else None
    pre = pc.chunk_prefill_attn(q, kk, v, w=w, rope_theta=1e4)
    if given:
        want_score, kept = score, pc.select_chunks(score, m, True)
    else:
        want_score, kept = pc.score_select_chunks(pre["win_lse"], m, True)
    idx = pc.select_tokens(pre["win_score"], kept, L - w, k)
    kc, vc, pos = pc.gather_kv(pre["k_rot"], v, kept, idx)
    fg = pc.parallel_attn(q[0:1, L - w:].contiguous(), kc[None], vc[None], pre["k_rot"][0:1, L - w:].contiguous(),
                          v[0:1, L - w:].contiguous(), q_pos0=L - w, rope_theta=1e4)["out"]
    want = {"o": pre["o"], "k_rot": pre["k_rot"], "win_score": pre["win_score"], "win_lse": pre["win_lse"], "chunk_score": want_score,
            "kept": kept, "idx": idx, "kc": kc, "vc": vc, "pos": pos, "fg": fg}
    junk = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (1, 2, 64)]        # freed: fresh memory is not zero
    del junk
    buffers = {}
    for b in (None, buffers, buffers):
        got = pc.hot_path(q, kk, v, w=w, rope_theta=1e4, m=m, k_keep=k, chunk_score=score, buffers=b)
        torch.cuda.synchronize()
        assert int(got["status"].item()) == 0
        for key, t in want.items():
            assert torch.equal(got[key], t), key
    for bad, stage in ((dict(w=L), "pc_chunk_prefill_attn"), (dict(k_keep=0), "pc_select_tokens"),
                       (dict(m=C + 1), "pc_select_chunks" if given else "pc_score_select_chunks")):
        with pytest.raises(pc.PcError, match=stage):
            pc.hot_path(q, kk, v, **{**dict(w=w, rope_theta=1e4, m=m, k_keep=k, chunk_score=score), **bad})


def test_hot_path_takes_scores_as_contiguous_float32_of_its_chunks_only():
    import paper_2502_14317_b200 as pc
    q, k = (torch.zeros((4, 200, h, 64), dtype=torch.bfloat16, device="cuda") for h in (4, 2))
    score = torch.zeros(8, device="cuda")
    for bad, why in ((score[:4].double(), "float32"), (score[::2], "contiguous"), (score[:1].expand(4), "contiguous"), (score, "invalid")):
        with pytest.raises(pc.PcError, match=why):
            pc.hot_path(q, k, k, w=16, rope_theta=1e4, m=2, k_keep=50, chunk_score=bad)
    torch.cuda.synchronize()


@pytest.mark.parametrize("C,Hkv,odd", [(2, 1, "k"), (2, 1, "v"), (2, 1, "kv"), (1, 2, "k"), (1, 2, "v"), (1, 2, "kv")])
def test_strides_of_dimensions_of_one_entry_do_not_matter(C, Hkv, odd):
    """One kv-head seen through a transposed view, or one chunk cut out of longer ones: contiguous all the same."""
    import paper_2502_14317_b200 as pc
    L, w, Hq, d, m, k_keep = 300, 16, 2, 64, 1, 50
    g = torch.Generator(device="cuda").manual_seed(C)
    q, k, v = (torch.randn((C, L, h, d), generator=g, device="cuda").bfloat16() for h in (Hq, Hkv, Hkv))

    def same_values_other_strides(t):
        if Hkv == 1:
            t = t[:, :, 0].clone()[:, None].transpose(1, 2)
        else:
            t = torch.cat([t, t], dim=1)[:, :L]
        assert t.is_contiguous() and t.stride() != q.new_empty(t.shape).stride()
        return t

    k2, v2 = (same_values_other_strides(t) if n in odd else t for n, t in (("k", k), ("v", v)))
    args = dict(w=w, rope_theta=1e4, m=m, k_keep=k_keep)
    want, got = pc.hot_path(q, k, v, **args), pc.hot_path(q, k2, v2, **args)
    by_batch = pc.hot_path_streaming(q, k2, v2, batch=1, **args)
    kc, vc, pos = pc.gather_kv(k2, v2, want["kept"], want["idx"])
    want_kc, want_vc, _ = pc.gather_kv(k, v, want["kept"], want["idx"])
    for key in ("o", "k_rot", "idx", "kc", "vc", "fg"):
        assert torch.equal(got[key], want[key]) and got[key].stride() == want[key].stride(), key
    assert torch.equal(by_batch["kc"], want["kc"]) and torch.equal(by_batch["vc"], want["vc"])
    assert torch.equal(kc, want_kc) and torch.equal(vc, want_vc)
    with pytest.raises(pc.PcError, match="strides"):
        pc.hot_path(q, k, torch.cat([v, v], dim=3)[..., :d], **args)


def test_hot_path_from_host_matches_device_path(cfg0_inputs):
    """Uploading the chunks in groups on a copy stream must give exactly what the all-on-device path gives."""
    import paper_2502_14317_b200 as pc
    cfg, inp = cfg0_inputs
    pin = lambda bits: torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).pin_memory()
    hq, hk, hv = pin(inp["q"]), pin(inp["k"]), pin(inp["v"])
    ref = pc.hot_path(hq.cuda(), hk.cuda(), hv.cuda(), w=cfg.w, rope_theta=cfg.rope_theta, m=cfg.m, k_keep=cfg.k)
    buffers = {}
    for _ in range(2):                                            # second call reuses buffers, streams and events
        got = pc.hot_path_from_host(hq, hk, hv, w=cfg.w, rope_theta=cfg.rope_theta, m=cfg.m, k_keep=cfg.k, n_groups=3,
                                    buffers=buffers)
        torch.cuda.synchronize()
        assert int(got["status"].item()) == 0
        for key in ("o", "k_rot", "win_score", "win_lse", "kept", "idx", "kc", "vc", "fg"):
            assert torch.equal(got[key], ref[key]), key


@pytest.mark.parametrize("path", ["at once", "streamed", "from host"])
def test_buffers_of_a_call_of_other_sizes(path):
    """One dict for prompts of other sizes (larger, smaller, the same elements in another shape), head counts, head sizes, windows and kept
    tokens: the same results as with buffers of the call's own, to the bit."""
    import paper_2502_14317_b200 as pc
    run = {"at once": pc.hot_path, "streamed": lambda *t, **kw: pc.hot_path_streaming(*t, batch=2, **kw),
           "from host": lambda *t, **kw: pc.hot_path_from_host(*(x.cpu().pin_memory() for x in t), n_groups=3, **kw)}[path]
    g = torch.Generator(device="cuda").manual_seed(5)
    b = {}
    for C, L, Hq, Hkv, d, w, m, kk in [(4, 300, 4, 2, 64, 16, 2, 64), (4, 300, 8, 4, 128, 32, 3, 128), (4, 300, 2, 1, 128, 64, 1, 100),
                                       (6, 200, 4, 2, 64, 8, 4, 32), (2, 700, 8, 2, 64, 64, 2, 300)]:
        q, k, v = (torch.randn((C, L, H, d), generator=g, device="cuda").bfloat16() for H in (Hq, Hkv, Hkv))
        args = dict(w=w, rope_theta=1e4, m=m, k_keep=kk)
        want, got = run(q, k, v, **args), run(q, k, v, buffers=b, **args)
        torch.cuda.synchronize()
        assert int(got["status"].item()) == 0
        for n in ("o", "k_rot", "win_score", "win_lse", "chunk_score", "kept", "idx", "kc", "vc", "pos", "fg"):
            if n in want:
                assert got[n].shape == want[n].shape and torch.equal(got[n], want[n]), n


@pytest.mark.parametrize("path", ["at once", "streamed", "from host"])
def test_buffers_dropped_on_another_stream(path):
    """Buffers of one stream, used and then replaced on another that has not come there yet: their memory is not given out meanwhile."""
    import paper_2502_14317_b200 as pc
    run = {"at once": pc.hot_path, "streamed": lambda *t, **kw: pc.hot_path_streaming(*t, batch=2, **kw), "from host": pc.hot_path_from_host}[path]
    g = torch.Generator(device="cuda").manual_seed(6)

    def inputs(L, Hq, Hkv):
        t = [torch.randn((4, L, H, 64), generator=g, device="cuda").bfloat16() for H in (Hq, Hkv, Hkv)]
        return [x.cpu().pin_memory() for x in t] if path == "from host" else t
    # (the streamed path keeps a set of buffers for each batch shape: other head counts there)
    small, large = inputs(500, 4, 2), inputs(500, 8, 4) if path == "streamed" else inputs(900, 4, 2)
    small_args, args, b = dict(w=16, rope_theta=1e4, m=2, k_keep=100), dict(w=16, rope_theta=1e4, m=3, k_keep=200), {}

    def tensors(x):
        return [t for v in x.values() for t in (tensors(v) if isinstance(v, dict) else [v] if torch.is_tensor(v) else [])]
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):                                  # kernels are loaded, the side stream has memory to give
        want = {n: t.clone() for n, t in run(*large, **args).items()}
    run(*small, buffers=b, **small_args)
    old = {t.untyped_storage().data_ptr(): t.untyped_storage().nbytes() for t in tensors(b)}
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(1 << 30)                                 # half a second
        out = run(*large, buffers=b, **args)
        done = torch.cuda.Event()
        done.record()
    dropped = set(old) - {t.untyped_storage().data_ptr() for t in tensors(b)}
    new = [torch.empty(old[p], dtype=torch.uint8, device="cuda") for p in dropped]
    assert not done.query() and len(dropped) >= 8
    assert not dropped & {t.data_ptr() for t in new}
    torch.cuda.synchronize()
    assert int(out["status"].item()) == 0
    for n in ("kept", "kc", "vc", "pos", "fg"):
        assert torch.equal(out[n], want[n]), n
