"""Kernels of the draft path at the sizes where their tilings have edges, against the oracle.

The checks and tolerances are those of tests/harness.py (fp32 storage: 1e-5 element by element with the
floor at the tensor's rms; bf16 storage: 2e-2, see there)."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import synth
from tests.harness import GpuSide, check_kv, check_rows, check_tokens, f64, oracle_for

pytestmark = pytest.mark.gpu


def _shape(**kw):
    base = dict(d=256, n_draft_layers=2, n_target_layers=2, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=256,
                vocab=700, block=8)
    base.update(kw)
    return synth.Shape(**base)


def _step_matches_oracle(w, flags=0, **variant):
    """A fill of w.ctx_lens in one call, every cached key and value, and one drafted block."""
    W = dict(synth.weights(w))
    if variant:
        W.update(synth.variant_weights(w))
    g = GpuSide(w, flags=flags, weights=W)
    o = oracle_for(w, W, **variant)
    got = f64(g.fuse(w.ctx_lens))
    for b, n in enumerate(w.ctx_lens):
        F = o.fuse_context(b, synth.hidden_states(w, b, 0, n))
        for i in range(w.shape.n_draft_layers):
            slot = 0 if variant.get("dflash_fc") else i
            check_rows(w, got[slot, b, :n], F[slot], f"F seq {b} layer {i}")
            k, v = g.lib.read_kv(i, b, 0, n)
            check_kv(w, o, f64(k), f64(v), got[slot, b, :n], np.arange(n), i, f"seq {b} layer {i}")
    x_t = synth.initial_tokens(w)
    tok, logits, hidden = g.draft(x_t)
    for b in range(w.batch):
        ot, ol, oh = o.draft_block(b, int(x_t[b]))
        for i in range(oh.shape[0]):
            check_rows(w, hidden[i, b], oh[i], f"seq {b} hidden after layer {i - 1}")
        check_rows(w, logits[b], ol, f"seq {b} logits")
        check_tokens(w, o, tok[b], logits[b], hidden[-1, b], ot, ol, f"seq {b}")
    assert g.lib.device_error() == 0


# fp32: 8- and 16-token CTAs (7, 8, 9, 16, 17 and 34 rows), contractions that are no multiple of 128,
# feature counts that are no multiple of 32 (the vocabulary), one and several key splits, a tile of
# keys that the context and the block share, more than one 16-row query tile, both head sizes
F32_CASES = [
    synth.Workload("f32_b1", _shape(dtype="f32", d=192, ffn=320, vocab=1003, block=8), (56,), 0.8, 31, False),
    synth.Workload("f32_block9", _shape(dtype="f32", d=320, block=9, vocab=129), (184, 1), 0.8, 32, False),
    synth.Workload("f32_block17_hd128", _shape(dtype="f32", head_dim=128, n_q_heads=8, block=17, vocab=97), (700, 65), 0.8, 33, False),
    synth.Workload("f32_block1", _shape(dtype="f32", block=1, n_q_heads=2), (191,), 0.8, 34, False),
]


@pytest.mark.parametrize("w", F32_CASES, ids=lambda w: w.name)
def test_fp32_kernels_match_oracle(w):
    _step_matches_oracle(w)


def test_simt_gemm_on_bf16_matches_oracle():
    """The CUDA-core GEMM on bf16 weights (a cross-check of the tensor-core GEMM)."""
    from paper_2606_02091_gb300 import FLAG_SIMT_GEMM
    _step_matches_oracle(synth.Workload("simt_bf16", _shape(d=320, ffn=192, vocab=333, block=9), (40, 3), 0.8, 35), FLAG_SIMT_GEMM)


# the CUDA-core GEMM's 128 x 64 tiles (more than 1520 CTAs of the other form): 2048 block rows through every
# projection, features that end inside a tile (448, 461 and 2 x 320 of 128), a fill of 4602 rows
TILED = _shape(dtype="f32", d=448, n_draft_layers=1, ffn=320, vocab=461, block=32)
TILED_BLOCK = synth.Workload("tiled_block", TILED, tuple(1 + b % 5 for b in range(64)), 0.8, 38, False)
TILED_FILL = synth.Workload("tiled_fill", _shape(dtype="f32", n_draft_layers=2, head_dim=128, n_target_layers=3), (2301, 3), 0.8, 39, False)


def test_fp32_tiles_of_many_block_rows_match_oracle():
    _step_matches_oracle(TILED_BLOCK)


def test_simt_tiles_of_many_block_rows_on_bf16_match_oracle():
    from paper_2606_02091_gb300 import FLAG_SIMT_GEMM
    w = TILED_BLOCK.with_(shape=dataclasses.replace(TILED, dtype="bf16"))
    _step_matches_oracle(w, FLAG_SIMT_GEMM)


# the tiles of a short K: 16 tokens in the LM head (240 rows x 1003; 15 x 58401 at K 192) and in Q/K/V (256 x 1024, rotary), more
# in gate/up (256 x 640) and, with 16 query heads and 2049 features, in Q/K/V and the LM head
SHORT_K = [
    synth.Workload("short_64", _shape(dtype="f32", d=64, n_draft_layers=1, n_q_heads=8, n_kv_heads=4, ffn=640, vocab=1003,
                                      block=16), tuple(1 + b % 5 for b in range(16)), 0.8, 60, False),
    synth.Workload("short_64_wide", _shape(dtype="f32", d=64, n_draft_layers=1, n_q_heads=16, n_kv_heads=8, ffn=64, vocab=2049,
                                           block=16), tuple(1 + b % 5 for b in range(16)), 0.8, 61, False),
    synth.Workload("short_128", _shape(dtype="f32", d=128, n_draft_layers=1, n_q_heads=16, n_kv_heads=8, ffn=64, vocab=2049,
                                       block=16), tuple(1 + b % 5 for b in range(16)), 0.8, 62, False),
    synth.Workload("short_192", _shape(dtype="f32", d=192, n_draft_layers=1, vocab=58401, block=16), (3,), 0.8, 63, False),
]


@pytest.mark.parametrize("w", SHORT_K, ids=lambda w: w.name)
def test_fp32_tiles_of_a_short_k_match_oracle(w):
    _step_matches_oracle(w)


def test_simt_tiles_of_a_short_k_on_bf16_match_oracle():
    from paper_2606_02091_gb300 import FLAG_SIMT_GEMM
    w = SHORT_K[0]
    _step_matches_oracle(w.with_(shape=dataclasses.replace(w.shape, dtype="bf16")), FLAG_SIMT_GEMM)


@pytest.mark.parametrize("flag,kw", [("", {}), ("FLAG_FUSION_FC", dict(fusion_fc=True)), ("FLAG_DFLASH_FC", dict(dflash_fc=True)),
                                     ("FLAG_SHARED_KV", dict(shared_kv=True))], ids=lambda x: x if isinstance(x, str) else "")
def test_fp32_tiles_of_a_fill_match_oracle(flag, kw):
    """The context projection (rotary epilogue, grouped weights), biased and grouped stores, a contraction across
    stacked token groups."""
    import paper_2606_02091_gb300 as P
    _step_matches_oracle(TILED_FILL, getattr(P, flag) if flag else 0, **kw)


# bf16 projections of more than 128 token rows (two-SM tiles of 256 rows x 64 to 256 features): one row
# past 128 (gate/up only) with a vocabulary that no 16-byte row fits, the summed projections (Q/K/V, O, down)
# at their last 224 rows on the single-SM GEMM and one past them, second 256-row tiles of one row (a fill) and of 32, odd counts of
# 64-wide k-blocks (5, 3, 17), feature counts that end inside a tile, both head sizes, and fills whose token
# tiles are partly or all padding
PAIR_CASES = [
    synth.Workload("pair_129", _shape(block=3, vocab=1003, ffn=192, d=320), tuple(3 + b % 5 for b in range(43)), 0.8, 41),
    synth.Workload("pair_192", _shape(block=32, vocab=1000, ffn=1088, d=320, n_q_heads=8), (40, 3, 33, 1, 17, 64), 0.8, 42),
    synth.Workload("pair_224", _shape(block=32, vocab=1000, ffn=1088, d=320, n_q_heads=8), (40, 3, 33, 1, 17, 64, 5), 0.8, 48),
    synth.Workload("pair_225", _shape(block=5, vocab=1000, ffn=1088, d=320, n_q_heads=8), tuple(3 + b % 7 for b in range(45)), 0.8, 49),
    synth.Workload("pair_160_odd_vocab", _shape(block=32, vocab=1003, ffn=320), (40, 3, 33, 1, 17), 0.8, 46),
    synth.Workload("pair_fill_257", _shape(head_dim=128, ffn=192), (257,), 0.8, 43),
    synth.Workload("pair_288", _shape(block=32, vocab=2004, head_dim=128, ffn=704, d=576), (300, 1, 2, 5, 257, 9, 3, 30, 64), 0.8, 44),
]


@pytest.mark.parametrize("w", PAIR_CASES, ids=lambda w: w.name)
@pytest.mark.parametrize("flag", ["", "FLAG_DETERMINISTIC"])
def test_two_sm_gemm_matches_oracle(w, flag):
    import paper_2606_02091_gb300 as P
    _step_matches_oracle(w, getattr(P, flag) if flag else 0)


def test_two_sm_gemm_of_one_ring_repeats_exactly():
    """Contractions of one to three k-blocks: every copy and commit of a launch belongs to its last ring, so
    a CTA that left before they had arrived would let them into the next launch's shared memory. Blocks drafted
    back to back with fixed sums hold the same bits, and the first agrees with the oracle."""
    import torch
    from paper_2606_02091_gb300 import FLAG_DETERMINISTIC
    w = synth.Workload("pair_one_ring", _shape(d=64, ffn=192, vocab=1000, block=32), (300, 1, 2, 5, 257, 9, 3, 30, 64), 0.8, 47)
    _step_matches_oracle(w, FLAG_DETERMINISTIC)
    g = GpuSide(w, flags=FLAG_DETERMINISTIC)
    g.fuse(w.ctx_lens, want_fused=False)
    s, n = w.shape, 16
    last = torch.tensor(synth.initial_tokens(w), device="cuda")
    toks = torch.zeros((n, w.batch, s.block - 1), dtype=torch.int32, device="cuda")
    logits = torch.zeros((n, w.batch, s.block - 1, s.vocab), dtype=torch.float32, device="cuda")
    for i in range(n):
        g.lib.draft_block(last, toks[i], logits[i])
    torch.cuda.synchronize()
    assert logits[0].any() and torch.equal(logits, logits[:1].expand_as(logits)) and torch.equal(toks, toks[:1].expand_as(toks))
    assert g.lib.device_error() == 0


@pytest.mark.parametrize("flag,kw", [("FLAG_FUSION_FC", dict(fusion_fc=True)), ("FLAG_DFLASH_FC", dict(dflash_fc=True)),
                                     ("FLAG_SHARED_KV", dict(shared_kv=True))], ids=lambda x: x if isinstance(x, str) else "")
@pytest.mark.parametrize("d", [256, 320])
def test_two_sm_gemm_of_the_variants_matches_oracle(flag, kw, d):
    """Biased and grouped stores, a contraction across stacked token groups (4 and 5 k-blocks each),
    token groups shared by all weight groups, weight groups with rows between them."""
    import paper_2606_02091_gb300 as P
    w = synth.Workload("pair_variant", _shape(d=d, n_target_layers=3), (150, 90), 0.8, 45)
    _step_matches_oracle(w, getattr(P, flag), **kw)


# gate/up tiles of 80 (125 and 152 SMs' worth), 112, 64 and 96 weight rows, token tiles of 16, 32, 48 and 64 rows (one
# and two of them), stages of four and of two k-blocks, the last one partly filled
SWIGLU_CASES = [
    synth.Workload("swiglu_9984", _shape(d=128, ffn=9984, block=9), (33,), 0.8, 61),
    synth.Workload("swiglu_16960", _shape(d=128, ffn=16960, block=16), (20, 40), 0.8, 62),
    synth.Workload("swiglu_9728", _shape(d=128, ffn=9728, block=11), (20, 40, 1, 7), 0.8, 63),
    synth.Workload("swiglu_12288", _shape(d=192, ffn=12288, block=16), (20, 40, 1, 7), 0.8, 64),
    synth.Workload("swiglu_6144", _shape(d=448, ffn=6144, block=24), (20, 40, 1, 7, 3), 0.8, 65),
]


@pytest.mark.parametrize("w", SWIGLU_CASES, ids=lambda w: w.name)
def test_gate_up_tiles_match_oracle(w):
    _step_matches_oracle(w)


# logit tiles of 96 and 64 weight rows, the last of 4, 36 and 64; 15, 60 and 155 token rows, the last with staging
# for 32 tokens in place of 64
LOGIT_CASES = [
    synth.Workload("logits_14500", _shape(d=192, n_draft_layers=1, vocab=14500, block=16), (20,), 0.8, 71),
    synth.Workload("logits_9700", _shape(d=192, n_draft_layers=1, vocab=9700, block=16), (20, 40, 1, 7), 0.8, 72),
    synth.Workload("logits_40000", _shape(d=192, n_draft_layers=1, vocab=40000, block=32), (20, 40, 1, 7, 3), 0.8, 73),
]


@pytest.mark.parametrize("w", LOGIT_CASES, ids=lambda w: w.name)
def test_logit_tiles_match_oracle(w):
    _step_matches_oracle(w)


# context fills of at least two positions per SM. The ring refilled by the warps in turn: one and two feature groups
# per thread (five and six draft layers), two CTAs per SM, warps with and without their second group; by a
# producer warp: one and two CTAs per SM, the widest rows of each, one feature past the narrow ones. Target-layer
# counts that end inside a stage of 6 (bf16) or 3 and 4 (fp32) rows, fewer target rows than a stage, positions past
# a sequence's end, one position per step of the grid
FILL_CASES = [
    synth.Workload("fill_d2112_D6_T7", _shape(d=2112, n_draft_layers=6, n_target_layers=7, ffn=64, block=2), (170, 140), 0.8, 51),
    synth.Workload("fill_d4096_D8_T3", _shape(d=4096, n_draft_layers=8, n_target_layers=3, ffn=64, block=2), (305,), 0.8, 52),
    synth.Workload("fill_d704_D5_T13", _shape(d=704, n_draft_layers=5, n_target_layers=13, ffn=64, block=2), (300, 9), 0.8, 53),
    synth.Workload("fill_d2816_D3_T6", _shape(d=2816, n_draft_layers=3, n_target_layers=6, ffn=64, block=2), (305,), 0.8, 54),
    synth.Workload("fill_f32_d320_D7_T5", _shape(dtype="f32", d=320, n_draft_layers=7, n_target_layers=5, ffn=64, block=2), (306,), 0.8, 55),
    synth.Workload("fill_d1088_D5_T13", _shape(d=1088, n_draft_layers=5, n_target_layers=13, ffn=64, block=2), (300, 9), 0.8, 56),
    synth.Workload("fill_d2816_D3_T9", _shape(d=2816, n_draft_layers=3, n_target_layers=9, ffn=64, block=2), (305,), 0.8, 57),
    synth.Workload("fill_d2048_D8_T8", _shape(d=2048, n_draft_layers=8, n_target_layers=8, ffn=64, block=2), (170, 1, 140), 0.8, 58),
    synth.Workload("fill_d1024_D1_T1", _shape(d=1024, n_draft_layers=1, n_target_layers=1, ffn=64, block=2), (700,), 0.8, 59),
    synth.Workload("fill_d64_D5_T36", _shape(d=64, n_draft_layers=5, n_target_layers=36, ffn=64, block=2), (160, 3, 150), 0.8, 60),
    synth.Workload("fill_d2048_D5_T8", _shape(d=2048, n_draft_layers=5, n_target_layers=8, ffn=64, block=2), (305,), 0.8, 74),
    synth.Workload("fill_d2560_D1_T1", _shape(d=2560, n_draft_layers=1, n_target_layers=1, ffn=64, block=2), (400,), 0.8, 80),
    synth.Workload("fill_d2560_D8_T7", _shape(d=2560, n_draft_layers=8, n_target_layers=7, ffn=64, block=2), (305,), 0.8, 81),
    synth.Workload("fill_d2304_D4_T8", _shape(d=2304, n_draft_layers=4, n_target_layers=8, ffn=64, block=2), (305,), 0.8, 82),
    synth.Workload("fill_f32_d2560_D1_T2", _shape(dtype="f32", d=2560, n_draft_layers=1, n_target_layers=2, ffn=64, block=2), (305,), 0.8, 83),
    synth.Workload("fill_f32_d2688_D6_T4", _shape(dtype="f32", d=2688, n_draft_layers=6, n_target_layers=4, ffn=64, block=2), (305,), 0.8, 84),
    synth.Workload("fill_d4096_D4_T8", _shape(d=4096, n_draft_layers=4, n_target_layers=8, ffn=64, block=2), (305,), 0.8, 75),
    synth.Workload("fill_f32_d2112_D6_T7", _shape(dtype="f32", d=2112, n_draft_layers=6, n_target_layers=7, ffn=64, block=2), (170, 140), 0.8, 76),
    synth.Workload("fill_f32_d1088_D2_T5", _shape(dtype="f32", d=1088, n_draft_layers=2, n_target_layers=5, ffn=64, block=2), (305,), 0.8, 77),
    synth.Workload("fill_f32_d1024_D5_T9", _shape(dtype="f32", d=1024, n_draft_layers=5, n_target_layers=9, ffn=64, block=2), (300, 9), 0.8, 78),
    synth.Workload("fill_f32_d4096_D2_T4", _shape(dtype="f32", d=4096, n_draft_layers=2, n_target_layers=4, ffn=64, block=2), (305,), 0.8, 79),
]


@pytest.mark.parametrize("w", FILL_CASES, ids=lambda w: w.name)
def test_fill_fusion_matches_oracle(w):
    _step_matches_oracle(w)


@pytest.mark.parametrize("vocab,block,sampled", [(1000, 8, False), (1003, 8, False), (1000, 8, True), (1003, 5, True), (300, 1, False)])
def test_copies_to_aligned_and_unaligned_buffers_agree(vocab, block, sampled):
    """logits_out and hidden_out as written by the kernels (16-byte aligned buffers) and as copied
    afterwards (buffers 4 bytes further) hold the same bits; the deterministic mode repeats exactly."""
    import torch
    from paper_2606_02091_gb300 import FLAG_DETERMINISTIC
    w = synth.Workload("copies", _shape(vocab=vocab, block=block), (33, 70), 0.8, 36)
    g = GpuSide(w, flags=FLAG_DETERMINISTIC)
    g.fuse(w.ctx_lens, want_fused=False)
    s = w.shape
    last = torch.tensor(synth.initial_tokens(w), device="cuda")
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    got = []
    for off in (0, 1):
        toks = torch.zeros((w.batch, block - 1), dtype=torch.int32, device="cuda")
        logits = torch.zeros(w.batch * (block - 1) * vocab + 4, dtype=torch.float32, device="cuda")[off:]
        hidden = torch.zeros((s.n_draft_layers + 1) * w.batch * block * s.d + 4, dtype=torch.float32, device="cuda")[off:]
        if sampled:
            g.lib.draft_block_sampled(last, 1.0, 7, step, toks, logits, hidden)
        else:
            g.lib.draft_block(last, toks, logits, hidden)
        torch.cuda.synchronize()
        got.append([t.cpu().numpy() for t in (toks, logits[:w.batch * (block - 1) * vocab], hidden[:(s.n_draft_layers + 1) * w.batch * block * s.d])])
        assert got[-1][2].any() and (block == 1 or got[-1][1].all())
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("batch,block", [(9, 2), (31, 8), (33, 17), (64, 32)])
def test_verification_of_many_sequences_matches_oracle(batch, block):
    """The acceptance of up to four sequences at a time per warp: every prefix length, both entry points."""
    import torch
    w = synth.Workload("many", _shape(block=block, vocab=301), (1,) * batch, 0.8, 64)
    g, V, rng = GpuSide(w), w.shape.vocab, np.random.default_rng(64)
    draft = rng.integers(0, V, (batch, block - 1)).astype(np.int32)
    lg = rng.standard_normal((batch, block, V)).astype(np.float32)
    for b in range(batch):
        for k in range(b % block):
            lg[b, k, draft[b, k]] = 20.0
    want = [O.verify_from_logits(draft[b], lg[b]) for b in range(batch)]
    d, t = torch.from_numpy(draft).cuda(), torch.from_numpy(lg).cuda()
    for call, arg in ((g.lib.verify_logits, t), (g.lib.verify_accept, t.argmax(-1).int())):
        acc, nxt = (torch.zeros(batch, dtype=torch.int32, device="cuda") for _ in range(2))
        call(d, arg, acc, nxt)
        assert list(zip(acc.cpu().tolist(), nxt.cpu().tolist())) == want


def test_verification_reports_every_phase():
    """The trace hook sees the phases of the verification calls, also those whose work another launch does."""
    import torch
    import paper_2606_02091_gb300 as P
    w = synth.Workload("phases", _shape(), (9, 4), 0.8, 37)
    g, s, seen = GpuSide(w), w.shape, []
    g.fuse(w.ctx_lens, want_fused=False)
    g.draft(synth.initial_tokens(w))

    @P._lib.TRACE_FN
    def hook(user, name, phase, stream):
        seen.append((name.decode(), phase))

    drafts = torch.zeros((w.batch, s.block - 1), dtype=torch.int32, device="cuda")
    target = torch.randn((w.batch, s.block, s.vocab), device="cuda")
    acc, nxt = (torch.zeros(w.batch, dtype=torch.int32, device="cuda") for _ in range(2))
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    P.load().dflare_set_trace(g.lib.raw, hook, None)
    g.lib.verify_logits(drafts, target, acc, nxt)
    assert seen == [(n, p) for n in ("argmax_target", "verify") for p in (0, 1)]
    seen.clear()
    g.lib.verify_sampled(drafts, target, 1.0, 7, step, acc, nxt)
    assert seen == [(n, p) for n in ("spec_stats", "spec_accept", "spec_resample") for p in (0, 1)]
    P.load().dflare_set_trace(g.lib.raw, P._lib.TRACE_FN(), None)
    torch.cuda.synchronize()
