"""CTA-pair GEMM path (more than 16 rows): edges of its row padding and row tiles, whole and shared
tiles, ragged matrix ends, grouped-query k / v, bias and the embedding-only input (needs a B200)."""
import numpy as np
import pytest

import synth
from harness import Pair, logits_close

pytestmark = pytest.mark.gpu


# rows B * (k + 1): 17 and 33 (one past a padding step), 32 (none), 255 (one row tile, almost full),
# 258 (two row tiles), 1152 (five row tiles: more tiles than CTA pairs, so some go whole)
@pytest.mark.parametrize("B,k,kv_heads,bias,flags", [(17, 0, 6, False, 0), (33, 0, 2, True, 0), (16, 1, 6, False, 8),
                                                     (85, 2, 3, False, 0), (86, 2, 6, True, 0), (128, 8, 6, False, 0)])
def test_pair_gemm_rows_match_oracle(B, k, kv_heads, bias, flags):
    s = synth.CONFIGS["mini"].with_(k_masks=k, n_kv_heads=kv_heads)
    seqs = sorted({0, B // 2, B - 1})
    p = Pair(s, B, with_bias=bias, lens=[1 + (7 * b) % 41 for b in range(B)], flags=flags, oracle_seqs=seqs)
    got = p.gpu_step(top_n=1)
    for b in seqs:
        want = p.oracle_step(b)
        assert logits_close(got["logits"][b], want["logits"], s.dtype) <= 1.0, b     # the logits gate
    assert np.isfinite(got["logits"]).all()
    assert p.g.check_guards() == 0 and p.g.poll() == 0
    again = p.gpu_step(top_n=1)
    assert np.array_equal(got["logits"], again["logits"])     # sums are added in k order, whoever is first


# k ranges long enough that the q|k|v, gate|up and LM-head tiles are shared by several pairs: one row
# tile, one that is not full, two
@pytest.mark.parametrize("B,k", [(4, 4), (30, 4), (64, 4)])
def test_pair_gemm_shared_tiles_match_oracle(B, k):
    s = synth.CONFIGS["mini"].with_(k_masks=k, hidden=2048, n_heads=16, n_kv_heads=4, ffn=5504)
    seqs = [0, B - 1]
    p = Pair(s, B, lens=[1 + (5 * b) % 23 for b in range(B)], oracle_seqs=seqs)
    got = p.gpu_step(top_n=1)
    for b in seqs:
        assert logits_close(got["logits"][b], p.oracle_step(b)["logits"], s.dtype) <= 1.0, b     # the logits gate
    assert p.g.check_guards() == 0 and p.g.poll() == 0
    assert np.array_equal(got["logits"], p.gpu_step(top_n=1)["logits"])


# up to 128 rows hi and lo planes are one operand: full and one past a padding step, the last count that is, the
# first that is not; whole and shared tiles
@pytest.mark.parametrize("B,k", [(32, 1), (97, 0), (64, 1), (43, 2)])
def test_planes_as_one_operand_match_oracle(B, k):
    s = synth.CONFIGS["mini"].with_(k_masks=k, hidden=2048, n_heads=16, n_kv_heads=4, ffn=5504)
    seqs = [0, B - 1]
    p = Pair(s, B, lens=[1 + (5 * b) % 23 for b in range(B)], oracle_seqs=seqs)
    got = p.gpu_step(top_n=1)
    for b in seqs:
        assert logits_close(got["logits"][b], p.oracle_step(b)["logits"], s.dtype) <= 1.0, b     # the logits gate
    assert p.g.check_guards() == 0 and p.g.poll() == 0


def test_row_counts_change_on_one_context():
    s = synth.CONFIGS["mini"].with_(k_masks=4)
    B = 60
    p = Pair(s, B, lens=[1 + (7 * b) % 41 for b in range(B)], oracle_seqs=[0])
    want = p.oracle_step(0)["logits"]
    first = {}
    for n in (4, 60, 17, 4, 9, 33, 60, 17, 2, 9):     # rows 20, 300, 85, ..., and 10 on the kernels of up to 16
        out = p.g.draft_step(list(range(n)), p.to_device(p.hidden_last[:n]), p.to_device(p.token_last[:n]), top_n=1)
        got = out["logits"].cpu().numpy()
        assert logits_close(got[0], want, s.dtype) <= 1.0, n     # the logits gate
        assert np.array_equal(got, first.setdefault(n, got)), n
    assert p.g.poll() == 0


def test_many_steps_in_a_row():
    """30 000 GEMM launches of CTA pairs behind one another, each behind kernels whose blocks may hold one SM of
    a pair longer than the other (the pair's allocation of tensor memory must not mind)."""
    s = synth.CONFIGS["mini"].with_(k_masks=4)
    p = Pair(s, 6, lens=[1 + 5 * b for b in range(6)], oracle_seqs=[0])
    hl, tl = p.to_device(p.hidden_last), p.to_device(p.token_last)
    out = {}
    first = p.g.draft_step(list(range(6)), hl, tl, out=out)["logits"].cpu().numpy()
    for _ in range(5000):
        p.g.draft_step(list(range(6)), hl, tl, out=out)
    assert p.g.poll() == 0 and np.array_equal(first, out["logits"].cpu().numpy())
    assert logits_close(first[0], p.oracle_step(0)["logits"], s.dtype) <= 1.0     # the logits gate


def test_long_append_with_whole_and_shared_tiles():
    """2048 new rows, hidden 5120: the fc's 80 tiles are one wave of whole ones and six shared ones, all
    through slots; k | v of the same pass lie on top of the fc's input and slots.  Twice, so that a pass
    follows one of another length."""
    import paper_2410_05589_b200 as ps
    import torch
    from harness import oracle_for
    B, n, n2 = 128, 16, 3
    s = synth.CONFIGS["mini"].with_(hidden=5120, n_heads=2, n_kv_heads=2, ffn=64, vocab=1000, k_masks=1)
    W = synth.weights(s)
    g = ps.drafter_from_shape(s, W, max_batch=B, max_ctx=40)
    seqs = [0, 77, B - 1]
    o = oracle_for(s, W, B, 40)
    for part, m in ((0, n), (1, n2), (2, n)):
        h, t = synth.hidden_states(s, ("new", part), B * m), synth.token_ids(s, ("new", part), B * m)
        g.kv_append(list(range(B)), [m] * B, ps.to_device(h), ps.to_device(t))
        for b in seqs:
            assert o.kv_append(b, h[b * m:(b + 1) * m], t[b * m:(b + 1) * m]) == 0
    torch.cuda.synchronize()
    for b in seqs:
        got = [x.float().cpu().numpy() for x in g.kv_export(b)]
        for a, w in zip(got, o.kv_export(b)):
            # values that agree to fp32 sums of 5120 and 10240 terms, rounded to bf16: one unit in the last place
            assert (np.abs(a - w) <= 2.0 ** -7 * np.abs(w) + 1e-4).all(), b
    assert g.poll() == 0 and g.check_guards() == 0


def test_hidden_sizes_beyond_the_row_norm():
    """Rows of more than 32768 features run in groups of up to 16 rows, as before the CTA-pair GEMM."""
    s = synth.CONFIGS["mini"].with_(hidden=32776, n_heads=1, n_kv_heads=1, ffn=64, vocab=200, k_masks=4)
    W = synth.weights(s.with_(hidden=64))            # (8: no fc, whose 4 GB are not drawn)
    H, d = s.hidden, s.head_dim
    rnd = np.random.default_rng(1)
    for n, shape in dict(embed=(200, H), mask_embed=(4, H), mask_feat=(4, H), w_q=(d, H), w_k=(d, H), w_v=(d, H), w_o=(H, d),
                         w_gate=(64, H), w_up=(64, H), w_down=(H, 64), w_lm=(200, H), g_in=(H,), g_post=(H,), g_final=(H,)).items():
        x = rnd.standard_normal(shape, np.float32) * 0.02 + (1.0 if n[0] == "g" else 0.0)
        W[n] = synth.f32_to_bf16_bits(x.astype(np.float32))
    p = Pair(s, 5, lens=[3, 0, 9, 1, 2], flags=8, context="import", oracle_seqs=[0, 4], weights=W)
    got = p.gpu_step(top_n=1)
    for b in (0, 4):
        assert logits_close(got["logits"][b], p.oracle_step(b)["logits"], s.dtype) <= 1.0, b     # the logits gate
    assert p.g.poll() == 0


# 2304 new rows, hidden 5120, 40 kv heads: a pass of 1792 rows (70 and 140 tiles on 74 pairs) and one of 512 instead of
# 2048 and 256; where a pass takes 520 rows at most, 528 rows as one of 512 and one of 16, which runs as a chained launch
@pytest.mark.parametrize("B,n,max_ctx,passes", [(128, 18, 40, (1792, 512)), (8, 66, 130, (512, 16))])
def test_append_in_passes_that_fill_their_waves(B, n, max_ctx, passes):
    import ctypes as C
    import paper_2410_05589_b200 as ps
    import torch
    from harness import oracle_for
    s = synth.CONFIGS["mini"].with_(hidden=5120, n_heads=40, n_kv_heads=40, ffn=64, vocab=200, k_masks=1)
    W = synth.weights(s)
    g = ps.drafter_from_shape(s, W, max_batch=B, max_ctx=max_ctx)
    most = min(2048, B * max_ctx // 2)
    rows = g.lib.ps_debug_append_pass_rows(C.byref(g.cfg), torch.cuda.get_device_properties(0).multi_processor_count, B * n, most)
    assert rows == passes[0] < most and sum(passes) == B * n
    h, t = synth.hidden_states(s, "new", B * n), synth.token_ids(s, "new", B * n)
    before = g.launch_count()
    g.kv_append(list(range(B)), [n] * B, ps.to_device(h), ps.to_device(t))
    torch.cuda.synchronize()
    # a pass: gather, fc, norm, k | v, store, or gather, chain, store
    assert g.launch_count() - before >= sum(5 if p > 16 else 3 for p in passes)
    o = oracle_for(s, W, B, max_ctx)
    edge = passes[0] // n
    for b in sorted({0, edge, min(edge + 1, B - 1), B - 1}):       # (the edge's rows lie in both passes)
        assert o.kv_append(b, h[b * n:(b + 1) * n], t[b * n:(b + 1) * n]) == 0
        got = [x.float().cpu().numpy() for x in g.kv_export(b)]
        for a, w in zip(got, o.kv_export(b)):
            # values that agree to fp32 sums of 5120 and 10240 terms, rounded to bf16: one unit in the last place
            assert (np.abs(a - w) <= 2.0 ** -7 * np.abs(w) + 1e-4).all(), b
    assert g.poll() == 0 and g.check_guards() == 0


# 148 | 150 rows of 4224 features: the row norm with the slots of four contributors in flight, and with one and two
# blocks an SM; 4096 and 5248 features stay with the first
@pytest.mark.parametrize("heads,B", [(33, 74), (33, 75), (32, 75), (41, 75)])
def test_row_norm_of_more_rows_than_sms(heads, B):
    s = synth.CONFIGS["mini"].with_(hidden=128 * heads, n_heads=heads, n_kv_heads=heads, ffn=512, vocab=500, k_masks=1)
    seqs = [0, B - 1]
    p = Pair(s, B, lens=[1 + b % 7 for b in range(B)], oracle_seqs=seqs)
    got = p.gpu_step(top_n=1)
    for b in seqs:
        assert logits_close(got["logits"][b], p.oracle_step(b)["logits"], s.dtype) <= 1.0, b     # the logits gate
    assert p.g.check_guards() == 0 and p.g.poll() == 0
