"""Tensor-memory attention (draft steps of more than 16 rows, head_dim 128): edges of the key tiles
and of the 16-key groups, empty contexts, pairs shared by several CTAs and many pairs per CTA,
grouped query heads, scores that outgrow their reference (needs a B200)."""
import numpy as np
import pytest

import synth
from harness import Pair, as_f64, logits_close

pytestmark = pytest.mark.gpu


def _check(p, s, seqs):
    got = p.gpu_step(top_n=1)
    for b in seqs:
        want = p.oracle_step(b)
        assert logits_close(got["logits"][b], want["logits"], s.dtype) <= 1.0, b     # the logits gate
        assert logits_close(got["feat"][b], want["feat"], s.dtype) <= 1.0, b
    assert np.isfinite(got["logits"]).all()
    assert p.g.check_guards() == 0 and p.g.poll() == 0
    again = p.gpu_step(top_n=1)
    assert np.array_equal(got["logits"], again["logits"])


# (heads, kv heads, k): rows of a kv head's group 3 -> 8, 9 -> 16, 6 x 3 = 18 -> 24, 2 x 16 = 32
@pytest.mark.parametrize("heads,kv_heads,k", [(6, 6, 2), (6, 6, 8), (6, 1, 2), (6, 3, 15)])
def test_key_tile_edges(heads, kv_heads, k):
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=k)
    # (112 and 113: the new rows just fit behind the last tile's keys, and just do not)
    lens = [0, 1, 8, 15, 16, 17, 31, 33, 112, 113, 127, 128, 129, 255, 257, 300]
    p = Pair(s, len(lens), context="import", lens=lens)
    _check(p, s, range(len(lens)))


# 2 sequences x 1 kv head: 34 + 17 units, several CTAs per pair; 128 x 6 pairs: several pairs per CTA
@pytest.mark.parametrize("kv_heads,lens", [(1, [4300, 2100]), (6, [130 + b for b in range(128)])])
def test_units_dealt_to_ctas(kv_heads, lens):
    s = synth.CONFIGS["mini"].with_(n_kv_heads=kv_heads, n_heads=3 * kv_heads if kv_heads == 1 else 6, k_masks=8)
    seqs = [0, 1] if len(lens) == 2 else [0, 1, 63, 127]
    p = Pair(s, len(lens), context="import", lens=lens, oracle_seqs=seqs)
    _check(p, s, seqs)


def test_scores_outgrow_their_reference():
    """Keys whose scores exceed that of the first key by far more than 2^64, and keep growing from tile
    to tile: the sums and outputs so far are rescaled."""
    s = synth.CONFIGS["mini"].with_(k_masks=8)
    lens = [700, 260]
    p = Pair(s, 2, context="import", lens=lens)
    for b, n in enumerate(lens):
        K, V = synth.kv_rows(s, ("kv", b), n)
        Kf = synth.bf16_bits_to_f32(K) * np.linspace(1, 250, n, dtype=np.float32)[:, None]
        K = synth.f32_to_bf16_bits(Kf)
        p.o.kv_import(b, as_f64(K, s.dtype), as_f64(V, s.dtype))
        p.g.kv_import(b, p.to_device(K), p.to_device(V))
    _check(p, s, range(2))


# groups of 20 and 32 query rows run on a ring of five slots, whose slots alternate between the two MMA
# issuers; more K / V than the L2 holds, so that tiles come late and out of order
@pytest.mark.parametrize("kv_heads,k", [(8, 4), (16, 15)])
def test_odd_ring_with_late_tiles(kv_heads, k):
    import torch
    import paper_2410_05589_b200 as ps
    from harness import oracle_for
    B, L = 12, 4000
    s = synth.CONFIGS["mini"].with_(hidden=256, n_heads=32, n_kv_heads=kv_heads, ffn=256, vocab=1000, k_masks=k)
    W = synth.weights(s)
    g = ps.drafter_from_shape(s, W, max_batch=B, max_ctx=L + k + 1)
    o = oracle_for(s, W, 1, L + k + 1)
    K, V = synth.kv_rows(s, "kv", L)
    o.kv_import(0, as_f64(K, s.dtype), as_f64(V, s.dtype))
    for b in range(B):
        g.kv_import(b, ps.to_device(K), ps.to_device(V))
    h, t = synth.hidden_states(s, "last", 1), synth.token_ids(s, "last", 1)
    want = o.draft_step(0, h, int(t[0]))["logits"]
    hl, tl = ps.to_device(np.repeat(h, B, 0)), ps.to_device(np.repeat(t, B))
    outs = [g.draft_step(list(range(B)), hl, tl, top_n=1)["logits"] for _ in range(8)]
    torch.cuda.synchronize()
    got = outs[0].cpu().numpy()
    for b in range(B):
        assert logits_close(got[b], want, s.dtype) <= 1.0, b     # the logits gate
    assert all(torch.equal(outs[0], x) for x in outs[1:]) and g.poll() == 0


# The rule of the dispatch: 6 key tiles of a query head for every SM (16 with more than 16 query rows a kv
# head).  The edges once more in batches beyond it, 8 times the same lengths.
@pytest.mark.parametrize("heads,kv_heads,k", [(6, 6, 2), (6, 6, 8), (18, 3, 2), (16, 8, 15)])
def test_key_tile_edges_in_full_batches(heads, kv_heads, k):
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=k)
    lens = [0, 1, 8, 15, 16, 17, 31, 33, 112, 113, 127, 128, 129, 255, 257, 300] * 8
    p = Pair(s, len(lens), context="import", lens=lens, oracle_seqs=range(16))
    _check(p, s, range(16))


def test_long_sequences_dealt_to_several_ctas():
    s = synth.CONFIGS["mini"].with_(n_heads=24, n_kv_heads=8, k_masks=4)
    p = Pair(s, 4, context="import", lens=[4300, 2100, 900, 3000], oracle_seqs=[0, 2])
    _check(p, s, [0, 2])


def test_scores_outgrow_their_reference_in_a_full_batch():
    s = synth.CONFIGS["mini"].with_(k_masks=8)
    lens = [700, 260] + [700] * 24
    p = Pair(s, len(lens), context="import", lens=lens, oracle_seqs=[0, 1])
    for b in (0, 1):
        K, V = synth.kv_rows(s, ("kv", b), lens[b])
        Kf = synth.bf16_bits_to_f32(K) * np.linspace(1, 250, lens[b], dtype=np.float32)[:, None]
        K = synth.f32_to_bf16_bits(Kf)
        p.o.kv_import(b, as_f64(K, s.dtype), as_f64(V, s.dtype))
        p.g.kv_import(b, p.to_device(K), p.to_device(V))
    _check(p, s, range(2))


@pytest.mark.parametrize("heads,kv_heads,B,L", [(6, 6, 37, 500), (6, 6, 36, 500), (16, 4, 37, 500), (16, 4, 36, 500)])
def test_both_sides_of_the_line(heads, kv_heads, B, L):
    """6 heads x 37 sequences x 4 tiles are 888 = 6 x 148; 16 heads 2368 = 16 x 148."""
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=4)
    p = Pair(s, B, context="import", lens=[L] * B, oracle_seqs=[0, B - 1])
    _check(p, s, [0, B - 1])


# Training layout: groups of one slot share the query rows of a pair.  Rows of a sequence times sequences a
# bundle: 5 x 3 (all full; 1 and 2 left over; four slots, so passes of 3 + 1), 3 x 2 heads x 2, 9 x 1, 2 x 8 (from an empty
# context; 4 left over), 1 x 16; contexts that cross a tile within a bundle, more groups than slots
@pytest.mark.parametrize("heads,kv_heads,k,L0,n,slots", [(6, 6, 4, 200, 90, 90), (6, 6, 4, 200, 91, 91), (6, 6, 4, 200, 92, 92),
                                                         (18, 18, 4, 1600, 16, 4), (6, 3, 2, 120, 131, 128), (6, 6, 8, 250, 80, 80),
                                                         (18, 18, 1, 0, 100, 128), (18, 18, 0, 100, 70, 70)])
def test_groups_of_one_slot(heads, kv_heads, k, L0, n, slots):
    import torch
    import paper_2410_05589_b200 as ps
    from harness import oracle_for
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=k, vocab=600)
    assert _tiles(L0, min(n, slots)) * heads >= 6 * 148         # the rule of the dispatch, for the first pass
    W = synth.weights(s)
    g = ps.drafter_from_shape(s, W, max_batch=slots, max_ctx=L0 + n + k + 1)
    o = oracle_for(s, W, 1, L0 + n + k + 1)
    if L0:
        K, V = synth.kv_rows(s, "ctx", L0)
        g.kv_import(0, ps.to_device(K), ps.to_device(V))
        o.kv_import(0, as_f64(K, s.dtype), as_f64(V, s.dtype))
    h, t = synth.hidden_states(s, "new", n), synth.token_ids(s, "new", n)
    hid, tok = ps.to_device(h), ps.to_device(t)
    out = g.group_forward(0, hid, tok, want_feat=True)
    want = o.group_forward(0, h, t)
    for name in ("logits", "feat"):
        assert logits_close(out[name].double().cpu().numpy(), want[name], s.dtype) <= 1.0, name     # the logits gate
    assert g.check_guards() == 0 and g.poll() == 0
    again = g.group_forward(0, hid, tok, want_feat=True)
    assert torch.equal(out["logits"], again["logits"])


def _tiles(L0, n):
    return sum(max(1, -(-(L0 + t) // 128)) for t in range(n))


# A bundle reads keys that only some of its groups see: what those hold must not reach the others.  Position `bad` of the
# new ones is the first, the middle or the last of its bundle of 3 (5 rows a group), 8 (2), 2 (2 heads x 3) or 16 (1)
# groups; the cached keys of the bundle end before, in and behind a tile's edge (128, 256)
_BUNDLES = [(6, 6, 4, 201, 90, (30, 31, 32, 54, 55, 89)), (18, 18, 1, 125, 100, (0, 2, 3, 4, 7, 99)),
            (6, 3, 2, 120, 131, (6, 7, 8, 130)), (18, 18, 0, 125, 100, (2, 3, 15))]


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("heads,kv_heads,k,L0,n,bad", _BUNDLES)
def test_nonfinite_position_stays_out_of_the_groups_before_it(heads, kv_heads, k, L0, n, bad, value):
    import torch
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=k)
    assert _tiles(L0, n) * heads >= 6 * 148         # the rule of the dispatch
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=min(n, 128), max_ctx=L0 + n + k + 1)
    g.kv_import(0, *(ps.to_device(x) for x in synth.kv_rows(s, "ctx", L0)))
    hid, tok = ps.to_device(synth.hidden_states(s, "new", n)), ps.to_device(synth.token_ids(s, "new", n))
    clean = g.group_forward(0, hid, tok)["logits"].double().cpu().numpy()
    for t in bad:
        h = hid.clone()
        h[t, 100] = value
        out = g.group_forward(0, h, tok)["logits"]
        assert torch.isfinite(out[:t]).all() and torch.isnan(out[t:]).all(), t
        if t:
            assert logits_close(out[:t].double().cpu().numpy(), clean[:t], s.dtype) <= 1.0, t     # the logits gate
    assert g.check_guards() == 0


@pytest.mark.parametrize("heads,kv_heads,k,L0,n,bad", _BUNDLES)
def test_value_that_overflows_stays_out_of_the_groups_before_it(heads, kv_heads, k, L0, n, bad):
    """Finite keys, one channel of the value row infinite: channel 7 of the normalised row is 0 but at one position,
    and a value channel is 3e38 times it.  (The channel's way into the output has weight 0, so that nothing else
    changes.)"""
    import torch
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"].with_(n_heads=heads, n_kv_heads=kv_heads, k_masks=k)
    w = {name: ps.to_device(x) for name, x in synth.weights(s).items() if x is not None}
    w["w_fc"][7] = 0.0
    w["w_fc"][7, s.hidden + 3] = 8.0                # (fc reads embedding, then features)
    w["w_fc"][7, 3] = 8.0
    w["embed"][:, 3] = 0.0
    w["mask_embed"][:, 3] = 0.0
    w["mask_feat"][:, 3] = 0.0
    w["w_v"][5] = 0.0
    w["w_o"].view(s.hidden, heads, s.head_dim)[:, :heads // kv_heads, 5] = 0.0
    kw = dict(dtype=s.dtype, hidden=s.hidden, n_heads=heads, n_kv_heads=kv_heads, head_dim=s.head_dim, ffn=s.ffn, vocab=s.vocab,
              k_masks=k, max_batch=min(n, 128), max_ctx=L0 + n + k + 1)
    ctx = [ps.to_device(x) for x in synth.kv_rows(s, "ctx", L0)]
    hid, tok = ps.to_device(synth.hidden_states(s, "new", n)), ps.to_device(synth.token_ids(s, "new", n))
    hid[:, 3] = 0.0
    plain = ps.Drafter(weights=w, **kw)
    w_v = w["w_v"].clone()
    w_v[5, 7] = 3e38
    huge = ps.Drafter(weights=dict(w, w_v=w_v), **kw)
    for g in (plain, huge):
        g.kv_import(0, *ctx)
    for t in bad:
        h = hid.clone()
        h[t, 3] = 1.0
        want = plain.group_forward(0, h, tok)["logits"]
        out = huge.group_forward(0, h, tok)["logits"]
        assert torch.isfinite(want).all() and torch.isfinite(out[:t]).all() and torch.isnan(out[t:]).all(), t
        if t:
            assert logits_close(out[:t].double().cpu().numpy(), want[:t].double().cpu().numpy(), s.dtype) <= 1.0, t     # the logits gate
    assert huge.check_guards() == 0
