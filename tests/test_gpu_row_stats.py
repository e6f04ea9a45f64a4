"""One-pass row statistics of stored logits: edges of the vocabulary's split over blocks and
threads (needs a B200).  fp32 drafter, so the kernel reads exactly the logits it is compared on."""
import numpy as np
import pytest
import torch

import oracle
import synth
from harness import Pair

pytestmark = pytest.mark.gpu


# vocab 5: fewer tokens than a warp; 1003: rows that are not 16-byte aligned; 2050 / 40001: shares
# of blocks and threads with a remainder; B = 1, 40, 128 rows x 2: 8, 4 or 2 blocks a row and one
@pytest.mark.parametrize("vocab,B", [(5, 1), (1003, 2), (2050, 3), (4100, 1), (16384, 40), (40001, 1), (33000, 128)])
def test_row_stats_edges(vocab, B):
    s = synth.CONFIGS["mini32"].with_(hidden=64, n_heads=1, n_kv_heads=1, ffn=64, vocab=vocab, k_masks=1)
    W = synth.weights(s)
    W["w_lm"] = W["w_lm"] * np.float32(20.0)
    if vocab == 2050:
        W["w_lm"][:] = W["w_lm"][:1]        # every logit of a row is equal: more ties than the list takes
    p = Pair(s, B, lens=[3] * B, weights=W, oracle_seqs=[])
    n = min(5, vocab)
    out = p.g.draft_step_sampled(list(range(B)), p.to_device(p.hidden_last), p.to_device(p.token_last), 0.9, 3, 4, top_n=n)
    torch.cuda.synchronize()
    lg = out["logits"].double().cpu().numpy().reshape(-1, vocab)
    order = np.argsort(-lg, axis=-1, kind="stable")[:, :n]      # ties to the lower id
    assert np.array_equal(out["top_ids"].cpu().numpy().reshape(-1, n), order)
    assert np.array_equal(out["top_logit"].cpu().numpy().reshape(-1, n), np.take_along_axis(lg, order, -1).astype(np.float32))
    assert np.array_equal(out["row_max"].cpu().numpy().ravel(), lg.max(-1).astype(np.float32))
    lse = lg.max(-1) + np.log(np.exp(lg - lg.max(-1, keepdims=True)).sum(-1))
    # exponentials to 2^-20 each, fp32 sums over a tree of depth < 20: 2^-19 on ln(sum), plus the
    # rounding of the stored value
    assert np.abs(out["row_lse"].cpu().numpy().ravel() - lse).max() < 2.0 ** -18 + 2.0 ** -23 * np.abs(lse).max()
    ids = np.array([b | (j << 8) for b in range(B) for j in range(s.rows)], np.int32)
    tok, margin = oracle.gumbel_sample(lg, 0.9, 3, 4, ids)
    got = out["sampled"].cpu().numpy().ravel()
    # single-precision noise: 2^-21 of values up to 17
    assert all(g == t or m < 2e-5 for g, t, m in zip(got, tok, margin))


# Without the sampler the blocks a row takes depend on how many clusters find room: counts of rows on both sides of a
# wave's last places (80 | 82 of clusters of 5, 100 | 102 of 4, 136 | 138 of 3, 222 | 224 of 2)
@pytest.mark.parametrize("vocab", [10241, 32000])
def test_row_stats_around_a_wave(vocab):
    s = synth.CONFIGS["mini32"].with_(hidden=64, n_heads=1, n_kv_heads=1, ffn=64, vocab=vocab, k_masks=1)
    W = synth.weights(s)
    W["w_lm"] = W["w_lm"] * np.float32(20.0)
    p = Pair(s, 112, lens=[3] * 112, weights=W, oracle_seqs=[])
    h, t = p.to_device(p.hidden_last), p.to_device(p.token_last)
    for B in (39, 40, 41, 50, 51, 68, 69, 111, 112):
        out = p.g.draft_step(list(range(B)), h[:B], t[:B], top_n=3)
        lg = out["logits"].double().cpu().numpy().reshape(-1, vocab)
        order = np.argsort(-lg, axis=-1, kind="stable")[:, :3]
        assert np.array_equal(out["top_ids"].cpu().numpy().reshape(-1, 3), order), B
        assert np.array_equal(out["row_max"].cpu().numpy().ravel(), lg.max(-1).astype(np.float32)), B
        lse = lg.max(-1) + np.log(np.exp(lg - lg.max(-1, keepdims=True)).sum(-1))
        assert np.abs(out["row_lse"].cpu().numpy().ravel() - lse).max() < 2.0 ** -18 + 2.0 ** -23 * np.abs(lse).max(), B
