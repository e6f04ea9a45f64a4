"""Streaming chain verify (many row pairs): edges of the vocabulary's shares, cluster sizes 1 to 8,
references far below the maximum, rows without a distribution (needs a B200)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from harness import assert_verify_same

pytestmark = pytest.mark.gpu


def _drafter(vocab, k, B):
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini32"].with_(hidden=64, n_heads=1, n_kv_heads=1, ffn=64, vocab=vocab, k_masks=k)
    return ps, ps.drafter_from_shape(s, synth.weights(s), max_batch=B, max_ctx=k + 2)


# pairs: 40 (8 blocks each), 80 (4), 160 (2), 330 (1); vocab 4 and 132: shares of blocks without tokens
@pytest.mark.parametrize("vocab,B,n_draft,bonus,T", [(4, 40, 1, 0, 1.0), (132, 10, 4, 0, 0.7), (1000, 20, 3, 1, 1.0),
                                                     (32000, 16, 4, 1, 0.7), (4100, 82, 4, 0, 1.0), (32000, 32, 5, 0, 0.0),
                                                     (128256, 5, 5, 0, 1.0)])
@pytest.mark.parametrize("odd", [False, True])
def test_stream_verify_matches_oracle(vocab, B, n_draft, bonus, T, odd):
    ps, g = _drafter(vocab, n_draft - 1, B)
    n_target = n_draft + bonus
    tl = synth.zipf_logits(7, (vocab, B), B, n_target, vocab)
    dl = synth.noisy_draft_logits(7, (vocab, B), tl[:, :n_draft], 0.4)
    tok = synth.sample_from_logits(7, (vocab, B), dl, max(T, 0.5))
    if odd:
        tl[0, 0, -1] += 200.0                # the maximum is the last token, far above the first batch
        dl[4, 0, -1] += 200.0                # (in one of the rows only: p = q = 1 there would leave a residual of 1e-87)
        tl[1, 0, : vocab // 2] = -np.inf     # a reference batch without any finite logit
        dl[1, 0, : vocab // 2] = -np.inf
        tl[2, n_draft - 1] = -np.inf         # no distribution at all
        dl[3, 0, vocab // 3] = np.nan
        tl[B - 1, 0, 1] = np.inf
    for drafts in (dl, None):                # None: q is the point mass
        want = oracle.verify(tok, drafts, tl, T, 11, 5)
        out = g.verify(ps.to_device(tok), ps.to_device(drafts), ps.to_device(tl), T, 11, 5)
        torch.cuda.synchronize()
        assert_verify_same({k: v.cpu().numpy() for k, v in out.items()}, want)
        status = g.poll()
        assert T == 0.0 or status == (-6 if want["nonfinite"].any() else 0)


# both sides of the dispatch's lines: one block and clusters of 8 and 4 from 6144 tokens on, arg-max of many
# rows beyond 131072
@pytest.mark.parametrize("vocab,B,n_draft,bonus", [(6144, 2, 5, 0), (6148, 2, 5, 0), (8192, 1, 13, 0), (8192, 1, 14, 0),
                                                   (8192, 4, 5, 0), (8192, 4, 5, 1), (8192, 7, 5, 1), (131076, 11, 10, 0),
                                                   (131076, 12, 10, 0)])
@pytest.mark.parametrize("T", [0.0, 0.7])
def test_verify_dispatch_lines(vocab, B, n_draft, bonus, T):
    ps, g = _drafter(vocab, n_draft - 1, B)
    tl = synth.zipf_logits(9, (vocab, B), B, n_draft + bonus, vocab)
    dl = synth.noisy_draft_logits(9, (vocab, B), tl[:, :n_draft], 0.4)
    tok = synth.sample_from_logits(9, (vocab, B), dl, 0.7)
    want = oracle.verify(tok, dl, tl, T, 3, 8)
    out = g.verify(ps.to_device(tok), ps.to_device(dl), ps.to_device(tl), T, 3, 8)
    torch.cuda.synchronize()
    assert_verify_same({k: v.cpu().numpy() for k, v in out.items()}, want)
