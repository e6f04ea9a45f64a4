"""Kernels with fp32 activations: edges of the key tiles, of the row and feature blocks and of the column
chunks, both storage types and head sizes (needs a B200)."""
import numpy as np
import pytest

import synth
from harness import Pair, logits_close

pytestmark = pytest.mark.gpu


# rows 1, 4, 5, 8, 9 and 96; hidden 64 / 520 / 320 (columns below, just past and between chunks of 512);
# ffn 72 / 1032; contexts around tiles of 256 keys
@pytest.mark.parametrize("name,over,B,k,lens,bias", [
    ("mini32", dict(hidden=64, n_heads=1, n_kv_heads=1, ffn=72, vocab=9), 1, 0, [5], False),
    ("mini32", dict(), 2, 1, [0, 255], True),
    ("mini32", dict(n_kv_heads=1), 1, 4, [256], False),
    ("mini32", dict(hidden=520, ffn=1032, vocab=1003), 4, 1, [1, 31, 257, 600], False),
    ("mini32", dict(head_dim=128, n_heads=4, n_kv_heads=2), 3, 2, [7, 300, 64], False),
    ("mini", dict(), 6, 15, [0, 1, 254, 256, 258, 513], True),
])
def test_plain_draft_step_matches_oracle(name, over, B, k, lens, bias):
    s = synth.CONFIGS[name].with_(k_masks=k, **over)
    p = Pair(s, B, with_bias=bias, lens=lens, flags=2)      # 2: these kernels for bf16 models too
    got = p.gpu_step(top_n=2)
    for b in range(B):
        want = p.oracle_step(b)
        assert logits_close(got["logits"][b], want["logits"], s.dtype) <= 1.0, b     # the logits gate
        assert logits_close(got["feat"][b], want["feat"], s.dtype) <= 1.0, b
    assert np.isfinite(got["logits"]).all() and p.g.check_guards() == 0


# feature and logit rows one float off a 16-byte boundary: fp32, bf16 on these kernels, the chained
# launches, CTA pairs (H and vocab multiples of 4, so that every row is off)
@pytest.mark.parametrize("name,B,flags", [("mini32", 2, 0), ("mini", 2, 2), ("mini", 2, 0), ("mini", 6, 0), ("mini", 2, 4)])
def test_outputs_at_any_address(name, B, flags):
    import torch
    s = synth.CONFIGS[name]
    p = Pair(s, B, lens=[9 + 7 * b for b in range(B)], flags=flags)
    want = p.gpu_step(top_n=2)
    R, V, H = s.rows, s.vocab, s.hidden
    out = {"top_ids": torch.empty((B, R, 2), dtype=torch.int32, device="cuda"), "top_logit": torch.empty((B, R, 2), device="cuda"),
           "row_max": torch.empty((B, R), device="cuda"), "row_lse": torch.empty((B, R), device="cuda"),
           "logits": torch.empty(B * R * V + 1, device="cuda")[1:].view(B, R, V),
           "feat": torch.empty(B * R * H + 1, device="cuda")[1:].view(B, R, H)}
    p.g.draft_step(list(range(B)), p.to_device(p.hidden_last), p.to_device(p.token_last), top_n=2, out=out)
    assert p.g.poll() == 0
    for k in ("logits", "feat", "top_ids"):
        assert np.array_equal(out[k].cpu().numpy(), want[k]), k
