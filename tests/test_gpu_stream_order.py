"""Inputs written by the kernel just ahead of a call, which lets its dependents start before it
writes: every call must find them written (needs a B200)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from harness import assert_verify_same

pytestmark = pytest.mark.gpu


# one block per row pair (vocabulary up to 8192), 8-block clusters, 4-block clusters (16 to 33 row
# pairs), 16-block clusters, the streaming kernel, one block and three passes (odd vocabulary)
@pytest.mark.parametrize("vocab,B,n_draft,bonus", [(1000, 1, 5, 0), (8192, 3, 5, 1), (32000, 1, 5, 0), (32000, 4, 5, 1),
                                                   (16384, 7, 5, 0), (128256, 1, 5, 0), (32000, 16, 4, 1), (1001, 2, 3, 0)])
@pytest.mark.parametrize("T", [0.0, 1.0])
def test_verify_finds_late_target_logits(vocab, B, n_draft, bonus, T):
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini32"].with_(hidden=64, n_heads=1, n_kv_heads=1, ffn=64, vocab=vocab, k_masks=n_draft - 1)
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=B, max_ctx=n_draft + 1)
    tl = synth.zipf_logits(3, (vocab, B), B, n_draft + bonus, vocab)
    dl = synth.noisy_draft_logits(3, (vocab, B), tl[:, :n_draft], 0.4)
    tok = synth.sample_from_logits(3, (vocab, B), dl, 1.0)
    want = oracle.verify(tok, dl, tl, T, 2, 9)
    dtok, ddl, late = ps.to_device(tok), ps.to_device(dl), ps.to_device(tl)
    stale = ps.to_device(np.ascontiguousarray(tl[:, :, ::-1]))
    out = g.verify(dtok, ddl, late, T, 2, 9)     # (module load and the device's answers are out of the way)
    for _ in range(3):
        target = stale.clone()
        torch.cuda.synchronize()
        g.debug_late_copy(target, late, 30)
        g.verify(dtok, ddl, target, T, 2, 9, out=out)
        torch.cuda.synchronize()
        assert_verify_same({k: v.cpu().numpy() for k, v in out.items()}, want)


# a chained step, a step of more than 16 rows, fp32: target features and tokens arrive late
@pytest.mark.parametrize("name,B", [("mini", 2), ("mini", 6), ("tiny", 2)])
def test_draft_step_and_append_find_late_inputs(name, B):
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS[name].with_(batch=B)
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=B, max_ctx=64)
    n = 9
    hid, tok = ps.to_device(synth.hidden_states(s, "ctx", n * B)), ps.to_device(synth.token_ids(s, "ctx", n * B))
    last, tlast = ps.to_device(synth.hidden_states(s, "last", B)), ps.to_device(synth.token_ids(s, "last", B))
    slots = list(range(B))

    def run(late):
        def give(x):
            if not late:
                return x
            y = torch.zeros_like(x)
            torch.cuda.synchronize()
            g.debug_late_copy(y, x, 30)
            return y
        for b in slots:
            g.kv_reset(b)
        h = give(hid)
        g.kv_append(slots, [n] * B, h, tok)
        h2 = give(last)
        o = g.draft_step(slots, h2, tlast, top_n=2)
        t2 = give(tlast)
        o2 = g.draft_step(slots, last, t2, top_n=2)
        torch.cuda.synchronize()
        return [o["logits"].cpu().numpy(), o2["logits"].cpu().numpy()] + [x.float().cpu().numpy() for x in g.kv_export(B - 1)]

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)


# weights written by the kernel just ahead (an optimiser's step): fp32 activations (2: these kernels), chained
# launches, CTA pairs; 8: no fc
@pytest.mark.parametrize("name,B,flags", [("tiny", 1, 0), ("mini", 1, 2), ("mini", 1, 10), ("mini", 1, 0), ("mini", 6, 0),
                                          ("mini", 1, 8), ("mini", 6, 8)])
def test_draft_step_finds_late_weights(name, B, flags):
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS[name].with_(batch=B)
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=B, max_ctx=32, flags=flags)
    hl, tl = ps.to_device(synth.hidden_states(s, "last", B)), ps.to_device(synth.token_ids(s, "last", B))
    slots = list(range(B))
    want = g.draft_step(slots, hl, tl)["logits"].clone()
    for n in ("w_fc", "w_q", "w_o", "w_up", "w_down", "w_lm"):
        if flags & 8 and n == "w_fc":
            continue
        w = g.weights[n]
        true = w.clone()
        w.zero_()
        torch.cuda.synchronize()
        g.debug_late_copy(w, true, 30)
        got = g.draft_step(slots, hl, tl)["logits"]
        torch.cuda.synchronize()
        assert torch.equal(got, want), n
