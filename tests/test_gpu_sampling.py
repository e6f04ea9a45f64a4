"""Parity of ps_draft_step_sampled (draft sampling fused in the LM head) with the CPU oracle
(needs a B200).

  * the sampled token of every row equals the arg-max of (the kernel's own logits / T + the
    oracle's Gumbel noise), unless two perturbed values are closer than fp32 rounding allows;
  * it equals the oracle's sample from the ORACLE's logits unless the runner-up is within the
    logits tolerance of the winner;
  * over many offsets the tokens follow softmax(logits / T) (chi-square on bins of equal mass);
  * sampled drafts + ps_verify accept a draft with probability sum_v min(p_v, q_v) (Eq. 1).
"""
import numpy as np
import pytest
import torch
from scipy import stats

import oracle
import synth
from harness import Pair

pytestmark = pytest.mark.gpu


def _gumbel(V, seed, offset, row_id):
    key = [(seed & 0xFFFFFFFF) ^ 0x6D756247, seed >> 32]
    g = np.empty(V)
    for v in range(V):
        w = oracle.philox4x32(key, [v, row_id, offset & 0xFFFFFFFF, offset >> 32])
        u = ((int(w[0]) >> 8) + 0.5) / 2 ** 24
        g[v] = -np.log(-np.log(u))
    return g


def _check_rows(s, got, want_logits_of, T, seed, offset, B):
    R = s.rows
    for b in range(B):
        want = want_logits_of(b)
        for j in range(R):
            row_id = b | (j << 8)
            tok = int(got["sampled"][b, j])
            assert 0 <= tok < s.vocab
            # (1) consistent with the kernel's own logits
            if got["logits"] is not None and s.vocab <= 5000:
                y = got["logits"][b, j].astype(np.float64) / T + _gumbel(s.vocab, seed, offset, row_id)
                assert y[tok] >= y.max() - 1e-4 * max(1.0, abs(y.max())), (b, j)
            # (2) the oracle's sample from the oracle's logits, up to the logits tolerance
            t_o, margin = oracle.gumbel_sample(want["logits"][j][None], T, seed, offset, np.array([row_id], np.int32))
            if tok != int(t_o[0]):
                wl = want["logits"][j]
                tol = (1e-4 * max(abs(wl).max(), 1.0) if s.dtype == 0 else 1e-2 + 2e-2 * abs(wl).max()) / T
                assert margin[0] <= 2 * tol, (b, j, tok, int(t_o[0]), margin[0])


@pytest.mark.parametrize("name,B,flags", [("mini", 3, 0), ("tiny", 1, 0), ("mini", 1, 0), ("mini", 3, 4), ("mini", 2, 2), ("mini", 3, 16)])
def test_sampled_tokens_match_oracle(name, B, flags):
    """flags 16: one launch per GEMM stage instead of the chained stages; flags 4 / 2: the
    mma.sync GEMMs and the plain kernels, where one block per row draws the token from the
    stored logits."""
    s = synth.CONFIGS[name]
    p = Pair(s, B, flags=flags)
    T, seed, offset = 0.8, 5, 12
    out = p.g.draft_step_sampled(list(range(B)), p.to_device(p.hidden_last), p.to_device(p.token_last),
                                 T, seed, offset, top_n=1)
    torch.cuda.synchronize()
    got = {k: (v.cpu().numpy() if v is not None else None) for k, v in out.items()}
    _check_rows(s, got, p.oracle_step, T, seed, offset, B)
    # the other outputs are those of ps_draft_step
    ref = p.gpu_step(top_n=1)
    assert np.array_equal(ref["logits"], got["logits"]) and np.array_equal(ref["top_ids"], got["top_ids"])
    assert p.g.poll() == 0


def test_sampled_tokens_of_a_batch_beyond_one_launch():
    """28 sequences x 5 rows exceed one tensor-core launch: the groups the batch is cut into
    keep each sequence's own counter (its index in the caller's batch)."""
    s = synth.CONFIGS["mini"]
    B = 28
    p = Pair(s, B, lens=[7 + 3 * b for b in range(B)])
    T, seed, offset = 1.0, 11, 3
    out = p.g.draft_step_sampled(list(range(B)), p.to_device(p.hidden_last), p.to_device(p.token_last),
                                 T, seed, offset, top_n=1)
    torch.cuda.synchronize()
    got = {k: (v.cpu().numpy() if v is not None else None) for k, v in out.items()}
    _check_rows(s, got, p.oracle_step, T, seed, offset, B)
    assert p.g.poll() == 0


def test_sampled_tokens_follow_softmax_and_verify_accepts_at_the_closed_form_rate():
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"]
    p = Pair(s, 1, lens=[40])
    T, n = 1.0, 3000
    hl, tl = p.to_device(p.hidden_last), p.to_device(p.token_last)
    out = {}
    picks = np.empty((n, s.rows), np.int64)
    for off in range(n):
        p.g.draft_step_sampled([0], hl, tl, T, 9, off, top_n=1, out=out)
        picks[off] = out["sampled"][0].cpu().numpy()
    logits = out["logits"][0].cpu().numpy().astype(np.float64)
    for j in (0, s.rows - 1):
        z = logits[j] / T
        q = np.exp(z - z.max())
        q /= q.sum()
        order = np.argsort(-q)
        edges = np.searchsorted(np.cumsum(q[order]), np.linspace(0, 1, 13)[1:-1])   # 12 bins of equal mass
        bin_of = np.empty(s.vocab, np.int64)
        bin_of[order] = np.searchsorted(edges, np.arange(s.vocab), side="right")
        exp = np.bincount(bin_of, weights=q, minlength=12) * n
        obs = np.bincount(bin_of[picks[:, j]], minlength=12)
        assert stats.chisquare(obs, exp).pvalue > 1e-3, j
    # Eq. 1 end to end: drafts sampled on the device, verified against a shifted target
    tgt = (logits[None, :, :] * 0.7 + synth.gauss_logits(3, "e2e", (1, s.rows, s.vocab)) * 0.5).astype(np.float32)
    d_tgt = ps.to_device(tgt)
    acc0 = 0
    for off in range(n):
        p.g.draft_step_sampled([0], hl, tl, T, 9, off, top_n=1, out=out)
        v = p.g.verify(out["sampled"], out["logits"], d_tgt, T, seed=2, offset=off)
        acc0 += int(v["accept_len"][0].item() >= 1)
    pt = np.exp(tgt[0, 0].astype(np.float64) - tgt[0, 0].max())
    pt /= pt.sum()
    z = logits[0] / T
    q = np.exp(z - z.max())
    q /= q.sum()
    want = np.minimum(pt, q).sum()
    assert abs(acc0 / n - want) < 5 * np.sqrt(want * (1 - want) / n)


def test_sampling_argument_errors():
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"]
    p = Pair(s, 1, lens=[10])
    with pytest.raises(ps.PsError):
        p.g.draft_step_sampled([0], p.to_device(p.hidden_last), p.to_device(p.token_last), 0.0, 1, 0)


@pytest.mark.parametrize("name", ["mini", "tiny"])
def test_round_host_is_lossless(name):
    """ps_round_host (host buffers in, results out).  At temperature > 0 its drafts are drawn from
    q = softmax(draft logits / T), the only case in which Eq. 1 keeps the target distribution:
    (a) every round equals the oracle's verify applied to the tokens ps_draft_step_sampled draws
    with the same seed and offset, (b) over many offsets the first emitted token follows
    softmax(target row 0) (chi-square on 12 bins of equal mass) although the draft distribution
    differs from it, (c) at temperature 0 the round is the greedy chain."""
    from harness import assert_verify_same
    s = synth.CONFIGS[name]
    p = Pair(s, 1, lens=[33])
    V, R, T, seed = s.vocab, s.rows, 1.0, 21
    hl_d, tl_d = p.to_device(p.hidden_last), p.to_device(p.token_last)
    ref = p.g.draft_step([0], hl_d, tl_d, top_n=1)
    torch.cuda.synchronize()
    logits = ref["logits"].cpu().numpy()
    tgt = synth.noisy_draft_logits(s.seed, "rh", logits, 0.8 * float(logits.std()))
    hl_h = torch.from_numpy(p.hidden_last.view(np.int16) if p.hidden_last.dtype == np.uint16 else p.hidden_last).pin_memory()
    tl_h = torch.from_numpy(p.token_last).pin_memory()
    tgt_h = torch.from_numpy(tgt).pin_memory()
    n = 2400
    first = np.empty(n, np.int64)
    n_acc = 0
    s_out, r_out = {}, {}
    for off in range(n):
        p.g.round_host([0], hl_h, tl_h, tgt_h, T, seed, off, out=r_out)
        first[off] = int(r_out["out_tokens"][0, 0])
        n_acc += int(r_out["accept_len"][0])
        if off < 24:
            o = p.g.draft_step_sampled([0], hl_d, tl_d, T, seed, off, top_n=1, out=s_out)
            torch.cuda.synchronize()
            want = oracle.verify(o["sampled"].cpu().numpy(), o["logits"].cpu().numpy(), tgt, T, seed, off)
            got = {k: r_out[k].numpy().copy() for k in ("accept_len", "out_tokens", "n_out")}
            assert_verify_same(got, want, max_excused=1)
    assert 0 < n_acc < n * R          # acceptances and rejections both happened
    z = tgt[0, 0].astype(np.float64) / T
    pr = np.exp(z - z.max())
    pr /= pr.sum()
    order = np.argsort(-pr)
    edges = np.searchsorted(np.cumsum(pr[order]), np.linspace(0, 1, 13)[1:-1])
    bin_of = np.empty(V, np.int64)
    bin_of[order] = np.searchsorted(edges, np.arange(V), side="right")
    exp = np.bincount(bin_of, weights=pr, minlength=12) * n
    obs = np.bincount(bin_of[first], minlength=12)
    keep = exp > 5
    assert stats.chisquare(obs[keep], exp[keep] * obs[keep].sum() / exp[keep].sum()).pvalue > 1e-3
    # the arg-max drafts of the old behaviour would be accepted too often: the drafter's own
    # distribution q_0 is not the law of the first token unless it equals p_0
    zq = logits[0, 0].astype(np.float64) / T
    q = np.exp(zq - zq.max())
    q /= q.sum()
    exp_q = np.bincount(bin_of, weights=q, minlength=12) * n
    assert stats.chisquare(obs[keep], exp_q[keep] * obs[keep].sum() / exp_q[keep].sum()).pvalue < 1e-3
    # temperature 0: greedy chain of arg-max drafts
    p.g.round_host([0], hl_h, tl_h, tgt_h, 0.0, seed, 0, out=r_out)
    want = oracle.verify(logits.argmax(-1).astype(np.int32), None, tgt, 0.0, seed, 0)
    for k in ("accept_len", "out_tokens", "n_out"):
        assert np.array_equal(r_out[k].numpy(), want[k]), k
    assert p.g.poll() == 0


@pytest.mark.parametrize("k", [0, 4, 5, 6])
@pytest.mark.parametrize("top_n", [0, 1, 2])
def test_kept_logits_on_both_sides_of_the_epilogue_rule(k, top_n):
    """Up to 5 rows (6 with a draw) and one pick take their statistics in the LM head's epilogue, the rest in a
    pass over the stored logits: the same values, ranks and draws from the logits that come back."""
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"].with_(k_masks=k)
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=1, max_ctx=32)
    hl, tl = ps.to_device(synth.hidden_states(s, "last", 1)), ps.to_device(synth.token_ids(s, "last", 1))
    for o in (g.draft_step([0], hl, tl, top_n=top_n), g.draft_step_sampled([0], hl, tl, 0.9, 3, 4, top_n=top_n)):
        torch.cuda.synchronize()
        lg = o["logits"][0].double().cpu().numpy()
        assert np.array_equal(o["row_max"][0].cpu().numpy(), lg.max(-1).astype(np.float32))
        # exponentials to 2^-20 each, fp32 sums over a tree of depth < 20, the stored value's rounding
        lse = lg.max(-1) + np.log(np.exp(lg - lg.max(-1, keepdims=True)).sum(-1))
        assert np.abs(o["row_lse"][0].cpu().numpy() - lse).max() < 2.0 ** -18 + 2.0 ** -23 * np.abs(lse).max()
        if top_n:
            assert np.array_equal(o["top_ids"][0].cpu().numpy(), np.argsort(-lg, axis=-1, kind="stable")[:, :top_n])
        if "sampled" in o:
            ids = np.arange(k + 1, dtype=np.int32) << 8
            tok, margin = oracle.gumbel_sample(lg, 0.9, 3, 4, ids)
            # single-precision noise: 2^-21 of values up to 17
            assert all(a == b or m < 2e-5 for a, b, m in zip(o["sampled"][0].cpu().numpy(), tok, margin))
