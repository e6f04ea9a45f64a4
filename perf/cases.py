"""The calls that a program serving a ParallelSpec drafter makes, at the sizes it makes them.

A serving loop drafts and verifies once per round (``draft_step`` / ``draft_step_sampled``, then
``verify`` or ``build_tree`` + ``verify_tree``), appends the positions the target accepted to the
drafter's cache (``kv_append``), fills the cache from a prompt with the same call when a request
arrives, and may hand whole rounds over from host memory (``round_host``).  The training side runs
``group_forward``.  Every case below is one of these, on the model shapes that the repository's
configurations name; ``draw`` gives others of the same ranges.

A case is a dict of plain values:

  call         "round" | "tree" | "host" | "append" | "group"
  model        a key of MODELS
  batch        sequences of the call ("group": 1)
  k            [MASK] positions of a draft step (k + 1 rows per sequence)
  ctx_lo/hi    range of the cached context lengths, ragged over the sequences
  temperature  0: arg-max drafts and greedy verify; above: drafts drawn from q in the LM head
  top_n        candidates per row that the draft step returns
  logits       the draft step keeps its logits and verify uses them as q ("round")
  bonus        the target also scored the position after the last draft ("round")
  new_lo/hi    "append": range of new positions per sequence; "group": number of groups
"""
from __future__ import annotations

import math
import random

import torch

import paper_2410_05589_b200 as ps

# dtype, hidden, heads, kv heads, head dim, ffn, vocab, rope base
MODELS = {
    "tiny": ("f32", 256, 4, 4, 64, 688, 1000, 1e4),
    "mini32": ("f32", 320, 5, 5, 64, 872, 1500, 1e4),
    "mini": ("bf16", 768, 6, 6, 128, 2072, 5000, 1e4),
    "7b": ("bf16", 4096, 32, 32, 128, 11008, 32000, 1e4),
    "13b": ("bf16", 5120, 40, 40, 128, 13824, 32000, 1e4),
    "33b": ("bf16", 6656, 52, 52, 128, 17920, 32000, 1e4),
    "llama3_8b": ("bf16", 4096, 32, 8, 128, 14336, 128256, 5e5),
}

# 23 nodes: the 26-node tree of the benchmark cut to the five depths that k = 4 masks draft.
TREE = (-1, -1, -1, -1, 0, 0, 0, 1, 1, 2, 4, 4, 5, 7, 10, 10, 11, 12, 13, 14, 14, 16, 18)
RANK = tuple(sum(1 for j in range(i) if TREE[j] == TREE[i]) for i in range(len(TREE)))


def _case(name, call, model, batch, k, ctx_lo, ctx_hi, temperature=1.0, top_n=1, logits=True, bonus=False,
          new_lo=0, new_hi=0):
    return {"name": name, "call": call, "model": model, "batch": batch, "k": k, "ctx_lo": ctx_lo, "ctx_hi": ctx_hi,
            "temperature": temperature, "top_n": top_n, "logits": logits, "bonus": bonus, "new_lo": new_lo,
            "new_hi": new_hi}


def listed():
    return [
        # the smallest call: a toy drafter in fp32, as one debugs an integration with; launches and latency only
        _case("tiny_fp32_round", "round", "tiny", 1, 4, 64, 64),
        # a chat at temperature 0 on a 7B target: arg-max drafts, logits never leave the LM head
        _case("7b_greedy_b1", "round", "7b", 1, 4, 512, 512, temperature=0.0, logits=False),
        # the single-stream case that the benchmark quotes: lossless sampling on a 13B target
        _case("13b_sampled_b1", "round", "13b", 1, 4, 1024, 1024),
        # the same round for a caller whose target runs elsewhere: everything comes from and returns to host memory
        _case("13b_host_b1", "host", "13b", 1, 4, 1024, 1024),
        # grouped-query target with a 128k vocabulary, token tree drafted and verified
        _case("llama3_8b_tree_b1", "tree", "llama3_8b", 1, 4, 1024, 1024, top_n=4),
        # a handful of concurrent users, ragged contexts; the target scored the bonus position too
        _case("13b_sampled_b4", "round", "13b", 4, 4, 256, 2048, bonus=True),
        # a small server's batch
        _case("13b_sampled_b16", "round", "13b", 16, 4, 256, 2048),
        # a large target with long contexts and more masks; candidates for the caller's own tree
        _case("33b_sampled_b16", "round", "33b", 16, 8, 1024, 4096, top_n=8),
        # a full batch: 576 rows
        _case("13b_sampled_b64", "round", "13b", 64, 8, 256, 2048),
        # after a round: the accepted positions of four sequences enter their caches
        _case("13b_append_b4", "append", "13b", 4, 4, 0, 0, new_lo=1, new_hi=5),
        # four prompts arrive: the caches are filled
        _case("13b_prefill_b4", "append", "13b", 4, 4, 0, 0, new_lo=256, new_hi=2048),
        # training layout: 128 consecutive positions of a text, each heading a group of masks
        _case("13b_group_128", "group", "13b", 1, 4, 300, 300, logits=True, new_lo=128, new_hi=128),
    ]


def draw(rng):
    """One more case: any model, batch and contexts over the whole range, odd sizes included, never
    more work than the largest listed case."""
    largest = [work(c) for c in listed()]
    most = {"bytes": max(w["bytes"] for w in largest), "flops": max(w["flops"] for w in largest)}

    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))

    while True:
        call = rng.choice(("round",) * 5 + ("tree", "host", "append", "append", "group"))
        model = rng.choice(("13b", "13b", "7b", "33b", "llama3_8b", "mini", "tiny", "mini32"))
        small = MODELS[model][0] == "f32"
        k = rng.randint(1, 8) if call != "tree" else 4
        batch = 1 if call == "group" else log_int(1, 8 if small else 64)
        lo = log_int(16, 256 if small else 2048)
        hi = min(2 * lo + rng.randint(0, lo), 512 if small else 4096)
        c = _case("", call, model, batch, k, lo, hi, temperature=rng.choice((0.0, 0.7, 1.0, 1.0)))
        c["top_n"] = rng.choice((1, 1, 4, 8)) if call == "round" and c["temperature"] > 0 else 1
        if call == "round":
            c["logits"] = c["temperature"] > 0
            c["bonus"] = rng.random() < 0.5
        elif call == "tree":
            c["top_n"] = rng.choice((4, 8))
        elif call == "append":
            c["ctx_lo"] = c["ctx_hi"] = 0
            if rng.random() < 0.5:
                c["new_lo"], c["new_hi"] = 1, k + 1
            else:
                c["new_lo"] = log_int(8, 512)
                c["new_hi"] = min(3 * c["new_lo"], 100 if small else 2048)
                c["batch"] = min(batch, 8)
        elif call == "group":
            c["new_lo"] = c["new_hi"] = log_int(2, 24 if small else 160)
            c["ctx_hi"] = c["ctx_lo"]
        del c["name"]
        w = work(c)
        if w["bytes"] <= most["bytes"] and w["flops"] <= most["flops"]:
            return c


def _ragged(case, lo, hi, n):
    """n lengths over [lo, hi], the same for every seed: a case's work does not depend on its inputs."""
    r = random.Random("%s %d %d %d" % (case["model"], lo, hi, n))
    return [r.randint(lo, hi) for _ in range(n)]


def _weights(model, k, gen):
    dt, H, nh, nkv, d, F, V, _ = MODELS[model]
    dtype = torch.float32 if dt == "f32" else torch.bfloat16

    def normal(shape, mean=0.0):
        return torch.randn(shape, generator=gen, device="cuda", dtype=dtype).mul_(0.02).add_(mean)

    shapes = dict(embed=(V, H), mask_embed=(k, H), mask_feat=(k, H), w_fc=(H, 2 * H), w_q=(nh * d, H), w_k=(nkv * d, H),
                  w_v=(nkv * d, H), w_o=(H, nh * d), w_gate=(F, H), w_up=(F, H), w_down=(H, F), w_lm=(V, H))
    w = {n: normal(s) for n, s in shapes.items()}
    for n in ("g_in", "g_post", "g_final"):
        w[n] = normal((H,), 1.0)
    return w


def _target_logits(gen, batch, rows, vocab):
    """N(0, 1) plus a Zipf(1.1) rank bias, ranks permuted per row: a few tokens dominate."""
    z = torch.randn((batch, rows, vocab), generator=gen, device="cuda")
    bias = torch.arange(1, vocab + 1, device="cuda", dtype=torch.float64).log_().mul_(-1.1).float()
    rank = torch.rand((batch, rows, vocab), generator=gen, device="cuda").argsort(-1)
    return z.add_(bias[rank])


class State:
    """What a serving program holds between calls: the drafter with its caches, the call's inputs and
    the output buffers that it reuses."""


def prepare(case, seed):
    dt, H, nh, nkv, d, F, V, base = MODELS[case["model"]]
    B, k, R = case["batch"], case["k"], case["k"] + 1
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.float32 if dt == "f32" else torch.bfloat16
    st = State()
    st.case, st.seed = case, seed
    call = case["call"]
    lens = _ragged(case, case["ctx_lo"], case["ctx_hi"], B)
    n_new = _ragged(case, case["new_lo"], case["new_hi"], B) if call in ("append", "group") else [0]
    rows = sum(n_new) if call in ("append", "group") else B
    st.d = ps.Drafter(dtype=ps.PS_DTYPE_F32 if dt == "f32" else ps.PS_DTYPE_BF16, hidden=H, n_heads=nh, n_kv_heads=nkv,
                      head_dim=d, ffn=F, vocab=V, k_masks=k, max_batch=min(128, n_new[0]) if call == "group" else B,
                      max_ctx=max(lens) + max(n_new) + R, weights=_weights(case["model"], k, gen), rope_base=base)
    for b in range(B):
        if lens[b] > 0:
            kv = torch.randn((2, lens[b], nkv * d), generator=gen, device="cuda", dtype=dtype)
            st.d.kv_import(b, kv[0], kv[1])
    st.slots = list(range(B))
    st.n_new = n_new
    # target features (last hidden states) and tokens of the positions that the call starts from
    st.hidden = torch.randn((rows, H), generator=gen, device="cuda", dtype=dtype).mul_(0.02 if dt == "f32" else 1.0)
    st.tokens = torch.randint(0, V, (rows,), generator=gen, device="cuda", dtype=torch.int32)
    st.draft, st.verify = {}, {}
    if call == "round":
        st.target = _target_logits(gen, B, R + (1 if case["bonus"] else 0), V)
    elif call == "tree":
        st.target = _target_logits(gen, B, len(TREE) + 1, V)
        st.tree_tokens = torch.empty((B, len(TREE)), dtype=torch.int32, device="cuda")
    elif call == "host":
        st.target = _target_logits(gen, B, R, V).cpu().pin_memory()
        st.hidden, st.tokens = st.hidden.cpu().pin_memory(), st.tokens.cpu().pin_memory()
    return st


def run(st):
    c, d, T = st.case, st.d, st.case["temperature"]
    if c["call"] == "round":
        if T > 0:
            o = d.draft_step_sampled(st.slots, st.hidden, st.tokens, T, st.seed, 7, top_n=c["top_n"],
                                     want_logits=c["logits"], out=st.draft)
            drafts = o["sampled"]
        else:
            o = d.draft_step(st.slots, st.hidden, st.tokens, top_n=1, want_logits=c["logits"], out=st.draft)
            drafts = o["top_ids"][:, :, 0]
        return [o, d.verify(drafts, o["logits"], st.target, T, st.seed, 7, out=st.verify)]
    if c["call"] == "tree":
        o = d.draft_step(st.slots, st.hidden, st.tokens, top_n=c["top_n"], want_logits=True, out=st.draft)
        d.build_tree(TREE, RANK, o["top_ids"], out=st.tree_tokens)
        return [o, st.tree_tokens,
                d.verify_tree(TREE, st.tree_tokens, o["logits"], st.target, T, st.seed, 7, out=st.verify)]
    if c["call"] == "host":
        return d.round_host(st.slots, st.hidden, st.tokens, st.target, T, st.seed, 7, out=st.verify)
    if c["call"] == "append":
        for b in st.slots:
            d.kv_reset(b)
        d.kv_append(st.slots, st.n_new, st.hidden, st.tokens)
        return [d.kv_export(b) for b in st.slots]   # the state that the call updated
    return d.group_forward(0, st.hidden, st.tokens, top_n=1, want_logits=True, want_feat=True)


def work(case):
    dt, H, nh, nkv, d, F, V, _ = MODELS[case["model"]]
    B, R, e = case["batch"], case["k"] + 1, 4 if dt == "f32" else 2
    Hq, Hkv, call = nh * d, nkv * d, case["call"]
    new = sum(_ragged(case, case["new_lo"], case["new_hi"], B)) if call in ("append", "group") else 0
    if call == "append":   # fc and k | v of every new position; the rows exported again
        params = 2 * H * H + 2 * H * Hkv
        return {"bytes": e * (params + 2 * new * H + 3 * new * 2 * Hkv), "flops": 2.0 * params * new}
    M = (new if call == "group" else B) * R
    params = 2 * H * H + H * (Hq + 2 * Hkv) + Hq * H + 3 * H * F + V * H
    if call == "group":    # the context once, every group's own view of it in the products
        ctx, seen = case["ctx_lo"] + new, sum(case["ctx_lo"] + t for t in range(new))
    else:
        ctx = seen = sum(_ragged(case, case["ctx_lo"], case["ctx_hi"], B))
    nbytes = e * (params + 2 * Hkv * ctx + 2 * M * H)
    if call == "group":
        nbytes += 4 * M * (V + H)
    elif call == "tree":
        nbytes += 4 * V * (2 * M + B * (len(TREE) + 1))
    else:
        target_rows = B * (R + (1 if case["bonus"] else 0))
        nbytes += 4 * V * (target_rows + (2 * M if case["logits"] else 0))
    flops = 2.0 * params * M + 4.0 * Hq * R * seen
    if call == "group":
        flops += 2.0 * new * 2 * H * Hkv
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Four times what was measured on the listed cases.  fp32: the logits are 2.3e-7 (2-norm) and
    9.1e-7 (largest) from the same arithmetic in 64 bits.  bf16: new k / v rows are rounded to the
    cache's type, so sums in another order move single entries by one unit in the last place
    (the exported rows of two sets of kernels differ by 1.8e-4, at most 7.8e-3), and the logits
    are up to 2e-4 / 4.8e-3 from 64 bits, 3.5e-4 / 5.5e-3 where the context itself was appended.
    Whole values: of ranked candidates 5e-3 changed places (neighbours in a list of eight)."""
    if MODELS[case["model"]][0] == "f32":
        return {"rel": 2e-6, "max": 1e-5, "differ": 0.01}
    if case["call"] == "append":
        return {"rel": 8e-4, "max": 1.6e-2, "differ": 0.01}
    return {"rel": 1.4e-3, "max": 2e-2, "differ": 0.01}
