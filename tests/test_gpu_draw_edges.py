"""Draws whose sampling point falls on the edge between two holders of weight, where sums of
doubles round: the token drawn has weight (needs a B200)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# Weights of 1 / parts in every part of the row, a part being what a warp (V = 2048, one block) or a block (V =
# 32768, eight of them) holds, plus some units in the last place of 1 / parts.  A scan over the parts rounds
# (part 0 + part 1) up, so that its difference from part 1 lies above part 0; the last part makes the total such
# that u2 x total is part 0 exactly, with the seed for which u2 = 1 / parts.
WARPS = dict(V=2048, parts=16, own=4, first=3, last=45, seed=45330390)
BLOCKS = dict(V=32768, parts=8, own=8, first=3, last=20, seed=9544493)


def _scan(sums):
    """The running sums of a shuffle scan, lane by lane, in doubles."""
    x = np.array(sums, np.float64)
    o = 1
    while o < len(x):
        x[o:] = x[o:] + x[:-o]
        o *= 2
    return x


def _row(V, parts, own, first, last, **_):
    row = np.full(V, -200.0, np.float32)            # no weight
    at = [p * (V // parts) + 5 * own for p in range(parts)]
    row[at] = 0.0
    unit = np.float32(-52 * np.log(2.0))            # exp() of it: one unit in the last place of 1
    row[[at[0] + 1 + e for e in range(first)]] = unit
    row[at[-1] + 1] = unit + np.float32(np.log(float(last)))
    return row, at


@pytest.mark.parametrize("case", [WARPS, BLOCKS], ids=["warps", "blocks"])
@pytest.mark.parametrize("walk", ["tree", "chain"])
def test_token_on_an_edge_has_weight(case, walk):
    import torch
    import paper_2410_05589_b200 as ps
    V, parts = case["V"], case["parts"]
    row, at = _row(**case)
    # what the case rests on, in the arithmetic of the kernels (a thread adds its tokens one after another)
    assert oracle.uniforms(case["seed"], 0, 0, 1)[1] == 1.0 / parts
    w = np.exp(row.astype(np.float64)).astype(np.float32) / np.float32(parts)
    sums = []
    for p in range(parts):
        s = np.float64(0)
        for v in range(at[p], at[p] + 4):
            s += np.float64(w[v])
        sums.append(s)
    run = _scan(sums)
    assert run[1] - sums[1] > run[0] and run[-1] / parts == run[0]
    s = synth.CONFIGS["mini32"].with_(hidden=64, n_heads=1, n_kv_heads=1, ffn=64, vocab=V, k_masks=0)
    g = ps.drafter_from_shape(s, synth.weights(s), max_batch=1, max_ctx=8)
    first = synth.gauss_logits(1, "edge", (1, 1, V))
    target = ps.to_device(np.concatenate([first, row[None, None]], 1))
    draft, tok = ps.to_device(first), torch.zeros((1, 1), dtype=torch.int32, device="cuda")
    if walk == "tree":
        out = g.verify_tree([-1], tok, draft, target, 1.0, case["seed"], 0)
    else:
        out = g.verify(tok, draft, target, 1.0, case["seed"], 0)
    got = int(out["out_tokens"][0, 1])
    assert int(out["n_out"][0]) == 2                # (p = q at the first row: always accepted)
    assert got in (at[0] + case["first"], at[1]), got   # the last holder of part 0, the first of part 1
    assert g.poll() == 0
