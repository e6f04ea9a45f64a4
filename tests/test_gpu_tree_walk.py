"""Two-launch token-tree verification: edges of the vocabulary's shares, leaves without a distribution,
maxima far from the first batch, more rows than are resident at once (needs a B200)."""
import numpy as np
import pytest

import synth
from test_gpu_verify import _ctx
from test_gpu_verify_tree import TREE26, _assert_same, _case, _run_both

pytestmark = pytest.mark.gpu


# vocab 4 / 132: blocks and threads without tokens; 65540: 16-block clusters; B = 40: several waves of rows
@pytest.mark.parametrize("V,B,T", [(4, 3, 1.0), (132, 5, 0.7), (4100, 40, 1.0), (65536, 3, 1.0), (65540, 3, 0.8), (4100, 6, 0.0)])
@pytest.mark.parametrize("odd", [False, True])
def test_tree_walk_edges(V, B, T, odd):
    g = _ctx(V)
    toks, dl, tl = _case(TREE26, B, V, seed=5, T=T)
    if odd:
        tl[0, 0, -1] += 300.0                 # the maximum far above the first batch's
        dl[1, 0, : V // 2] = -np.inf
        tl[2, 1 + 25] = -np.inf               # a leaf without a distribution
        tl[1, 1 + 6, V // 2] = np.inf         # a leaf with +inf
        tl[2, 1 + 0, 1] = np.nan              # an inner row with NaN
    for offset in (3, 4):
        got, want = _run_both(g, TREE26, toks, dl, tl, T, 9, offset)
        _assert_same(got, want)
    assert g.poll() in (0, -6) and g.check_guards() == 0


# the walk's clusters of 1, 2, 4 and 8 blocks (few trees and 14 or more: the fewest that hold a row), leaves
# with statistics of their own and without (B = 1 and 30)
@pytest.mark.parametrize("V", [4096, 4100, 8196, 16388])
@pytest.mark.parametrize("B", [1, 14, 30])
@pytest.mark.parametrize("tree", ["26", "chain"])
def test_tree_walk_cluster_sizes(V, B, tree):
    parent = TREE26 if tree == "26" else [-1, 0, 1, 2]
    g = _ctx(V)
    toks, dl, tl = _case(parent, B, V, seed=7, T=0.8)
    for offset in (1, 2, 3):
        got, want = _run_both(g, parent, toks, dl, tl, 0.8, 4, offset)
        _assert_same(got, want)
    assert g.poll() == 0
