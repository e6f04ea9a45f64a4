"""Cache import / export: 16-byte vectors and, where the caller's arrays are not aligned, single
elements; lengths around a block, grouped heads, both storage types (needs a B200)."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,kv_heads", [("mini", 6), ("mini", 3), ("mini32", 5)])
@pytest.mark.parametrize("aligned", [True, False])
def test_import_export_round_trip(name, kv_heads, aligned):
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS[name].with_(n_kv_heads=kv_heads, vocab=64, ffn=64)
    d = ps.drafter_from_shape(s, synth.weights(s), max_batch=3, max_ctx=300)
    width, held = kv_heads * s.head_dim, {}
    for slot, n in ((0, 1), (1, 299), (2, 37)):
        flat = torch.randn(2, n * width + 1, device="cuda").to(d.torch_dtype)
        K, V = (flat[i].clone()[0 if aligned else 1:][:n * width].view(n, width) for i in (0, 1))
        assert (K.data_ptr() % 16 == 0) == aligned
        d.kv_import(slot, K, V)
        held[slot] = K, V
    for slot, (K, V) in held.items():
        out = torch.empty((2, K.numel() + 1), dtype=K.dtype, device="cuda")
        Ko, Vo = (out[i].clone()[0 if aligned else 1:][:K.numel()].view_as(K) for i in (0, 1))
        rc = d.lib.ps_kv_export(d.h, slot, Ko.data_ptr(), Vo.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == 0 and torch.equal(Ko, K) and torch.equal(Vo, V)
    assert d.check_guards() == 0


def test_copy_of_more_rows_than_one_launch_indexes():
    import paper_2410_05589_b200 as ps
    s = synth.CONFIGS["mini"].with_(vocab=64, ffn=64)
    width = s.n_kv_heads * s.head_dim
    n = (1 << 30) // width + 5                        # single elements, more than 2^30 of them
    d = ps.drafter_from_shape(s, synth.weights(s), max_batch=1, max_ctx=n + s.rows)
    flat = torch.empty(n * width + 1, dtype=torch.bfloat16, device="cuda").uniform_(-1, 1)
    K = flat[1:].view(n, width)
    d.kv_import(0, K, K)
    Ko, Vo = d.kv_export(0)                           # aligned: vectors, one launch
    assert torch.equal(Ko, K) and torch.equal(Vo, K)
