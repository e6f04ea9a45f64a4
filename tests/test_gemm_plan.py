"""How GEMMs of more than 16 rows are dealt to the CTA pairs: host code, no GPU."""
import ctypes as C
import time

import pytest

from paper_2410_05589_b200.binding import load_library

SLOTS = 24 << 20
P = 148 // 2


def plan(rows, k, mats, zip_=0, planes=2, raw=0, slots=SLOTS, n_sm=148):
    out = (C.c_int * 12)()
    rc = load_library().ps_debug_gemm_plan(rows, k, len(mats), (C.c_int * len(mats))(*mats), zip_, planes, raw, slots, n_sm, out)
    assert rc == 0, (rows, k, mats, rc)
    keys = "wt Np row_tiles KB T whole shared split pairs most contributors slots"
    return dict(zip(keys.split(), out))


def stages(H, nq, nkv, F, V):
    return [dict(k=2 * H, mats=[H], planes=1, raw=1), dict(k=H, mats=[nq * 128, nkv * 128, nkv * 128]),
            dict(k=nq * 128, mats=[H], raw=1), dict(k=H, mats=[F, F], zip_=1), dict(k=F, mats=[H], raw=1),
            dict(k=H, mats=[V])]


MODELS = {"7b": stages(4096, 32, 32, 11008, 32000), "13b": stages(5120, 40, 40, 13824, 32000),
          "llama3_8b": stages(4096, 32, 8, 14336, 128256), "mini": stages(768, 6, 6, 2072, 5000)}


@pytest.mark.parametrize("model", sorted(MODELS))
def test_every_row_count_has_a_plan_that_covers_its_tiles(model):
    for rows in list(range(17, 130, 7)) + [160, 255, 256, 257, 288, 576, 640, 903, 1152, 2048]:
        for st in MODELS[model]:
            p = plan(rows, **st)
            assert p["Np"] * p["row_tiles"] >= rows and p["Np"] % 32 == 0 and p["Np"] <= 256
            assert p["whole"] % P == 0 and p["whole"] + p["shared"] == p["T"]
            if not p["shared"]:
                continue
            # the runs of blocks, by their definition
            S = p["shared"] * p["split"]
            edges = [S * c // p["pairs"] for c in range(p["pairs"] + 1)]
            tiles = [set(x // p["split"] for x in range(a, b)) for a, b in zip(edges, edges[1:])]
            per_tile = [sum(t in r for r in tiles) for t in range(p["shared"])]
            assert all(tiles) and max(per_tile) == p["most"] and sum(per_tile) == p["contributors"]
            assert p["slots"] * p["Np"] * 256 * p["wt"] <= SLOTS


def test_last_wave_of_a_long_append_keeps_the_pairs_busy():
    """fc of 2048 rows, 13B shape: 80 tiles on 74 pairs.  With slots for two contributors of every tile the six
    tiles of the last wave could be cut in two only, and 62 pairs waited for them: 72% of the pairs' time."""
    cap = (2048 + 256) * 5120 + 96 * 512 * 256
    p = plan(2048, 10240, [5120], planes=1, raw=1, slots=cap)
    whole = p["whole"] // P * p["KB"]
    blocks = -(-p["shared"] * p["split"] // p["pairs"])
    most = whole + blocks * -(-p["KB"] // p["split"])
    assert p["T"] * p["KB"] / (P * most) > 0.9, p


@pytest.mark.parametrize("rows", [17, 160, 257, 1000, 2048])
def test_row_norm_finds_the_slots_of_the_widest_rows(rows):
    """Contributors in 6 bits, the first slot's place in vectors in the other 26."""
    for k, planes in ((65536, 1), (32768, 2), (98304, 2)):
        p = plan(rows, k, [32768], planes=planes, raw=1, slots=1 << 30)
        assert 0 < p["most"] < 64 and p["slots"] * p["Np"] * 256 * p["wt"] // 4 < 1 << 26, p


def pass_rows(hidden, kv_heads, total, most=2048, n_sm=148):
    from paper_2410_05589_b200.binding import ps_config
    cfg = ps_config(1, hidden, kv_heads, kv_heads, 128, 2 * hidden, 1000, 4, 1, 1024, 1e4, 1e-5, 0)
    return load_library().ps_debug_append_pass_rows(C.byref(cfg), n_sm, total, most)


def test_passes_of_an_append():
    """13B: 1792 rows leave fc 70 tiles and k | v 140 on 74 pairs, 2048 rows 80 and 160; the others have no better pass
    than the largest, nor has an append that one pass takes or that gains less than 4%."""
    assert pass_rows(5120, 40, 4999) == pass_rows(5120, 40, 2304) == pass_rows(5120, 40, 2049) == 1792
    assert pass_rows(5120, 40, 528, most=520) == 512
    for total in (2049, 3000, 4999, 8000):
        assert pass_rows(4096, 32, total) == pass_rows(6656, 52, total) == pass_rows(4096, 8, total) == 2048
    assert pass_rows(5120, 40, 1792) == pass_rows(5120, 40, 3900) == 2048
    for total in (1, 16, 255, 256):
        assert pass_rows(5120, 40, total) == 2048 and pass_rows(5120, 40, total, most=128) == 128
    for most in (128, 256, 300, 1000, 2048):
        for total in range(1, 9000, 97):
            for hidden, kv, n_sm in ((5120, 40, 148), (768, 6, 148), (8192, 8, 148), (5120, 40, 132), (4096, 32, 2)):
                rows = pass_rows(hidden, kv, total, most, n_sm)
                assert rows == most or (0 < rows < most and rows % 256 == 0), (most, total, hidden, n_sm)
    from paper_2410_05589_b200.binding import load_library as lib
    assert lib().ps_debug_append_pass_rows(None, 148, 100, 100) == 0


def test_workspace_beside_the_caches():
    """Scratch of a context, in MB beside its K/V slabs (13B: 123, 311 and 794 with the earlier slots;
    the bounds: as it is, and 2%)."""
    from paper_2410_05589_b200.binding import ps_config
    lib = load_library()
    for shape, B, ctx, k, most in (((5120, 40, 40, 13824, 32000), 1, 1029, 4, 118), ((5120, 40, 40, 13824, 32000), 4, 2100, 4, 235),
                                   ((5120, 40, 40, 13824, 32000), 64, 2100, 8, 690), ((4096, 32, 8, 14336, 128256), 1, 1100, 4, 110)):
        H, nh, nkv, F, V = shape
        cfg = ps_config(1, H, nh, nkv, 128, F, V, k, B, ctx, 1e4, 1e-5, 0)
        n = lib.ps_workspace_bytes(C.byref(cfg)) - 2 * B * nkv * ctx * 128 * 2
        assert 0 < n <= most * 1e6, (shape, B, n)


def test_planning_a_step_is_quick():
    """A server whose row count changes plans anew: 110 us a step when contributors were counted tile by tile.  (Without
    plan()'s own dictionaries, which were half of what was timed.)"""
    call, out = load_library().ps_debug_gemm_plan, (C.c_int * 12)()
    args = [(st["k"], len(st["mats"]), (C.c_int * len(st["mats"]))(*st["mats"]), st.get("zip_", 0), st.get("planes", 2),
             st.get("raw", 0), SLOTS, 148, out) for st in MODELS["13b"]]
    best = 1e9
    for _ in range(5):
        t0 = time.perf_counter()
        for rows in range(20, 660, 20):
            for a in args:
                call(rows, *a)
        best = min(best, (time.perf_counter() - t0) / 32)
    assert best < 80e-6, best
