"""The cluster decode path (clusters of CTAs that share the n axis of a KV head's blocks) at the sizes where its tiling can go
wrong, against the fp64 oracle: block lengths around the 64-column groups and the cluster sizes they give, retained lengths around
the 64-row tiles and beyond 512 (two passes over the weights), units of many sequences and of a few blocks, more units than one wave,
text lengths around a chunk and beyond sixteen of them, per-sequence lengths with nothing in some sequences.

Bound: the regression bound of the parity tests; shapes whose operands are kept as two bf16 terms (16 bits) stay within it by a
wide margin, their error is the rounding of the output.
"""
import random

import pytest
import torch

from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("recipe", ["peaked", "structured"])
@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (1, 1, 1, 8, 1, 0, 600),         # n = 64: one CTA per cluster, one tile, no text
    (2, 7, 1, 9, 3, 1, 600),         # n = 81: two groups, the second with 17 columns
    (1, 8, 2, 16, 2, 127, 500),      # n = 256, m = 128: exactly two tiles
    (3, 12, 2, 17, 2, 128, 775),     # n = 289, m = 66: two rows in the second tile
    (2, 28, 4, 27, 3, 129, 600),     # n = 729
    (1, 4, 2, 31, 2, 40, 300),       # n = 961, m = 673: two passes over the weights
    (37, 2, 2, 10, 1, 20, 600),      # many sequences per unit
    (40, 16, 8, 13, 3, 3, 600),      # more units than one wave
    (1, 2, 1, 12, 1, 2200, 600),     # text beyond sixteen chunks
    (2, 2, 2, 9, 1, 8200, 600),      # text beyond sixty-four
    (8, 4, 4, 9, 1, 2100, 600),      # text beyond sixteen chunks of more items than warps
    (2, 16, 1, 11, 9, 30, 800),      # G = 16
    (2, 16, 1, 9, 15, 1500, 525),    # the text ends last and merges more partials than a warp has lanes
    (200, 8, 4, 9, 1, 40, 600),      # more text items than warps
])
def test_uniform(B, H_q, H_kv, grid, R, T, ratio, recipe, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "cluster")
    shape = wl.Shape("cluster", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    p = tl.make_problem(shape, 700 + grid + B, T=T, T_cap=T + 3, recipe=recipe)
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert counts["cluster"] == 1 and counts["scores"] == 0
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (9, 14, 2, 24, 3, 150, 600), (35, 8, 2, 9, 2, 40, 600), (4, 7, 1, 32, 3, 300, 200), (3, 6, 2, 15, 4, 64, 500),
])
def test_per_sequence_lengths(B, H_q, H_kv, grid, R, T, ratio, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "cluster")
    rng = random.Random(grid)
    R_b = [rng.randint(0, R) for _ in range(B)]
    T_b = [rng.choice([0, 1, T, rng.randint(0, T)]) for _ in range(B)]
    R_b[1], T_b[1] = 0, 0                              # nothing at all: a zero output row
    R_b[-1] = R
    shape = wl.Shape("cluster-ragged", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    counts, _ = tl.check_ragged(shape, 800 + grid, R_b, T_b)
    assert counts["cluster"] == 1 and counts["scores"] == 0


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio,where", [
    (64, 28, 4, 27, 1, 40, 600, range(0, 64, 9)),       # n = 729: eight of 64 sequences have a block
    (128, 14, 2, 9, 1, 300, 600, (0, 127)),             # the first and the last of 128, in one unit
    (60, 16, 1, 11, 2, 20, 600, (3, 59)),               # G = 16
    (300, 2, 2, 9, 3, 5, 600, (1, 2, 298)),             # G = 1
])
def test_long_runs_of_sequences_without_blocks(B, H_q, H_kv, grid, R, T, ratio, where, monkeypatch):
    """A unit's sequences may lie any number of block-less ones apart: its staged queries stay within its 128 rows."""
    monkeypatch.setenv("KVC_EXPANSION", "cluster")
    shape = wl.Shape("cluster-sparse", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    R_b = [R if b in where else 0 for b in range(B)]
    T_b = [T - b % 3 if b % 7 else 0 for b in range(B)]
    counts, _ = tl.check_ragged(shape, 820 + grid, R_b, T_b)
    assert counts["cluster"] == 1 and counts["scores"] == 0


@pytest.mark.parametrize("H_q,H_kv,B,R,grid,T,ratio,path", [
    (16, 16, 64, 2, 9, 60, 875, "phases"), (4, 4, 64, 2, 9, 700, 600, "phases"), (8, 2, 32, 1, 9, 700, 600, "phases"),
    (16, 16, 7, 2, 31, 60, 875, "phases"), (28, 4, 1, 1, 9, 60, 875, "cluster"), (28, 4, 40, 3, 9, 60, 600, "cluster"),
    (8, 2, 16, 5, 19, 60, 600, "spread"), (4, 4, 7, 2, 27, 60, 600, "spread"),
])
def test_routing_of_odd_block_lengths(H_q, H_kv, B, R, grid, T, ratio, path):
    """Block lengths off the tensor-core expansion of the three-phase kernels: every side of the rules, by default routing."""
    shape = wl.Shape("odd-route", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    p = tl.make_problem(shape, 850 + grid, T=T, T_cap=T, recipe="peaked")
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert [counts[k] for k in ("cluster", "spread", "scores")] == [int(path == k) for k in ("cluster", "spread", "phases")]
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,ratio", [(8, 28, 4, 27, 5, 600), (3, 16, 1, 11, 9, 800), (5, 8, 2, 20, 3, 300), (40, 14, 2, 9, 1, 600)])
def test_workspace_holds_every_shorter_text(B, H_q, H_kv, grid, R, ratio, monkeypatch):
    """A workspace of kvc_workspace_bytes(.., T_cap) serves every T <= T_cap, whatever the split of the clusters between units and text:
    nothing behind it is written."""
    monkeypatch.setenv("KVC_EXPANSION", "cluster")
    T_cap = 3000
    shape = wl.Shape("cluster-ws", 1, B, H_q, H_kv, 128, grid, R, T_cap, 1, "bf16", ratio)
    p = tl.make_problem(shape, 870 + grid, T=T_cap, T_cap=T_cap)
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), B, R, caps)
    need = kvc.kvc_workspace_bytes(layer, B, R, T_cap)
    ws = torch.full((need + (8 << 20),), 0xA5, dtype=torch.uint8, device=DEV)
    q, K_txt, V_txt = p["q"].to(DEV), p["K_txt"].to(DEV), p["V_txt"].to(DEV)
    out = torch.empty((B, H_q, 128), dtype=torch.bfloat16, device=DEV)
    full = torch.full((B,), R, dtype=torch.int32, device=DEV)
    for T in (0, 1, 100, 700, 2048, 2049, T_cap):
        counts, _ = tl.launches(lambda: kvc.kvc_decode_attend(layer, q, caps, B, R, K_txt, V_txt, T, T_cap, out, ws))
        assert counts["cluster"] == 1
        kvc.kvc_decode_attend_ragged(layer, q, caps, B, R, full, K_txt, V_txt, T, None, T_cap, out, ws)
        torch.cuda.synchronize()
        assert kvc.kvc_read_device_status(layer, B, R, T, ws) == 0
        assert bool((ws[need:] == 0xA5).all()), T


@pytest.mark.parametrize("path,forced", [("spread", None), ("cluster", "cluster")])
def test_static_entry_point_takes_the_path(path, forced, monkeypatch):
    """8 x 5 blocks of n = 729: the workspace of the call itself fits the fixed scratch, on the path it takes by default and on the cluster path."""
    if forced:
        monkeypatch.setenv("KVC_EXPANSION", forced)
    shape = wl.Shape("cluster-static", 1, 8, 28, 4, 128, 27, 5, 300, 1, "bf16", 600)
    p = tl.make_problem(shape, 890, T=300, T_cap=300, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, 8, 5)
    kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), 8, 5, caps)
    out = torch.full((8, 28, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    run = lambda: kvc.kvc_decode_attend_static(layer, p["q"].to(DEV), caps, 8, 5, p["K_txt"].to(DEV), p["V_txt"].to(DEV), 300, 300, out)
    run()
    counts, _ = tl.launches(run)
    assert [counts[k] for k in ("cluster", "spread", "scores")] == [int(path == "cluster"), int(path == "spread"), 0]
    assert kvc.kvc_workspace_bytes(layer, 8, 5, 300) <= kvc.kvc_static_scratch_bytes()
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")
