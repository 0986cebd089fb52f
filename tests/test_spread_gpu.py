"""The spread decode path (a cluster of CTAs per (sequence, KV head)) at the sizes where its tiling can go wrong, against the fp64
oracle: retained lengths and block lengths around the 16-row granules and the slices they are cut into, one to eight row tiles, one and
two head tiles, two boxes of columns, text lengths around a piece and around what the CTAs share, more pieces than ring slots,
several groups of blocks, per-sequence lengths with nothing in some sequences or groups.

Bound: the regression bound of the parity tests.
"""
import random

import numpy as np
import pytest
import torch

from oracle import kvcapsule_oracle as orc
from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (1, 1, 1, 8, 1, 0, 600),         # n = 64, m = 26: two granules, two CTAs, one row, no text
    (1, 8, 2, 8, 1, 1, 200),         # m = 52: four granules over four CTAs, the last of 4 rows
    (2, 7, 1, 9, 3, 15, 600),        # n = 81: the last column group has one column
    (1, 16, 2, 12, 1, 16, 600),      # n = 144
    (1, 32, 32, 24, 5, 128, 600),    # one row per block
    (2, 28, 4, 27, 5, 300, 600),     # n = 729: two terms, 35 rows
    (8, 28, 4, 27, 5, 33, 600),      # more pairs: four CTAs each
    (3, 14, 2, 32, 9, 513, 600),     # 63 rows, n = 1024
    (8, 8, 4, 32, 3, 47, 400),       # sixteen column groups per CTA: two boxes
    (32, 8, 2, 16, 4, 70, 600),      # two CTAs per pair
    (1, 16, 1, 11, 4, 30, 800),      # two head tiles, 64 rows
    (2, 24, 2, 17, 2, 129, 500),     # G = 12
    (1, 2, 1, 12, 1, 4097, 600),     # long text
    (7, 28, 4, 10, 10, 168, 250),    # 70 rows: two groups of blocks
    (2, 8, 2, 24, 23, 60, 375),      # 92 rows: groups of twelve and eleven blocks
    (1, 16, 2, 9, 31, 33, 600),      # several groups, fewer text items than CTAs
    (24, 28, 4, 12, 2, 40, 600),     # more pairs than clusters the device holds at once
    (11, 32, 8, 11, 18, 30, 600),    # the same with groups
    (1, 4, 1, 31, 4, 40, 300),       # n = 961, m = 673: six granules per CTA, two terms
])
@pytest.mark.parametrize("recipe", ["peaked", "structured"])
def test_uniform(B, H_q, H_kv, grid, R, T, ratio, recipe, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "spread")
    shape = wl.Shape("spread", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    p = tl.make_problem(shape, 600 + grid + B, T=T, T_cap=T + 3, recipe=recipe)
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert counts["spread"] == 1 and counts["cluster"] == counts["scores"] == 0
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (9, 14, 2, 24, 3, 150, 600), (5, 8, 2, 9, 2, 40, 600), (4, 7, 1, 32, 3, 300, 200), (3, 12, 1, 15, 4, 64, 500),
    (5, 8, 2, 12, 23, 70, 600), (3, 28, 4, 13, 20, 40, 600),
])
def test_per_sequence_lengths(B, H_q, H_kv, grid, R, T, ratio, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "spread")
    rng = random.Random(grid)
    R_b = [rng.randint(0, R) for _ in range(B)]
    T_b = [rng.choice([0, 1, T, rng.randint(0, T)]) for _ in range(B)]
    R_b[1], T_b[1] = 0, 0                              # nothing at all: a zero output row
    R_b[-1] = R
    shape = wl.Shape("spread-ragged", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    counts, _ = tl.check_ragged(shape, 650 + grid, R_b, T_b)
    assert counts["spread"] == 1 and counts["cluster"] == counts["scores"] == 0


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,ratio", [(2, 8, 2, 24, 23, 375), (3, 28, 4, 27, 8, 750), (1, 16, 2, 9, 31, 600), (2, 14, 2, 32, 9, 200)])
def test_workspace_holds_every_shorter_text(B, H_q, H_kv, grid, R, ratio, monkeypatch):
    """The number of groups a pair's blocks are split into depends on the text, and at n = 1024, m = 820 the terms on whether the lengths are
    given per sequence: a workspace for T_cap rows serves every T below and both calls, and nothing behind it is written."""
    monkeypatch.setenv("KVC_EXPANSION", "spread")
    T_cap = 6000
    shape = wl.Shape("spread-ws", 1, B, H_q, H_kv, 128, grid, R, T_cap, 1, "bf16", ratio)
    p = tl.make_problem(shape, 690 + grid, T=T_cap, T_cap=T_cap)
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    kvc.kvc_compress(layer, p["K_vis"].cuda(), p["V_vis"].cuda(), B, R, caps)
    need = kvc.kvc_workspace_bytes(layer, B, R, T_cap)
    ws = torch.full((need + (4 << 20),), 0xA5, dtype=torch.uint8, device="cuda")
    q, K_txt, V_txt = p["q"].cuda(), p["K_txt"].cuda(), p["V_txt"].cuda()
    out = torch.empty((B, H_q, 128), dtype=torch.bfloat16, device="cuda")
    full = torch.full((B,), R, dtype=torch.int32, device="cuda")
    for T in (0, 1, 100, 700, 3000, T_cap):
        counts, _ = tl.launches(lambda: kvc.kvc_decode_attend(layer, q, caps, B, R, K_txt, V_txt, T, T_cap, out, ws))
        assert counts["spread"] == 1
        assert kvc.kvc_read_device_status(layer, B, R, T, ws) == 0
        ragged = lambda: kvc.kvc_decode_attend_ragged(layer, q, caps, B, R, full, K_txt, V_txt, T, None, T_cap, out, ws)
        counts, _ = tl.launches(ragged)
        assert counts["spread"] == 1
        assert kvc.kvc_read_device_status(layer, B, R, T, ws) == 0
        assert bool((ws[need:] == 0xA5).all()), T


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio,lengths", [
    (4, 28, 4, 32, 3, 300, 200, True),       # n = 1024, m = 820
    (2, 8, 8, 32, 2, 60, 250, True),         # m = 768, one query head per KV head
    (1, 4, 1, 32, 1, 40, 280, True),         # m = 738
    (2, 8, 2, 36, 1, 100, 200, False),       # n = 1296, m = 1037: no whole multiple of 64
])
def test_long_score_rows_keep_both_terms(B, H_q, H_kv, grid, R, T, ratio, lengths):
    """Rows of scores too long for the tensor-core expansion of the three-phase kernels keep scores and probabilities in two bf16 terms or in
    fp32 on every path that serves them, by default routing.

    Bound, relative 2-norm against 64 bits on the stored capsules: the rounding of the output, at most 2^-9 of every entry, and 1e-4 for
    two terms (16 bits: 5e-6 on this recipe at m = 820; one term 3.8e-3)."""
    shape = wl.Shape("spread-terms", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    p = tl.make_problem(shape, 640 + grid + B, T=T, T_cap=T, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    kvc.kvc_compress(layer, p["K_vis"].cuda(), p["V_vis"].cuda(), B, R, caps)
    K_t, V_t = (tl.np64(x) for x in kvc.capsule_views(layer, caps, B, R))
    q, K_txt, V_txt = p["q"].cuda(), p["K_txt"].cuda(), p["V_txt"].cuda()
    out = torch.empty((B, H_q, 128), dtype=torch.bfloat16, device="cuda")
    ws = kvc.alloc_workspace(layer, B, R, T)
    R_b, T_b = [R - b % R for b in range(B)], [T - b for b in range(B)]
    if lengths:
        i32 = lambda x: torch.tensor(x, dtype=torch.int32, device="cuda")
        kvc.kvc_decode_attend_ragged(layer, q, caps, B, R, i32(R_b), K_txt, V_txt, T, i32(T_b), T, out, ws)
    else:
        R_b, T_b = [R] * B, [T] * B
        kvc.kvc_decode_attend(layer, q, caps, B, R, K_txt, V_txt, T, T, out, ws)
    want = orc.decode_attend_ragged(tl.np64(p["q"]), K_t, V_t, tl.np64(p["theta"]), tl.np64(p["U"]), tl.np64(p["mu"]), tl.np64(p["K_txt"]),
                                    tl.np64(p["V_txt"]), R_b, T_b, "kv")
    err = float(np.linalg.norm(tl.np64(out) - want) / np.linalg.norm(want))
    assert err <= 2.0 ** -9 + 1e-4, err


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio,path", [
    (8, 16, 1, 16, 1, 26, 875, "one"), (5, 12, 1, 16, 2, 267, 850, "one"), (1, 12, 1, 8, 12, 197, 875, "one"),
    (3, 12, 1, 16, 2, 576, 275, "spread"), (3, 12, 1, 24, 5, 260, 750, "spread"), (11, 16, 1, 32, 1, 1, 550, "spread"),
    (9, 16, 1, 23, 4, 3, 550, "spread"), (13, 10, 1, 32, 12, 325, 725, "split"),
    (2, 48, 4, 38, 2, 16, 500, "spread"),        # n = 1444: longer than the cluster path takes
])
def test_routing_with_more_than_eight_query_heads_per_kv_head(B, H_q, H_kv, grid, R, T, ratio, path):
    """Both sides of the rule that compares the path's estimate with one of the path it stands before, by default routing."""
    shape = wl.Shape("spread-route", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    p = tl.make_problem(shape, 670 + grid + B, T=T, T_cap=T, recipe="peaked")
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert [counts["spread"], counts["fused"] - counts["spread"], counts["split_output"]] == [int(path == x) for x in ("spread", "one", "split")]
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")
