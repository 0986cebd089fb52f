"""The fp32 form of the spread decode path at the sizes where its tiling can go wrong, against the fp64 oracle: few and many columns per CTA,
column counts and rows of U off 16 bytes, one and several chunks of U, row and head tiles of 4, 8 and 16, groups of blocks, text shares of
nothing, one row and many, per-sequence lengths with nothing in some sequences or groups.

Bound: the regression bound of the parity tests (5e-6 of the largest output).
"""
import random

import pytest
import torch

from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (1, 8, 2, 24, 1, 32, 600),       # n = 576: 72 columns per CTA
    (1, 1, 1, 8, 1, 0, 600),         # one row, no text
    (2, 6, 2, 9, 3, 1, 600),         # n = 81: the last quad has one column; one text row for all CTAs
    (1, 16, 1, 13, 1, 50, 600),      # G = 16, n = 169
    (3, 28, 4, 16, 2, 200, 500),     # clusters of four
    (12, 8, 4, 20, 2, 33, 600),      # clusters of two
    (1, 8, 2, 32, 2, 300, 400),      # n = 1024, m = 615: several chunks of U
    (2, 8, 2, 17, 11, 70, 775),      # n = 289, eleven blocks: groups
    (1, 2, 2, 12, 30, 2100, 600),    # many blocks and text rows
    (13, 28, 4, 13, 3, 61, 450),     # more groups than clusters the device holds at once
    (1, 4, 1, 31, 4, 10, 300),       # n = 961, m = 673
])
@pytest.mark.parametrize("recipe", ["peaked", "structured"])
def test_uniform(B, H_q, H_kv, grid, R, T, ratio, recipe):
    shape = wl.Shape("spread-f32", 1, B, H_q, H_kv, 128, grid, R, T, 1, "f32", ratio)
    p = tl.make_problem(shape, 640 + grid + B, T=T, T_cap=T + 3, recipe=recipe)
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert counts["spread"] == 1 and counts["scores"] == 0
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "f32")


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [(5, 8, 2, 24, 3, 150, 600), (4, 4, 4, 9, 13, 40, 600), (6, 7, 1, 15, 5, 300, 500)])
def test_per_sequence_lengths(B, H_q, H_kv, grid, R, T, ratio, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "spread")
    rng = random.Random(grid)
    R_b = [rng.randint(0, R) for _ in range(B)]
    T_b = [rng.choice([0, 1, T, rng.randint(0, T)]) for _ in range(B)]
    R_b[1], T_b[1] = 0, 0                              # nothing at all: a zero output row
    R_b[-1] = R
    shape = wl.Shape("spread-f32-ragged", 1, B, H_q, H_kv, 128, grid, R, T, 1, "f32", ratio)
    counts, _ = tl.check_ragged(shape, 660 + grid, R_b, T_b)
    assert counts["spread"] == 1 and counts["scores"] == 0
