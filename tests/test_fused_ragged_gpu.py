"""The one-kernel decode path with per-sequence lengths, against the fp64 oracle: one, two and four sequences per unit, an odd
number of them, the block axis split over units of which some hold no block, one and two row tiles, one and two head tiles, the
three splits of the warps (n up to 256, 640, 1024), sequences with nothing at all.  Whatever lies past a sequence's lengths is NaN.

Bound: the regression bound of the parity tests (scores and probabilities in bf16 as on the kernels' other calls, the weights as
two bf16 terms).
"""
import random

import pytest

from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio", [
    (5, 4, 4, 24, 3, 70, 600),       # two sequences per unit, an odd number of them
    (9, 2, 2, 16, 3, 33, 600),       # four sequences per unit, n = 256
    (3, 16, 1, 16, 9, 50, 500),      # G = 16, two row tiles, the block axis in five units
    (3, 14, 2, 24, 7, 300, 600),     # G = 7, four units along the block axis, some without any block of their sequence
    (3, 6, 6, 32, 2, 130, 600),      # n = 1024
    (4, 32, 2, 24, 2, 20, 300),      # G = 16, n = 576, m = 403
    (70, 2, 2, 8, 2, 5, 600),        # more sequences than threads of a warp to sort
])
def test_per_sequence_lengths(B, H_q, H_kv, grid, R, T, ratio, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "mma")
    rng = random.Random(grid)
    R_b = [rng.randint(0, R) for _ in range(B)]
    T_b = [rng.choice([0, 1, T, rng.randint(0, T)]) for _ in range(B)]
    R_b[1], T_b[1] = 0, 0                              # nothing at all: a zero output row
    R_b[-1] = R
    shape = wl.Shape("one-kernel-ragged", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio)
    counts, _ = tl.check_ragged(shape, 900 + grid, R_b, T_b)
    assert counts["fused"] == 1 and counts["cluster"] == counts["plain"] == counts["scores"] == 0
