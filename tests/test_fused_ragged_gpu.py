"""The one-kernel decode path with per-sequence lengths, against the fp64 oracle: one, two and four sequences per unit, an odd
number of them, the block axis split over units of which some hold no block, one and two row tiles, one and two head tiles, the
three splits of the warps (n up to 256, 640, 1024), sequences with nothing at all.  Whatever lies past a sequence's lengths is NaN.

Bound: the regression bound of the parity tests (scores and probabilities in bf16 as on the kernels' other calls, the weights as
two bf16 terms).
"""
import random

import pytest
import torch

from oracle import kvcapsule_oracle as orc
from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

import kvc_testlib as tl

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    kvc_build.build()


def _launches(fn):
    kvc.kvc_profile_start(64)
    try:
        out = fn()
        torch.cuda.synchronize()
    finally:
        kvc.kvc_profile_stop()
    counts = {k: v[1] for k, v in kvc.kvc_profile_read().items()}
    kvc.kvc_profile_start(0)
    kvc.kvc_profile_stop()
    return counts, out


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
    p = tl.make_problem(shape, 900 + grid, T=T, T_cap=T, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), B, R, caps)
    K_g, V_g = kvc.capsule_views(layer, caps, B, R)
    K_txt, V_txt = p["K_txt"].to(DEV), p["V_txt"].to(DEV)
    for b in range(B):                                 # whatever lies past a sequence's lengths must not be used
        K_g[b, :, R_b[b]:] = float("nan"); V_g[b, :, R_b[b]:] = float("nan")
        K_txt[b, :, T_b[b]:] = float("nan"); V_txt[b, :, T_b[b]:] = float("nan")
    kvc.kvc_layer_capsules_written(layer)
    ws = kvc.alloc_workspace(layer, B, R, T)
    ws.fill_(0xFF)
    out = torch.full((B, H_q, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    i32 = lambda x: torch.tensor(list(x), dtype=torch.int32, device=DEV)
    run = lambda: kvc.kvc_decode_attend_ragged(layer, p["q"].to(DEV), caps, B, R, i32(R_b), K_txt, V_txt, T, i32(T_b), T, out, ws)
    counts, _ = _launches(run)
    assert counts["fused"] == 1 and counts["scores"] == 0
    run()                                              # a second call on the same workspace
    torch.cuda.synchronize()
    assert kvc.kvc_read_device_status(layer, B, R, T, ws) == 0
    K_o, V_o = orc.compress(tl.np64(p["K_vis"]), tl.np64(p["V_vis"]), p["idx"].numpy(), tl.np64(p["U"]), tl.np64(p["mu"]), shape.n, False)
    want = orc.decode_attend_ragged(tl.np64(p["q"]), K_o, V_o, tl.np64(p["theta"]), tl.np64(p["U"]), tl.np64(p["mu"]),
                                    tl.np64(p["K_txt"]), tl.np64(p["V_txt"]), R_b, T_b, "kv")
    tl.assert_close(tl.np64(out), want, "bf16")
    assert (tl.np64(out)[1] == 0).all()
    # a length out of range is clamped and reported
    R_b[0] = R + 1
    run()
    torch.cuda.synchronize()
    assert kvc.kvc_read_device_status(layer, B, R, T, ws) == -8
