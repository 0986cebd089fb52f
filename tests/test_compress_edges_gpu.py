"""The one-kernel bf16 compression at the sizes where its tiling can go wrong, against the fp64 oracle: block lengths around and
off the 64-column stages, retained lengths around the 128-row tiles, odd block counts (a unit takes blocks in pairs) and per-sequence
lengths from nothing to all blocks with rows left over.

Bound: the products are exact in fp32 and summed over n terms, then rounded once to bf16, so an element is within half a bf16 step
of its magnitude (2^-8 relative) plus the fp32 sums' error, n 2^-24 of sum |U| |V - mu|, below 1e-4 of the largest element here.
"""
import numpy as np
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


def _assert_capsules(got, want, what):
    assert np.isfinite(got).all(), what
    assert (np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-4 * np.abs(want).max()).all(), what


@pytest.mark.parametrize("B,H,grid,R,ratio", [
    (1, 1, 3, 1, 500),       # n = 9, m = 5: one partial tile, one block
    (1, 2, 8, 3, 10),        # n = 64, m = 64
    (2, 1, 11, 3, 400),      # n = 121, odd rows of U; 6 blocks
    (1, 3, 16, 5, 500),      # m = 128: exactly one row tile; an odd number of blocks
    (1, 1, 16, 1, 495),      # m = 130: two rows in the second tile
    (3, 1, 13, 1, 200),      # n = 169, m = 136
    (1, 2, 27, 3, 600),      # n = 729
    (2, 33, 24, 3, 600),     # more units than SMs: accumulators and stages go round
])
def test_uniform_compression(B, H, grid, R, ratio):
    shape = wl.Shape("compress-edge", 1, B, H, H, 128, grid, R, 1, 1, "bf16", ratio)
    p = tl.make_problem(shape, 900 + grid + R, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    counts, _ = tl.launches(lambda: kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), B, R, caps))
    assert counts["compress"] == 1
    assert kvc.kvc_read_compress_status(layer) == 0
    K_t, V_t = orc.compress(tl.np64(p["K_vis"]), tl.np64(p["V_vis"]), p["idx"].numpy(), tl.np64(p["U"]), tl.np64(p["mu"]), shape.n, False)
    K_g, V_g = (tl.np64(x) for x in kvc.capsule_views(layer, caps, B, R))
    assert (K_g == K_t).all()
    _assert_capsules(V_g, V_t, "values")


@pytest.mark.parametrize("grid,mode", [(8, "kv"), (11, "kv"), (16, "k"), (13, "v")])
def test_ragged_compression(grid, mode):
    n, B, H, R_max, T_cap = grid * grid, 35, 2, 3, grid * grid + 5
    lengths = ([0, 1, n - 1, n, n + 1, 2 * n, 3 * n, 3 * n + n // 2, 2 * n + n - 1] * 4)[:B]
    shape = wl.Shape("compress-ragged", 1, B, H, H, 128, grid, 4, 1, 1, "bf16", 600)
    p = tl.make_problem(shape, 950 + grid, recipe="peaked")
    layer = tl.gpu_layer(shape, p, DEV, mode)
    caps = kvc.alloc_capsules(layer, B, R_max)
    caps.fill_(0)
    K, V = p["K_vis"].to(DEV), p["V_vis"].to(DEV)
    kt, vt = (torch.full((B, H, T_cap, 128), 7.0, dtype=torch.bfloat16, device=DEV) for _ in range(2))
    for b, nv in enumerate(lengths):                  # whatever lies past a sequence's length must not be used
        K[b, :, nv:] = float("nan"); V[b, :, nv:] = float("nan")
    i32 = lambda x: torch.tensor(list(x), dtype=torch.int32, device=DEV)
    R_b, T_b = i32([-1] * B), i32([-1] * B)
    kvc.kvc_compress_ragged(layer, K, V, B, 4 * n, i32(lengths), R_max, caps, kt, vt, T_cap, R_b, T_b)
    torch.cuda.synchronize()
    assert kvc.kvc_read_compress_status(layer) == 0
    assert R_b.tolist() == [nv // n for nv in lengths] and T_b.tolist() == [nv % n for nv in lengths]
    K_o, V_o = orc.compress(tl.np64(p["K_vis"]), tl.np64(p["V_vis"]), p["idx"].numpy(), tl.np64(p["U"]), tl.np64(p["mu"]), n, False, mode)
    K_g, V_g = (tl.np64(x) for x in kvc.capsule_views(layer, caps, B, R_max))
    for b, nv in enumerate(lengths):
        r, t = nv // n, nv % n
        assert (K_g[b, :, :r] == K_o[b, :, :r]).all() and (K_g[b, :, r:] == 0).all() and (V_g[b, :, r:] == 0).all()
        if mode == "k":
            assert (V_g[b, :, :r] == V_o[b, :, :r]).all()
        elif r:
            _assert_capsules(V_g[b, :, :r], V_o[b, :, :r], f"values of sequence {b}")
        assert torch.equal(kt[b, :, :t].cpu(), p["K_vis"][b, :, r * n:r * n + t]) and (kt[b, :, t:] == 7).all()
        assert torch.equal(vt[b, :, :t].cpu(), p["V_vis"][b, :, r * n:r * n + t]) and (vt[b, :, t:] == 7).all()


@pytest.mark.parametrize("over", ["R_b", "T_b"])
def test_lengths_may_be_written_over_the_row_counts(over):
    """N_v and R_b (or T_b) one array: capsules, rows left over and lengths as with arrays of their own."""
    n, B, H, R, N_cap = 81, 40, 4, 3, 4 * 81
    shape = wl.Shape("compress-in-place", 1, B, H, H, 128, 9, 4, 1, 1, "bf16", 600)
    p = tl.make_problem(shape, 961, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    K, V = p["K_vis"].to(DEV), p["V_vis"].to(DEV)
    lengths = [(37 * b) % (3 * n + 50) for b in range(B)]
    i32 = lambda x: torch.tensor(list(x), dtype=torch.int32, device=DEV)
    got = []
    for shared in (False, True):
        caps = kvc.alloc_capsules(layer, B, R)
        caps.fill_(0)
        kt, vt = (torch.zeros((B, H, n, 128), dtype=torch.bfloat16, device=DEV) for _ in range(2))
        N_v, out = i32(lengths), dict(R_b=i32([-1] * B), T_b=i32([-1] * B))
        if shared:
            out[over] = N_v
        kvc.kvc_compress_ragged(layer, K, V, B, N_cap, N_v, R, caps, kt, vt, n, out["R_b"], out["T_b"])
        torch.cuda.synchronize()
        assert kvc.kvc_read_compress_status(layer) == 0
        got.append((caps, kt, vt, out["R_b"], out["T_b"]))
    assert got[0][3].tolist() == [x // n for x in lengths] and got[0][4].tolist() == [x % n for x in lengths]
    for a, b in zip(*got):
        assert torch.equal(a, b)
