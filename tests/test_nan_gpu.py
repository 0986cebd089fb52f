"""A NaN that a call reads comes back as NaN, in the heads and channels that depend on it and in no others: a query, a retained key row, a
text key row, a value row, for one and several groups of blocks per (sequence, KV head) in both storage types.  A sequence with nothing to
attend to still gets a zero row beside it.

Reference: the fp64 oracle, which passes a NaN on through its maximum; finite entries to the regression bound of the parity tests.
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


def _check(B, H_q, H_kv, grid, R, T, ratio, dtype, where, lengths):
    shape = wl.Shape("nan", 1, B, H_q, H_kv, 128, grid, R, T, 1, dtype, ratio)
    p = tl.make_problem(shape, 910 + grid, T=T, T_cap=T, recipe="peaked")
    layer = tl.gpu_layer(shape, p)
    caps = kvc.alloc_capsules(layer, B, R)
    kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), B, R, caps)
    K_t, V_t = kvc.capsule_views(layer, caps, B, R)
    q, K_txt, V_txt = (p[k].to(DEV) for k in ("q", "K_txt", "V_txt"))
    R_b, T_b = [R] * B, [T] * B
    if lengths:
        R_b[0], T_b[0] = 0, 0                          # nothing at all: a zero output row
    nan, b, h = float("nan"), B - 1, H_kv - 1
    if where == "query":
        q[b, -1, 5] = nan                              # one head
    elif where == "key":
        K_t[b, h, R - 1, layer.m // 2, 7] = nan        # every head of the group
    elif where == "text key":
        K_txt[b, h, T - 1, 3] = nan
    elif where == "value":
        V_t[b, h, R - 1, layer.m - 1, 9] = nan         # one channel
    elif where == "text value":
        V_txt[b, h, T // 2, 127] = nan
    kvc.kvc_layer_capsules_written(layer)
    ws = kvc.alloc_workspace(layer, B, R, T)
    out = torch.empty((B, H_q, 128), dtype=wl.torch_dtype(dtype), device=DEV)
    i32 = lambda x: torch.tensor(x, dtype=torch.int32, device=DEV)
    if lengths:
        run = lambda: kvc.kvc_decode_attend_ragged(layer, q, caps, B, R, i32(R_b), K_txt, V_txt, T, i32(T_b), T, out, ws)
    else:
        run = lambda: kvc.kvc_decode_attend(layer, q, caps, B, R, K_txt, V_txt, T, T, out, ws)
    counts, _ = tl.launches(run)
    want = orc.decode_attend_ragged(tl.np64(q), tl.np64(K_t), tl.np64(V_t), tl.np64(p["theta"]), tl.np64(p["U"]), tl.np64(p["mu"]),
                                    tl.np64(K_txt), tl.np64(V_txt), R_b, T_b, "kv")
    got = tl.np64(out)
    assert np.isnan(want).any() and np.isfinite(want).any()
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    tl.assert_close(np.nan_to_num(got), np.nan_to_num(want), dtype)
    if lengths:
        assert (got[0] == 0).all()
    return counts


@pytest.mark.parametrize("lengths", [False, True])
@pytest.mark.parametrize("where", ["query", "key", "text key", "value", "text value"])
@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T,ratio,dtype", [
    (2, 8, 2, 24, 2, 70, 600, "bf16"),       # one group of blocks
    (2, 28, 4, 27, 3, 40, 600, "bf16"),      # two terms
    (2, 8, 2, 24, 23, 60, 375, "bf16"),      # several groups
    (2, 8, 2, 24, 1, 32, 600, "f32"),
    (2, 8, 2, 17, 11, 70, 775, "f32"),       # several groups
])
def test_spread_path(B, H_q, H_kv, grid, R, T, ratio, dtype, where, lengths, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", "spread")
    counts = _check(B, H_q, H_kv, grid, R, T, ratio, dtype, where, lengths)
    assert counts["spread"] == 1 and counts["cluster"] == counts["scores"] == 0


@pytest.mark.parametrize("lengths", [False, True])
@pytest.mark.parametrize("where", ["query", "key", "text key", "value", "text value"])
@pytest.mark.parametrize("path,grid,dtype", [("phases", 24, "bf16"), ("phases", 24, "f32"), ("phases", 27, "bf16"), ("resident", 16, "bf16"),
                                             ("mma", 24, "bf16"), ("tcgen05", 24, "bf16"), ("split", 32, "bf16"), ("cluster", 24, "bf16")])
def test_other_paths(path, grid, dtype, where, lengths, monkeypatch):
    monkeypatch.setenv("KVC_EXPANSION", path)
    counts = _check(2, 8, 2, grid, 2, 70, 600, dtype, where, lengths)
    assert counts["spread"] == 0


@pytest.mark.parametrize("lengths", [False, True])
@pytest.mark.parametrize("path,grid,R,dtype", [
    ("resident", 16, 12, "bf16"), ("phases", 16, 12, "bf16"), ("phases", 16, 12, "f32"), ("mma", 24, 12, "bf16"), ("tcgen05", 24, 12, "bf16"),
    ("split", 32, 6, "bf16"), ("cluster", 24, 24, "bf16"), ("spread", 24, 24, "bf16"), ("spread", 17, 11, "f32"),
])
def test_whole_parts_of_nan(path, grid, R, dtype, lengths, monkeypatch):
    """No text row, one query of NaN: every part that is joined has a NaN for a sum and nothing for a maximum."""
    monkeypatch.setenv("KVC_EXPANSION", path)
    _check(2, 8, 2, grid, R, 0, 600, dtype, "query", lengths)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("S", [1, 70, 3000])
def test_uncompressed_attention(S, dtype):
    gen = torch.Generator().manual_seed(S)
    B, H_q, H_kv = 2, 8, 2
    q, K, V = (torch.randn(x, generator=gen).to(wl.torch_dtype(dtype)) for x in ((B, H_q, 128), (B, H_kv, S, 128), (B, H_kv, S, 128)))
    q[1, -1, 5] = float("nan")
    K[0, 0, S // 2, 3] = float("nan")
    V[0, 1, S - 1, 9] = float("nan")
    layer = kvc.Layer(H_q, H_kv, 128, 64, 0, wl.torch_dtype(dtype))
    ws = kvc.alloc_workspace(layer, B, 0, S)
    out = torch.empty((B, H_q, 128), dtype=wl.torch_dtype(dtype), device=DEV)
    kvc.kvc_attend_full(layer, q.to(DEV), K.to(DEV), V.to(DEV), B, S, S, out, ws)
    x = torch.einsum("bhgd,bhsd->bhgs", q.double().view(B, H_kv, -1, 128) * 128 ** -0.5, K.double())
    want = torch.einsum("bhgs,bhsd->bhgd", torch.softmax(x, -1), V.double()).reshape(B, H_q, 128).numpy()
    got = tl.np64(out)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    tl.assert_close(np.nan_to_num(got), np.nan_to_num(want), dtype)
