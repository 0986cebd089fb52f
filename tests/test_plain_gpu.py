"""Plain attention (uncompressed K/V, text alone, stores of ratio 0) at the sizes where the split over CTAs and warps can go wrong: one row,
rows around the 16-row steps, fewer steps than warps, pairs shared by many CTAs, one CTA per pair, more pairs than SMs with whole and
with crossing runs, both kinds of rows in one pair, G of 1 to 16, NaN behind the last row.

Bound: the regression bound of the parity tests.
"""
import numpy as np
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


@pytest.mark.parametrize("B,H_q,H_kv,S", [
    (1, 1, 1, 1), (1, 7, 1, 15), (2, 4, 2, 17), (1, 8, 1, 191), (1, 7, 1, 769), (1, 16, 1, 3000), (1, 2, 2, 9000), (3, 12, 1, 800),
    (37, 8, 4, 50), (75, 4, 2, 33), (80, 4, 2, 1600), (151, 1, 1, 1700), (40, 28, 4, 300),
    (80, 1, 1, 7200), (20, 4, 4, 7150),        # one pair per CTA with crossing runs (a pair on up to three CTAs), and just not
])
def test_attend_full(B, H_q, H_kv, S):
    gen = torch.Generator().manual_seed(S + B)
    bf = lambda *s, std=1.0: (torch.randn(s, generator=gen) * std).to(torch.bfloat16)
    S_cap = S + 5
    q, K, V = bf(B, H_q, 128), bf(B, H_kv, S_cap, 128, std=2.5), bf(B, H_kv, S_cap, 128, std=0.5)
    K[:, :, S:] = float("nan"); V[:, :, S:] = float("nan")
    layer = kvc.Layer(H_q, H_kv, 128, 64, 0, torch.bfloat16)
    ws = kvc.alloc_workspace(layer, B, 0, S_cap)
    ws.fill_(0xFF)
    out = torch.full((B, H_q, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    Kd, Vd, qd = K.to(DEV), V.to(DEV), q.to(DEV)
    for _ in range(2):                                 # the second call meets the first one's arrival words
        counts, _ = tl.launches(lambda: kvc.kvc_attend_full(layer, qd, Kd, Vd, B, S, S_cap, out, ws))
        assert counts["plain"] == 1
    assert kvc.kvc_read_device_status(layer, B, 0, S, ws) == 0
    k64, v64 = (np.repeat(tl.np64(x)[:, :, :S], H_q // H_kv, axis=1) for x in (K, V))
    logits = np.einsum("bhd,bhsd->bhs", tl.np64(q), k64) / np.sqrt(128.0)
    p = np.exp(logits - logits.max(-1, keepdims=True))
    want = np.einsum("bhs,bhsd->bhd", p / p.sum(-1, keepdims=True), v64)
    tl.assert_close(tl.np64(out), want, "bf16", f"B={B} S={S}")


@pytest.mark.parametrize("B,H_q,H_kv,grid,R,T", [(1, 7, 1, 3, 1, 1), (2, 8, 2, 9, 3, 20), (1, 9, 1, 16, 8, 500), (5, 4, 4, 5, 2, 0)])
def test_ratio_zero_store_with_text(B, H_q, H_kv, grid, R, T):
    shape = wl.Shape("rho0", 1, B, H_q, H_kv, 128, grid, R, T, 1, "bf16", ratio_permille=0)
    p = tl.make_problem(shape, 640 + grid, T=T, T_cap=T + 4)
    counts, (_, _, _, out) = tl.launches(lambda: tl.gpu_run(shape, p))
    assert counts["plain"] == 1
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")
