"""The work a serving program has this library do, as cases that can be timed.

A program that serves a vision-language model with KVCapsule creates one layer handle per transformer layer, compresses
each layer's vision K/V once at prefill (`kvc_compress`, or `kvc_compress_ragged` for a batch of requests of different
lengths) and then, for every generated token, calls `kvc_decode_attend` (or `kvc_decode_attend_ragged`) on every layer in
turn.  Layers that stay uncompressed are attended with `kvc_attend_full`.  The parameters come from a calibration run with
the fits.  One pass of a case is one such step: all of its layers, each with its own capsules, text rows and queries.

Shapes are those of `workloads.CONFIGS` and of the configuration-4 sweep, or drawn around them: batches from 1 to 64,
square patch grids from 8 x 8 to 32 x 32 (most of them not a multiple of a tile), compression ratios from 0.2 to 0.9, text
tails from one row to a few thousand, MHA and GQA head layouts.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import workloads as wl

D = 128
DEV = "cuda"


def _decode(name, B, heads, grid, R, T, ratio=600, layers=1, dtype="bf16", ragged=False, video=False):
    return dict(name=name, kind="decode", B=B, H_q=heads[0], H_kv=heads[1], grid=grid, R=R, T=T, ratio=ratio, layers=layers,
                dtype=dtype, ragged=ragged, video=video)


def _compress(name, B, heads, grid, R, ratio=600, layers=1, dtype="bf16", ragged=False, video=False):
    return dict(name=name, kind="compress", B=B, H_q=heads[0], H_kv=heads[1], grid=grid, R=R, T=0, ratio=ratio, layers=layers,
                dtype=dtype, ragged=ragged, video=video)


def listed():
    return [
        # one layer, one sequence, one image in fp32: the smallest call there is, a debugging or edge deployment
        _decode("decode-f32-1seq-1layer", 1, (8, 2), 24, 1, 32, dtype="f32"),
        # interactive use: one request, one image of 5 crops, all 32 MHA layers
        _decode("decode-crops-1seq", 1, (32, 32), 24, 5, 128, layers=32),
        # the 7B benchmark configurations at the text length of the middle of the run
        _decode("decode-crops-8seq", 8, (32, 32), 24, 5, 256, layers=32),
        _decode("decode-images-16seq", 16, (28, 4), 32, 8, 512, layers=28),
        _decode("decode-video-4seq", 4, (28, 4), 16, 32, 1024, layers=28, video=True),
        # the largest batch of long multi-image requests of the sweep; a few layers of it fill the device
        _decode("decode-images-64seq-long", 64, (28, 4), 32, 32, 320, layers=2),
        # continuous batching: requests with different numbers of crops / images and different text lengths
        _decode("decode-crops-8seq-ragged", 8, (32, 32), 24, 5, 512, layers=32, ragged=True),
        # a vision tower whose patch grid is not a multiple of any tile (27 x 27)
        _decode("decode-grid27-8seq", 8, (28, 4), 27, 5, 300, layers=28),
        # prefill: the vision K/V of a batch compressed layer by layer
        _compress("compress-crops-8seq", 8, (32, 32), 24, 5, layers=4),
        # prefill of requests of different lengths: whole blocks compressed, the rest copied in front of the text rows
        _compress("compress-images-8seq-ragged", 8, (28, 4), 32, 8, layers=4, ragged=True),
        # layers left uncompressed (a pyramid schedule keeps some at ratio 0): plain decode attention over K and V
        dict(name="attend-full-16seq", kind="attend", B=16, H_q=28, H_kv=4, S=8704, layers=4),
        # calibration: value basis and key reconstructor of one layer fitted from activations
        dict(name="fit-grid16", kind="fit", B=4, H_kv=4, grid=16, R=8, ratio=600, dtype="bf16"),
    ]


_HEADS = ((32, 32), (28, 4), (28, 4), (32, 8), (8, 2), (16, 2))
_BUDGET = 6e9       # bytes of one pass and 36 flop to the byte: the largest listed cases move 6.5e9 bytes or take 2.2e11 flop


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("decode", "compress", "attend", "fit"), (14, 5, 2, 1))[0]
    heads = rng.choice(_HEADS)
    if kind == "attend":
        c = dict(kind=kind, B=_log(rng, 1, 64), H_q=heads[0], H_kv=heads[1], S=_log(rng, 64, 32768), layers=rng.choice((1, 2, 4, 28)))
        while work(c)["bytes"] > _BUDGET:
            c[("B", "layers")[c["B"] <= c["layers"]]] //= 2
        return c
    if kind == "fit":
        return dict(kind=kind, B=rng.randint(1, 4), H_kv=heads[1] % 7 + 1, grid=rng.randint(6, 16), R=rng.randint(4, 8),
                    ratio=rng.randrange(400, 901, 25), dtype=rng.choice(("bf16", "f32")))
    grid = rng.choice((16, 24, 32)) if rng.random() < 0.5 else rng.randint(8, 32)
    dtype = "f32" if rng.random() < 0.1 else "bf16"
    c = dict(kind=kind, B=_log(rng, 1, 64), H_q=heads[0], H_kv=heads[1], grid=grid, R=_log(rng, 1, 32),
             T=_log(rng, 1, 4096) if kind == "decode" else 0, ratio=rng.randrange(200, 901, 25),
             layers=rng.choice((1, 4, 28)) if kind == "decode" else rng.choice((1, 2, 4)), dtype=dtype,
             ragged=rng.random() < 0.3, video=grid <= 16 and rng.random() < 0.5)
    budget = _BUDGET if dtype == "bf16" else _BUDGET / 16      # fp32 is for checking, at the sizes people check at
    # bytes, and the dense products of large batches (they take long before they move much)
    while max(work(c)["bytes"], work(c)["flops"] / 36, c["layers"] * _vision_bytes(c)) > budget:
        k = max(("B", "R", "layers"), key=lambda x: c[x])
        c[k] = max(1, c[k] // 2)
        if c["B"] * c["R"] * c["layers"] == 1:
            break
    return c


# ---- sizes ---------------------------------------------------------------------------------------------------------
def _eb(c):
    return 4 if c.get("dtype", "bf16") == "f32" else 2


def _m(c):
    n = c["grid"] ** 2
    return (n * (1000 - c["ratio"]) + 999) // 1000


def _vision_bytes(c):
    return 2 * c["B"] * c["H_kv"] * c["R"] * c["grid"] ** 2 * D * _eb(c)


def _lengths(c):
    """(blocks, rows past the last whole block, text rows) of every sequence; the same for every seed of a case."""
    if not c["ragged"]:
        return [(c["R"], 0, c["T"])] * c["B"]
    rng = random.Random(c["B"] * 1000003 + c["R"] * 1009 + c["T"])
    out = []
    for _ in range(c["B"]):
        r = rng.randint((c["R"] + 1) // 2, c["R"])
        tail = rng.randrange(c["grid"] ** 2) if c["kind"] == "compress" and r < c["R"] else 0
        out.append((r, tail, rng.randint(max(1, c["T"] // 4), c["T"]) if c["T"] else 0))
    return out


def work(case):
    c = case
    if c["kind"] == "attend":
        kv = 2 * c["B"] * c["H_kv"] * c["S"] * D * 2
        return dict(bytes=c["layers"] * (kv + 4 * c["B"] * c["H_q"] * D), flops=c["layers"] * 4 * c["B"] * c["H_q"] * c["S"] * D)
    if c["kind"] == "fit":
        n, m = c["grid"] ** 2, _m(c)
        eb = _eb(c)
        # second moments of K and V, an eigen-decomposition of n x n and one of m x m (about 10 n^3 with the vectors), the solve
        per_head = 4 * c["B"] * c["R"] * n * n * D + 10 * n ** 3 + 10 * m ** 3 + 4 * m * m * n
        return dict(bytes=c["H_kv"] * (2 * c["B"] * c["R"] * n * D * eb + 2 * m * n * eb), flops=c["H_kv"] * per_head)
    n, m, eb, H_q, H_kv = c["grid"] ** 2, _m(c), _eb(c), c["H_q"], c["H_kv"]
    L = _lengths(c)
    blocks, tails, text = (sum(x[k] for x in L) for k in range(3))
    if c["kind"] == "compress":
        rows_in = blocks * (m + n) + 2 * tails           # the retained key rows and all value rows, rows left over twice
        rows_out = blocks * 2 * m + 2 * tails
        byt = H_kv * ((rows_in + rows_out) * D + m * n) * eb
        return dict(bytes=c["layers"] * byt, flops=c["layers"] * 2 * H_kv * blocks * m * n * D)
    byt = (2 * H_kv * (blocks * m + text) * D + 2 * c["B"] * H_q * D + 2 * H_kv * m * n) * eb
    flops = 4 * H_q * (blocks * (m * D + m * n) + text * D)
    return dict(bytes=c["layers"] * byt, flops=c["layers"] * flops)


def tolerance(case):
    """About four times the error measured against fp64 (relative 2-norm): fp32 sums 1e-6; bf16 storage: decode 4.5e-3 (stored
    capsules, scores and probabilities rounded), plain attention 2.1e-3, one rounding of the result (compress, fits) 1.7e-3;
    the fits compute in fp64, so in fp32 storage only their result is rounded (3e-8)."""
    kind = case["kind"]
    if case.get("dtype", "bf16") == "f32":
        return {"rel": 1e-6 if kind == "fit" else 1e-5}
    return {"rel": {"decode": 1.5e-2, "attend": 8e-3, "compress": 6e-3, "fit": 6e-3}[kind]}


# ---- inputs --------------------------------------------------------------------------------------------------------
def _noise(shape, gen, dtype, std=1.0):
    return (torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32) * std).to(dtype)


def _vision(c, seed, dtype, gain=1.0):
    """Vision K or V of one layer [B, H_kv, R n, d]: smoothed patch fields, frames of an AR(1) process for video."""
    x = wl.vision_kv(c["B"], c["H_kv"], c["R"], c["grid"], D, seed, DEV, torch.float32 if gain != 1.0 else dtype, 0.9 if c.get("video") else 0.0)
    return x if gain == 1.0 else (x * gain).to(dtype)


def _layer(c, k, seed, dtype):
    """One layer handle with parameters that give softmaxes a few positions dominate (the "peaked" recipe)."""
    n, m = c["grid"] ** 2, _m(c)
    theta, U, mu = wl.peaked_params(c["H_kv"], m, n, D, seed, DEV, dtype)
    return kvc.Layer(c["H_q"], c["H_kv"], D, n, c["ratio"], dtype, idx=wl.evenly_spaced_idx(n, m), theta=theta, U=U,
                     mu=(mu * 0.4).to(dtype), layer=k)


def _i32(values):
    return torch.tensor(list(values), dtype=torch.int32, device=DEV)


def _queries(s, c, gen, dtype):
    """Queries and outputs of all layers: slices of one tensor each."""
    q = _noise((c["layers"], c["B"], c["H_q"], D), gen, dtype)
    s["out"] = torch.empty_like(q)
    for k, p in enumerate(s["layers"]):
        p["q"], p["out"] = q[k], s["out"][k]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 17)
    dtype = wl.torch_dtype(c.get("dtype", "bf16"))
    s = dict(c=c, layers=[])
    if c["kind"] == "attend":
        for k in range(c["layers"]):
            p = dict(layer=kvc.Layer(c["H_q"], c["H_kv"], D, 64, 0, dtype, layer=k))
            p["K"] = _noise((c["B"], c["H_kv"], c["S"], D), gen, dtype, 3.5)
            p["V"] = _noise((c["B"], c["H_kv"], c["S"], D), gen, dtype, 0.4)
            s["layers"].append(p)
        _queries(s, c, gen, dtype)
        s["ws"] = kvc.alloc_workspace(s["layers"][0]["layer"], c["B"], 0, c["S"])
        return s
    if c["kind"] == "fit":
        n, m = c["grid"] ** 2, _m(c)
        s["K"], s["V"] = _vision(c, seed * 64 + 1, dtype), _vision(c, seed * 64 + 2, dtype)
        s["idx"], s["n"], s["m"] = wl.evenly_spaced_idx(n, m), n, m
        return s
    n, B, R, T = c["grid"] ** 2, c["B"], c["R"], c["T"]
    L = _lengths(c)
    order = list(range(B))
    random.Random(seed).shuffle(order)                   # another seed deals the same lengths to other requests
    L = [L[i] for i in order]
    for k in range(c["layers"]):
        p = dict(layer=_layer(c, k, seed * 64 + k, dtype))
        p["caps"] = kvc.alloc_capsules(p["layer"], B, R)
        s["layers"].append(p)
        K, V = _vision(c, (seed * 64 + k) * 2, dtype), _vision(c, (seed * 64 + k) * 2 + 1, dtype, 0.4)
        if c["kind"] == "compress":
            p["K"], p["V"] = K, V
            p["caps"].zero_()
            continue
        kvc.kvc_compress(p["layer"], K, V, B, R, p["caps"])
        p["K_txt"] = _noise((B, c["H_kv"], T, D), gen, dtype, 3.5)
        p["V_txt"] = _noise((B, c["H_kv"], T, D), gen, dtype, 0.4)
        del K, V
    if c["kind"] == "compress":
        if c["ragged"]:
            s["N_v"] = _i32(r * n + t for r, t, _ in L)
            s["R_b"], s["T_b"] = _i32([0] * B), _i32([0] * B)
            s["T_cap"] = n
            for p in s["layers"]:
                p["tails"] = torch.zeros((2, B, c["H_kv"], n, D), dtype=dtype, device=DEV)
        return s
    _queries(s, c, gen, dtype)
    s["ws"] = kvc.alloc_workspace(s["layers"][0]["layer"], B, R, T)
    if c["ragged"]:
        s["R_b"], s["T_b"], s["T_max"] = _i32(x[0] for x in L), _i32(x[2] for x in L), max(x[2] for x in L)
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------
def run(state):
    s = state
    c = s["c"]
    if c["kind"] == "fit":
        U, mu, eig, _ = kvc.kvc_fit_value_pca(s["V"], s["n"], s["m"], want_eig=True)
        theta, _ = kvc.kvc_fit_key_reconstructor(s["K"], s["idx"], s["n"])
        return U, mu, eig, theta
    if c["kind"] == "attend":
        for p in s["layers"]:
            kvc.kvc_attend_full(p["layer"], p["q"], p["K"], p["V"], c["B"], c["S"], c["S"], p["out"], s["ws"])
        return s["out"]
    B, R, T = c["B"], c["R"], c["T"]
    if c["kind"] == "compress":
        for p in s["layers"]:
            if c["ragged"]:
                kvc.kvc_compress_ragged(p["layer"], p["K"], p["V"], B, R * s["T_cap"], s["N_v"], R, p["caps"], p["tails"][0],
                                        p["tails"][1], s["T_cap"], s["R_b"], s["T_b"])
            else:
                kvc.kvc_compress(p["layer"], p["K"], p["V"], B, R, p["caps"])
        out = [kvc.capsule_views(p["layer"], p["caps"], B, R) for p in s["layers"]]
        return (out, [p["tails"] for p in s["layers"]], s["R_b"], s["T_b"]) if c["ragged"] else out
    for p in s["layers"]:
        if c["ragged"]:
            kvc.kvc_decode_attend_ragged(p["layer"], p["q"], p["caps"], B, R, s["R_b"], p["K_txt"], p["V_txt"], s["T_max"],
                                         s["T_b"], T, p["out"], s["ws"])
        else:
            kvc.kvc_decode_attend(p["layer"], p["q"], p["caps"], B, R, p["K_txt"], p["V_txt"], T, T, p["out"], s["ws"])
    return s["out"]
