"""What kvc_layer_create reads and keeps: parameters that are still being written on another stream, and device memory for padded copies only
where a kernel reads them."""
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


@pytest.mark.parametrize("grid", [9, 16, 27])
def test_parameters_on_their_way_on_another_stream(grid):
    shape = wl.Shape("create-late", 1, 2, 14, 2, 128, grid, 2, 20, 1, "bf16", 600)
    p = tl.make_problem(shape, 1100 + grid, T=20, T_cap=24, recipe="peaked")
    src = {k: p[k].to(DEV) for k in ("theta", "U", "mu")}
    late = {k: torch.zeros_like(v) for k, v in src.items()}
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)                 # some 50 ms
        for k in late:
            late[k].copy_(src[k])
    layer = kvc.Layer(14, 2, 128, shape.n, 600, torch.bfloat16, idx=p["idx"], **late)
    caps = kvc.alloc_capsules(layer, 2, 2)
    kvc.kvc_compress(layer, p["K_vis"].to(DEV), p["V_vis"].to(DEV), 2, 2, caps)
    ws = kvc.alloc_workspace(layer, 2, 2, 24)
    out = torch.full((2, 14, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    kvc.kvc_decode_attend(layer, p["q"].to(DEV), caps, 2, 2, p["K_txt"].to(DEV), p["V_txt"].to(DEV), 20, 24, out, ws)
    torch.cuda.synchronize()
    tl.assert_close(tl.np64(out), tl.oracle_run(shape, p, "fused")[2], "bf16")


@pytest.mark.parametrize("n,H_q,mode,copies", [
    (1000, 32, "kv", 0),             # one query head per KV head: three-phase kernels; rows of U start on 16 bytes
    (1000, 32, "k", 0), (1000, 32, "v", 0), (1002, 32, "k", 0), (1002, 32, "v", 1), (1002, 32, "kv", 2), (1000, 64, "kv", 1), (1024, 64, "kv", 0),
])
def test_padded_copies_only_where_a_kernel_reads_them(n, H_q, mode, copies):
    """32 KV heads of m = 400 or 401 rows: 26 MB a copy."""
    H, m = 32, kvc.kvc_retained_len(n, 600)
    par = torch.zeros((H, m, n), dtype=torch.bfloat16, device=DEV)
    mu = torch.zeros((H, 128), dtype=torch.bfloat16, device=DEV)
    torch.cuda.synchronize()
    kvc.Layer(H_q, H, 128, 64, 0, torch.bfloat16).close()            # whatever the first handle of a process loads
    before = torch.cuda.mem_get_info()[0]
    layer = kvc.Layer(H_q, H, 128, n, 600, torch.bfloat16, idx=wl.evenly_spaced_idx(n, m) if mode != "v" else None,
                      theta=par if mode != "v" else None, U=par if mode != "k" else None, mu=mu if mode != "k" else None, mode=tl.MODES[mode])
    used = before - torch.cuda.mem_get_info()[0]
    layer.close()
    copy = H * m * ((n + 63) // 64 * 64) * 2
    assert copies * copy - 1e6 <= used <= copies * copy + 6e6, used
