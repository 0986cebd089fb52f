"""The typed views of a capsule store: the same memory, shapes and strides whatever the byte buffer they are taken of (as large as the store,
larger, with an odd number of bytes, part of another buffer)."""
import pytest
import torch

from paper_2605_16439_b200 import binding as kvc
from paper_2605_16439_b200 import build as kvc_build
from paper_2605_16439_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("extra,skip", [(0, 0), (64, 0), (1, 0), (32, 16)])
@pytest.mark.parametrize("mode", [kvc.KVC_MODE_KV, kvc.KVC_MODE_V_ONLY])
def test_capsule_views(dtype, extra, skip, mode):
    kvc_build.build()
    B, H_kv, R, n = 2, 3, 2, 9
    m = kvc.kvc_retained_len(n, 600)
    U = torch.zeros((H_kv, m, n), dtype=dtype, device="cuda")
    both = dict(idx=wl.evenly_spaced_idx(n, m), theta=U) if mode == kvc.KVC_MODE_KV else {}
    layer = kvc.Layer(6, H_kv, 128, n, 600, dtype, U=U, mu=torch.zeros((H_kv, 128), dtype=dtype, device="cuda"), mode=mode, **both)
    total = kvc.kvc_capsule_bytes(layer, B, R)
    store = torch.arange(total + extra + skip, device="cuda").to(torch.uint8)[skip:]
    K, V = kvc.capsule_views(layer, store, B, R)
    kb = B * H_kv * R * layer.m_k * 128 * dtype.itemsize
    for t, rows, at, end in ((K, layer.m_k, 0, kb), (V, layer.m_v, kb, total)):
        assert t.shape == (B, H_kv, R, rows, 128) and t.is_contiguous() and t.dtype == dtype
        assert t.data_ptr() == store.data_ptr() + at
        assert torch.equal(t.view(torch.uint8).flatten(), store[at:end])
