"""The typed views of a capsule store under tracing: a graph recorded on one store reads the store it is called with, wherever that lies in
its buffer, and the views can be compiled without a break."""
import types

import pytest
import torch
from torch.fx.experimental.proxy_tensor import make_fx

from paper_2605_16439_b200 import binding as kvc

B, R = 2, 2
LAYER = types.SimpleNamespace(m_k=3, m_v=5, d=128, H_kv=2, dtype=torch.bfloat16)
PARTS = [(B, 2, R, rows, 128) for rows in (3, 5)]
TOTAL = sum(torch.Size(p).numel() for p in PARTS) * 2


def _views(store):
    return kvc.capsule_views(LAYER, store, B, R)


def _want(store):
    kb = torch.Size(PARTS[0]).numel() * 2
    return store[:kb].view(torch.bfloat16).view(PARTS[0]), store[kb:TOTAL].view(torch.bfloat16).view(PARTS[1])


@pytest.fixture
def raw():
    return torch.randn(3 * TOTAL // 2, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16).view(torch.uint8)


@pytest.mark.parametrize("recorded,called", [(0, TOTAL), (256, 0), (TOTAL, TOTAL + 512)])
def test_a_recorded_graph_reads_the_store_it_is_given(raw, recorded, called):
    graph = make_fx(_views)(raw[recorded:recorded + TOTAL])
    store = raw[called:called + TOTAL]
    for got, want in zip(graph(store), _want(store)):
        assert torch.equal(got, want)


def test_views_compile_in_one_graph(raw):
    store = raw[256:256 + TOTAL]
    for got, want in zip(torch.compile(lambda s: [x + 0 for x in _views(s)], backend="eager", fullgraph=True)(store), _want(store)):
        assert torch.equal(got, want)
