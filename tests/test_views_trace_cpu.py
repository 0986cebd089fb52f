"""The typed views of a capsule store under tracing: a graph recorded on one store reads the store it is called with, wherever that lies in
its buffer, and the views can be compiled without a break."""
import types

import pytest
import torch
from torch.fx.experimental.proxy_tensor import make_fx

from paper_2605_16439_b200 import binding as kvc

B, R = 2, 2
ROWS = pytest.mark.parametrize("rows", [(3, 5), (4, 4)])         # retained rows of a block on the key and the value side
TOTAL = B * 2 * R * 8 * 128 * 2


def _views(rows):
    layer = types.SimpleNamespace(m_k=rows[0], m_v=rows[1], d=128, H_kv=2, dtype=torch.bfloat16)
    return lambda store: kvc.capsule_views(layer, store, B, R)


def _want(rows, store):
    kb = B * 2 * R * rows[0] * 128 * 2
    return [x.view(torch.bfloat16).view(B, 2, R, m, 128) for x, m in zip((store[:kb], store[kb:TOTAL]), rows)]


@pytest.fixture
def raw():
    return torch.randn(3 * TOTAL // 2, generator=torch.Generator().manual_seed(3)).to(torch.bfloat16).view(torch.uint8)


@ROWS
@pytest.mark.parametrize("recorded,called", [(0, TOTAL), (256, 0), (TOTAL, TOTAL + 512)])
def test_a_recorded_graph_reads_the_store_it_is_given(raw, recorded, called, rows):
    graph = make_fx(_views(rows))(raw[recorded:recorded + TOTAL])
    store = raw[called:called + TOTAL]
    for got, want in zip(graph(store), _want(rows, store)):
        assert torch.equal(got, want)


@ROWS
def test_views_compile_in_one_graph(raw, rows):
    store, views = raw[256:256 + TOTAL], _views(rows)
    for got, want in zip(torch.compile(lambda s: [x + 0 for x in views(s)], backend="eager", fullgraph=True)(store), _want(rows, store)):
        assert torch.equal(got, want)


@ROWS
def test_views_share_the_store(raw, rows):
    store = raw[256:256 + TOTAL].clone()
    for x in _views(rows)(store):
        x.fill_(1.5)
    assert (store.view(torch.bfloat16) == 1.5).all()
