"""Sampled-block steps on input that the other tests do not have (needs a GB300).

col on 16 bytes, as the C ABI asks, but not on 32, so that every block of eight entries lies across
two 32-byte sectors; and weighted graphs with self-loops.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1805_00280_gb300 import graphs as G
from paper_1805_00280_gb300 import n2v
from test_gpu_blocks import hub_graph

pytestmark = pytest.mark.gpu

TUNES = [{}, dict(thread_max_deg=0), dict(thread_max_deg=0, smem_specials=32)]


@pytest.fixture(scope="module", autouse=True)
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    n2v.lib()


def check(g, graph, p, q):
    starts = np.arange(g.n, dtype=np.int32)
    want = oracle.walk(g.row_ptr, g.col, g.w, starts, 24, p, q, 3, np.arange(g.n), threads=8)
    got = n2v.walk(graph, starts, 1, 24, p, q, 3).cpu().numpy()
    assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
    np.testing.assert_array_equal(got, want)
    graph.close()


@pytest.mark.parametrize("kind", ["plain", "directed", "weighted"])
@pytest.mark.parametrize("tune", TUNES)
def test_col_on_16_bytes(kind, tune):
    g = hub_graph(kind, 7)
    room = torch.empty(g.nnz + 4, dtype=torch.int32, device="cuda")
    col = room[4:]
    col.copy_(torch.from_numpy(g.col))
    graph = n2v.Graph(torch.from_numpy(g.row_ptr), col, g.w, n2v.default_tune(**tune))
    assert graph.col.data_ptr() % 32 == 16
    check(g, graph, 0.25, 4.0)


@pytest.mark.parametrize("p,q", [(0.25, 4.0), (3.0, 0.4), (0.5, 1.0)])
@pytest.mark.parametrize("tune", TUNES)
def test_weighted_self_loops(p, q, tune):
    d = hub_graph("directed", 7)
    rng = np.random.default_rng(3)
    loops = np.repeat(np.arange(d.n), np.diff(d.row_ptr)) == d.col
    assert loops.sum() >= 5
    w = rng.integers(0, 10, d.nnz).astype(np.uint32)
    w[loops] = 500
    g = G.CSR(d.row_ptr, d.col, w, "weighted loops")
    check(g, n2v.Graph.from_csr(g, tune=n2v.default_tune(**tune)), p, q)
