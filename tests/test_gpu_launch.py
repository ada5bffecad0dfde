"""Which kernel a call launches, and on how many blocks (needs a GB300)."""
import numpy as np
import pytest
import torch

from launches import captured
from paper_1805_00280_gb300 import graphs as G
from paper_1805_00280_gb300 import n2v

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    n2v.lib()


@pytest.fixture(scope="module")
def rmat14():
    return G.rmat(14, 16, 0.57, 0.19, 0.19, 3)


def launches(graph, walks, l=10, q=2.0, noalloc=False):
    starts = torch.arange(walks, dtype=torch.int32, device="cuda") % graph.n
    out = torch.empty((walks, l), dtype=torch.int32, device="cuda")
    if noalloc:  # (the first call on a device looks up its scratch, which no capture may hold)
        n2v.n2v_walk_noalloc(graph.handle, starts, walks, 1, l, 0.5, q, 3, 0, walks, out)
        return captured(lambda s: n2v.n2v_walk_noalloc(graph.handle, starts, walks, 1, l, 0.5, q, 3, 0, walks, out, s))
    ws = torch.empty(n2v.n2v_walk_ws_bytes(graph.handle, walks, l, n2v.N2V_PERSISTENT) // 8 + 32, dtype=torch.int64,
                     device="cuda")
    return captured(lambda s: n2v.n2v_walk(graph.handle, starts, walks, 1, l, 0.5, q, 3, 0, walks, out, ws,
                                           n2v.N2V_PERSISTENT, s))


@pytest.mark.parametrize("weighted", [False, True])
def test_the_grid_follows_the_walkers_of_one_launch(rmat14, weighted):
    """Few walkers and many take different instances; a call in chunks counts one chunk's, and the
    call without a workspace counts as the other one does."""
    g = G.with_weights(rmat14, 2, 1, 100) if weighted else rmat14
    graph, chunked = n2v.Graph.from_csr(g), n2v.Graph.from_csr(g, tune=n2v.default_tune(chunk_walkers=100))
    few, many = launches(graph, 100), launches(graph, 16_000)
    assert len(few) == len(many) == 1 and few != many
    for _ in range(2):
        assert launches(graph, 100, noalloc=True) == few
        assert launches(graph, 16_000, noalloc=True) == many
    for noalloc in (False, True):
        assert launches(chunked, 16_000, noalloc=noalloc) == few * 160
    graph.close()
    chunked.close()
