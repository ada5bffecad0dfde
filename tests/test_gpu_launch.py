"""Which kernel a call launches, and on how many blocks (needs a GB300)."""
import numpy as np
import pytest
import torch

import oracle
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


@pytest.mark.parametrize("walks", [1, 33, 5000, 200_001])
def test_jobs_of_one_step_stay_on_lanes(rmat14, walks):
    """The first step does not read N(t): a job of one step is launched as a job at q = 1 is, whatever
    the graph's degrees, and its rows are the oracle's."""
    graph = n2v.Graph.from_csr(rmat14)
    assert launches(graph, walks, l=1) == launches(graph, walks, l=1, q=1.0) == launches(graph, walks, q=1.0)
    starts = np.arange(walks, dtype=np.int32) % rmat14.n
    got = n2v.walk(graph, starts, 1, 1, 0.5, 2.0, 3).cpu().numpy()
    want = oracle.walk(rmat14.row_ptr, rmat14.col, None, starts, 1, 0.5, 2.0, 3, np.arange(walks), threads=8)
    np.testing.assert_array_equal(got, want)
    graph.close()
