"""Serving many small jobs (needs a GB300).

The jobs of a tick run side by side on whichever instance the graph's tuning takes: with hashed
neighbour sets or the merge form (steps from the two lists), through sampled blocks (R-MAT), and
with most steps on lanes (Erdos-Renyi).  Job sizes lie around the 32 walkers of a warp.
"""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_1805_00280_gb300 import graphs as G
from paper_1805_00280_gb300 import n2v

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    n2v.lib()


def serve(graph, jobs) -> tuple[list, float]:
    """Every job's rows, and the seconds from the first tick to the last row."""
    server = n2v.Server(graph, 1 << 28)
    left = {server.submit(*job): i for i, job in enumerate(jobs)}
    rows = [None] * len(jobs)
    torch.cuda.synchronize()
    t0, t1 = time.perf_counter(), 0.0
    while left:
        server.step()
        for jid in server.poll():
            t1 = time.perf_counter()
            rows[left.pop(jid)] = server.rows(jid).clone()
            server.release(jid)
    server.close()
    return rows, t1 - t0


@pytest.mark.parametrize("tune", [dict(hub_count=64), dict(merge_ratio=10)])
def test_one_walk_jobs_run_side_by_side(tune):
    """A step's time is the whole warp's, so 32 jobs of one walk each on one warp would take about
    the time of one job 32 times over; on warps of their own they take about that of one."""
    g = G.rmat(16, 16, 0.57, 0.19, 0.19, 5)
    graph = n2v.Graph.from_csr(g, tune=n2v.default_tune(**tune))
    rng = np.random.default_rng(0)
    jobs = [(rng.integers(0, g.n, 1).astype(np.int32), 80, 0.5, 2.0, 100 + j) for j in range(32)]
    serve(graph, jobs)
    alone = max(min(serve(graph, [job])[1] for _ in range(2)) for job in jobs)
    together = min(serve(graph, jobs)[1] for _ in range(5))
    assert together < 6 * alone, f"32 jobs {1e3 * together:.2f} ms, the longest of them alone {1e3 * alone:.2f} ms"
    graph.close()


@pytest.mark.parametrize("kind", ["er", "rmat"])
@pytest.mark.parametrize("tune", [{}, dict(hub_count=64), dict(merge_ratio=10)])
@pytest.mark.parametrize("count,size", [(1, 1), (700, 1), (300, 31), (40, 32), (40, 33), (300, 200), (3, 30_000)])
def test_rows_of_many_jobs(kind, tune, count, size):
    g = G.er(5000, 50_000, 2) if kind == "er" else G.rmat(12, 16, 0.57, 0.19, 0.19, 5)
    graph = n2v.Graph.from_csr(g, tune=n2v.default_tune(**tune))
    rng = np.random.default_rng(size)
    jobs = [(rng.integers(0, g.n, size).astype(np.int32), 1 + j % 13, 0.5, 2.0 if j % 3 else 1.0, 100 + j)
            for j in range(count)]
    rows, _ = serve(graph, jobs)
    for i in range(0, count, 1 + count // 25):
        starts, l, p, q, seed = jobs[i]
        ids = np.arange(size) if size < 1000 else np.arange(0, size, 97)
        want = oracle.walk(g.row_ptr, g.col, None, starts, l, p, q, seed, ids, threads=8)
        np.testing.assert_array_equal(rows[i].cpu().numpy()[ids], want, err_msg=f"job {i}")
    assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
    graph.close()
