"""Graphs without samples of col: the instances that step from the two lists (needs a GB300).

n2v_graph_load accepts an aux buffer that lacks only the room for the samples.  Launches on such a
graph probe or stage the longer list, keep special positions in shared memory and a spill area, and
come at four register budgets; the tunings below force each of these, and the names of the launched
kernels say that they do.
"""
import numpy as np
import pytest
import torch

import oracle
from launches import captured
from paper_1805_00280_gb300 import graphs as G
from paper_1805_00280_gb300 import n2v
from small_graphs import small_graphs
from test_gpu_blocks import hub_graph
from test_gpu_serve_many import serve

pytestmark = pytest.mark.gpu

# tuning, and the blocks per SM that the launched instance is compiled for
TUNES = {
    "default": ({}, 5),
    "all_warp": (dict(thread_max_deg=0), 5),
    "all_thread": (dict(thread_max_deg=1 << 30), 5),
    "spill": (dict(thread_max_deg=0, smem_specials=32, spill_specials=64), 5),
    "chunks": (dict(chunk_walkers=1000), 5),
    "probe": (dict(thread_max_deg=0, stream_ratio=0), 5),
    "stage": (dict(thread_max_deg=0, stream_ratio=100_000, stage_window=64), 5),
    "stage4": (dict(thread_max_deg=0, stream_ratio=100_000, stage_window=64, stage_buffers=4), 5),
    "segments": (dict(thread_max_deg=0, smem_specials=32, spill_specials=0, stage_window=64, stream_ratio=100_000), 5),
    "warps16": (dict(blocks_per_sm=4), 4),
    "warps24": (dict(block_threads=256, blocks_per_sm=3), 6),
    "warps32": (dict(blocks_per_sm=8, stage_window=512), 8),
    "l2persist": (dict(l2_persist_mb=8), 5),
}


@pytest.fixture(scope="module", autouse=True)
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    n2v.lib()


def without_samples(g, **tune) -> n2v.Graph:
    """The graph, loaded again with an aux buffer one allocation unit short."""
    graph = n2v.Graph.from_csr(g, tune=n2v.default_tune(**tune))
    n2v.n2v_graph_free(graph.handle)
    need = n2v.n2v_graph_aux_bytes(graph.n, graph.nnz, graph.w is not None, graph.tune)
    graph.aux = torch.empty(need - 256, dtype=torch.uint8, device="cuda")
    graph.handle = n2v.n2v_graph_load(graph.row_ptr, graph.col, graph.w, graph.n, graph.nnz, graph.aux, graph.tune)
    return graph


def launched(graph, noalloc=False) -> set:
    """Names of the kernels that one step from every vertex launches."""
    starts = torch.arange(graph.n, dtype=torch.int32, device="cuda")
    out = torch.empty((graph.n, 2), dtype=torch.int32, device="cuda")
    ws = torch.empty(n2v.n2v_walk_ws_bytes(graph.handle, graph.n, 2, n2v.N2V_PERSISTENT) // 8 + 32, dtype=torch.int64,
                     device="cuda")
    if noalloc:
        n2v.n2v_walk_noalloc(graph.handle, starts, graph.n, 1, 2, 0.5, 2.0, 1, 0, graph.n, out)
        call = lambda s: n2v.n2v_walk_noalloc(graph.handle, starts, graph.n, 1, 2, 0.5, 2.0, 1, 0, graph.n, out, s)
    else:
        call = lambda s: n2v.n2v_walk(graph.handle, starts, graph.n, 1, 2, 0.5, 2.0, 1, 0, graph.n, out, ws,
                                      n2v.N2V_PERSISTENT, s)
    return {name for name, *_ in captured(call)}


def instance(weighted: bool, per_sm: int) -> str:
    return f"k_persistentILi{per_sm}ELi{1 if weighted else 2}E"  # 1: lean, 2: lean without weights


@pytest.mark.parametrize("kind", ["plain", "directed", "weighted"])
@pytest.mark.parametrize("tname", TUNES)
def test_hub_pairs_match_oracle(kind, tname):
    tune, per_sm = TUNES[tname]
    g = hub_graph(kind, 7)
    starts = np.arange(g.n, dtype=np.int32)
    want = oracle.walk(g.row_ptr, g.col, g.w, starts, 24, 0.25, 4.0, 3, np.arange(g.n), threads=8)
    graph = without_samples(g, **tune)
    names = launched(graph)
    assert len(names) == 1 and instance(g.w is not None, per_sm) in names.pop()
    got = n2v.walk(graph, starts, 1, 24, 0.25, 4.0, 3).cpu().numpy()
    assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
    np.testing.assert_array_equal(got, want)
    full = n2v.walk(graph, starts, 1, 24, 0.25, 4.0, 3, approx=(0.0, 64)).cpu().numpy()  # exact, by the full instance
    np.testing.assert_array_equal(full, want)
    graph.close()


@pytest.mark.parametrize("name", list(small_graphs()))
def test_small_graphs_match_oracle(name):
    g = small_graphs()[name]
    starts = np.arange(g.n, dtype=np.int32)
    for p, q in [(1.0, 1.0), (0.25, 4.0), (4.0, 0.25)]:
        want = oracle.walk(g.row_ptr, g.col, g.w, starts, 9, p, q, 5, np.arange(g.n * 37), threads=8)
        for tname, (tune, _) in TUNES.items():
            graph = without_samples(g, **tune)
            got = n2v.walk(graph, starts, 37, 9, p, q, 5).cpu().numpy()
            assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
            np.testing.assert_array_equal(got, want, err_msg=f"{tname} p={p} q={q}")
            graph.close()


def test_noalloc_specials_beyond_the_scratch_spill():
    """On K_800 a step at v from t has 799 special neighbours: more than 32 slots and the spill area that
    the 4 MiB scratch leaves a warp, so they are enumerated again segment by segment."""
    k = 800
    g = G.from_edges(k, [(i, j) for i in range(k) for j in range(i + 1, k)])
    graph = without_samples(g, smem_specials=32, thread_max_deg=0)
    names = launched(graph, noalloc=True)
    assert len(names) == 1 and instance(False, 5) in names.pop()
    _, blocks, threads = n2v.n2v_launch_shape(graph.handle)  # (what these instances launch)
    assert k - 1 > 32 + ((4 << 20) - 4096) // 4 // (blocks * threads // 32)
    starts = torch.arange(k, dtype=torch.int32, device="cuda")
    want = oracle.walk(g.row_ptr, g.col, None, np.arange(k, dtype=np.int32), 12, 0.5, 2.0, 31, np.arange(3 * k), threads=8)
    for _ in range(2):
        out = torch.full((3 * k, 12), -7, dtype=torch.int32, device="cuda")
        n2v.n2v_walk_noalloc(graph.handle, starts, k, 3, 12, 0.5, 2.0, 31, 0, 3 * k, out)
        assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
        np.testing.assert_array_equal(out.cpu().numpy(), want)
    graph.close()


@pytest.mark.parametrize("kind", ["plain", "weighted"])
@pytest.mark.parametrize("tune", [{}, dict(thread_max_deg=0, stage_window=64, stream_ratio=100_000), dict(hub_count=64)])
def test_serving_mix_matches_oracle(kind, tune):
    g = hub_graph(kind, 7)
    graph = without_samples(g, **tune)
    rng = np.random.default_rng(4)
    jobs = [(rng.integers(0, g.n, int(np.exp(rng.uniform(0, 6)))).astype(np.int32), 1 + j % 17, 0.5, 0.25 + j % 3,
             100 + j) for j in range(60)]
    rows, _ = serve(graph, jobs)
    for got, (starts, l, p, q, seed) in zip(rows, jobs):
        want = oracle.walk(g.row_ptr, g.col, g.w, starts, l, p, q, seed, np.arange(len(starts)), threads=8)
        np.testing.assert_array_equal(got.cpu().numpy(), want)
    assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
    graph.close()
