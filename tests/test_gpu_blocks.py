"""The step through sampled blocks (n2v_blocks.cuh) against the oracle, at the sizes where it can go wrong.

Hubs whose lists have lengths around a chunk (32 keys), a batch (128), the staged samples (64, 128
and 512 of every eighth entry) and the records, joined to each other and to leaves that know only
hubs: a walk meets every pair of them as (t, v), with the longer list on either side.  Rows start and
end inside blocks, and the last row ends col inside one.  Walks are integers: rows must be equal.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1805_00280_gb300 import graphs as G
from paper_1805_00280_gb300 import n2v

pytestmark = pytest.mark.gpu

DEGREES = [2, 3, 5, 9, 31, 33, 64, 65, 100, 127, 129, 200, 255, 257, 500, 513, 1000, 1025, 1500, 2049, 3000, 4097,
           6000, 9000, 11000]


@pytest.fixture(scope="module", autouse=True)
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    n2v.lib()


def hub_graph(kind: str, seed: int) -> G.CSR:
    """Hubs of the given degrees over 12,007 vertices; directed: half the leaves' edges have no way
    back, and every third hub has a self-loop; weighted: weights 0 .. 9, and one of 2^32 - 1."""
    rng = np.random.default_rng(seed)
    n = 12_007
    hubs = np.concatenate([[0, n - 1], np.sort(rng.choice(np.arange(1, n - 1), len(DEGREES) - 2, replace=False))])
    degs = np.array(DEGREES)[rng.permutation(len(DEGREES))]
    leaves = np.setdiff1d(np.arange(n), hubs)
    src, dst = [], []
    for h, d in zip(hubs, degs):
        first = rng.integers(0, len(leaves))
        run = leaves[first:first + d // 4]  # a run of neighbouring ids beside the scattered ones
        pick = np.unique(np.concatenate([run, rng.choice(leaves, d, replace=False)]))[:d]
        src.append(np.full(len(pick), h))
        dst.append(pick)
    src, dst = np.concatenate(src), np.concatenate(dst)
    back = np.ones(len(src), bool) if kind != "directed" else rng.random(len(src)) < 0.5
    hs, hd = (a.ravel() for a in np.meshgrid(hubs, hubs))
    keep = hs != hd if kind != "directed" else (hs != hd) | (hs % 3 == 0)
    a, b = leaves[0], leaves[1]
    e = np.concatenate([src * n + dst, dst[back] * n + src[back], hs[keep] * n + hd[keep], [a * n + b, b * n + a]])
    e = np.unique(e)
    row_ptr = np.searchsorted(e, np.arange(n + 1) * n).astype(np.int64)
    w = None
    if kind == "weighted":
        w = rng.integers(0, 10, len(e)).astype(np.uint32)
        w[rng.integers(0, len(e))] = 2**32 - 1
    return G.CSR(row_ptr, (e % n).astype(np.int32), w, kind)


def check(g, tunes, p, q):
    starts = np.arange(g.n, dtype=np.int32)
    ids = np.arange(g.n)
    want = oracle.walk(g.row_ptr, g.col, g.w, starts, 24, p, q, 3, ids, threads=8)
    assert (want[:, -1] >= 0).any()
    for tune in tunes:
        graph = n2v.Graph.from_csr(g, tune=n2v.default_tune(**tune))
        got = n2v.walk(graph, starts, 1, 24, p, q, 3).cpu().numpy()
        assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK
        np.testing.assert_array_equal(got, want, err_msg=f"{g.name} {tune} p={p} q={q}")
        graph.close()


@pytest.mark.parametrize("kind", ["plain", "directed", "weighted"])
@pytest.mark.parametrize("p,q", [(0.25, 4.0), (3.0, 0.4), (0.5, 1.0), (1.0, 1.0)])
def test_hub_pairs_match_oracle(kind, p, q):
    g = hub_graph(kind, 7)
    assert g.nnz % 8 != 0  # the last block of col is cut
    tunes = [{}, dict(thread_max_deg=0), dict(thread_max_deg=0, smem_specials=32), dict(thread_max_deg=1 << 20),
             dict(blocks_per_sm=8, smem_specials=8192)]
    check(g, tunes if (p, q) == (0.25, 4.0) else tunes[:2], p, q)


@pytest.mark.parametrize("walks", [1, 31, 33, 3039, 12_007])
def test_small_jobs_are_spread_over_the_warps(walks):
    """Fewer walkers than warps, and counts that leave the last warps a part of a batch."""
    g = hub_graph("plain", 8)
    starts = np.arange(walks, dtype=np.int32)
    want = oracle.walk(g.row_ptr, g.col, g.w, starts, 12, 2.0, 0.5, 9, np.arange(walks), threads=8)
    graph = n2v.Graph.from_csr(g)
    for ranged in ((0, walks), (walks // 3, walks - walks // 3)):
        got = n2v.walk(graph, starts, 1, 12, 2.0, 0.5, 9, walk_begin=ranged[0], walk_count=ranged[1]).cpu().numpy()
        np.testing.assert_array_equal(got, want[ranged[0]:ranged[0] + ranged[1]])
    assert n2v.n2v_stream_status(graph.handle) == n2v.N2V_OK


@pytest.mark.parametrize("kind", ["plain", "weighted"])
def test_an_aux_without_room_for_the_samples_still_walks(kind):
    """An aux buffer that holds everything but the samples of col is accepted; such a graph takes the
    instances that step from the two lists."""
    g = hub_graph(kind, 9)
    starts = np.arange(g.n, dtype=np.int32)
    row_ptr, col = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col).cuda()
    w = None if g.w is None else torch.from_numpy(g.w.view(np.int32)).cuda()
    need = n2v.n2v_graph_aux_bytes(g.n, g.nnz, g.weighted)
    aux = torch.empty(need - 4 * (g.nnz // 8), dtype=torch.uint8, device="cuda")
    h = n2v.n2v_graph_load(row_ptr, col, w, g.n, g.nnz, aux)
    ws = torch.empty(n2v.n2v_walk_ws_bytes(h, g.n, 24, n2v.N2V_PERSISTENT), dtype=torch.uint8, device="cuda")
    out = torch.empty((g.n, 24), dtype=torch.int32, device="cuda")
    n2v.n2v_walk(h, torch.from_numpy(starts).cuda(), g.n, 1, 24, 0.5, 2.0, 3, 0, g.n, out, ws, n2v.N2V_PERSISTENT)
    assert n2v.n2v_stream_status(h) == n2v.N2V_OK
    want = oracle.walk(g.row_ptr, g.col, g.w, starts, 24, 0.5, 2.0, 3, np.arange(g.n), threads=8)
    np.testing.assert_array_equal(out.cpu().numpy(), want)
    n2v.n2v_graph_free(h)
    with pytest.raises(n2v.N2VError):  # less than that is refused
        n2v.n2v_graph_load(row_ptr, col, w, g.n, g.nnz, aux[:256])
