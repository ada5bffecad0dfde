"""What this library is asked to do, as measured cases.

Each case is one job as a user's program runs it on a graph that stays on the GPU: a call of
``n2v.walk``, rows streamed to the host by ``n2v.walk_to_host``, or a mix of jobs through
``n2v.Server``.  The graphs are those of the workloads in ``paper_1805_00280_gb300.graphs`` (and
smaller ones of the same kinds): Erdos-Renyi, R-MAT with the social-network skew, and the Skew-S and
WeC-K sweeps, drawn here on the GPU so that they are quick to make.
"""
import math

import numpy as np
import torch

from paper_1805_00280_gb300 import n2v

# R-MAT quadrant probabilities (a, b, c) of the graph kinds
ABC = {
    "rmat": (0.57, 0.19, 0.19),  # social networks
    "skew5": (0.5 / 6.0, 0.25, 0.25),  # Skew-5: b = c = 0.25, d = 5 a
    "skew3": (0.5 / 4.0, 0.25, 0.25),
    "wec": (0.18, 0.25, 0.25),  # WeC-K: flat degrees
}


def _walk(name, graph, scale, ef, walks, l, p, q, **more):
    c = {"name": name, "call": "walk", "graph": graph, "scale": scale, "ef": ef, "weighted": False,
         "walks": walks, "r": 1, "l": l, "p": p, "q": q, "cuda_graph": False, "eps": -1.0, "popular": 0}
    c.update(more)
    return c


def listed():
    return [
        # a query for a few short walks on a small graph: what one call costs at least
        _walk("er_few", "er", 0, 0, 50, 10, 0.5, 2.0),
        # the Erdos-Renyi workload as it stands: every vertex ten times, short lists everywhere
        _walk("er_all", "er", 0, 0, 10_000, 80, 0.5, 2.0, r=10),
        # walks for one mini-batch of vertices of a social graph: few walkers, long lists
        _walk("rmat20_batch", "rmat", 20, 16, 999, 40, 0.25, 4.0),
        # p = q = 1, the first-order walk (DeepWalk), from every vertex
        _walk("rmat20_first_order", "rmat", 20, 16, 1 << 20, 80, 1.0, 1.0),
        # in-out parameter below 1 from every vertex of the same graph
        _walk("rmat20_p4", "rmat", 20, 16, 1 << 20, 80, 4.0, 0.25),
        # weighted edges, a graph beyond L2, a ragged number of starts
        _walk("rmat23_weighted", "rmat", 23, 16, 300_001, 80, 1.0, 0.5, weighted=True),
        # the largest: a graph many times L2, walks in rounds recorded as a CUDA graph
        _walk("rmat24_rounds", "rmat", 24, 16, 1 << 19, 80, 2.0, 0.5, cuda_graph=True),
        # the synthetic sweeps: flat degrees around 100, and a strong skew
        _walk("wec20", "wec", 20, 50, 1 << 19, 80, 0.5, 2.0),
        _walk("skew5", "skew5", 22, 50, 400_000, 80, 0.5, 2.0),
        # approximate walks at popular vertices (FN-Approx)
        _walk("rmat20_approx", "rmat", 20, 16, 1 << 18, 80, 0.5, 2.0, eps=1e-3, popular=1024),
        # rows streamed to host memory through a device ring
        _walk("rmat22_to_host", "rmat", 22, 16, 1 << 18, 40, 2.0, 0.5, call="to_host"),
        # serving: jobs of uneven size, length, p and q against one resident graph
        _walk("rmat22_serve", "rmat", 22, 16, 1 << 15, 80, 0.0, 0.0, call="serve", jobs=40),
    ]


def draw(rng):
    """One more case: the same calls, options and kinds of graph over their whole range of sizes."""
    kind = rng.choice(["er", "rmat", "rmat", "rmat", "wec", "skew3", "skew5"])
    call = rng.choice(["walk", "walk", "walk", "walk", "to_host", "serve"])
    scale = 0 if kind == "er" else rng.randint(12, 22 if kind == "rmat" else 20)
    ef = 0 if kind == "er" else (16 if kind == "rmat" else 50)
    l = rng.choice([1, 5, 10, 20, 37, 40, 80, 80, 100])
    most = 16e6 if kind == "rmat" else 32e6  # steps: below the largest listed case's
    walks = int(round(math.exp(rng.uniform(math.log(1), math.log(most / l)))))
    walks = max(1, min(walks, 1 << 20))
    p, q = (round(math.exp(rng.uniform(math.log(0.25), math.log(4.0))), 3) for _ in range(2))
    if rng.random() < 0.2:
        q = 1.0
    if call == "serve":
        walks = max(1, min(walks, 1 << 14))
        return _walk("", kind, scale, ef, walks, 80, 0.0, 0.0, call="serve", jobs=rng.randint(1, 30),
                     weighted=rng.random() < 0.25)
    eps = 1e-3 if call == "walk" and rng.random() < 0.15 else -1.0
    return _walk("", kind, scale, ef, walks, l, p, q, call=call, weighted=rng.random() < 0.25,
                 cuda_graph=call == "walk" and eps < 0 and rng.random() < 0.25, eps=eps,
                 popular=rng.choice([64, 256, 1024]) if eps >= 0 else 0)


# --------------------------------------------------------------------------
# inputs

ER_N, ER_M = 10_000, 100_000


def _edges(case, gen):
    """Undirected edges (u, v) as int64 tensors; duplicates and self-loops are dropped later."""
    if case["graph"] == "er":
        u = torch.randint(0, ER_N, (ER_M,), generator=gen, device="cuda")
        v = torch.randint(0, ER_N, (ER_M,), generator=gen, device="cuda")
        return ER_N, u, v
    a, b, c = ABC[case["graph"]]
    n = 1 << case["scale"]
    m = n * case["ef"]
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(case["scale"]):  # one quadrant per bit, from the most significant down
        x = torch.rand(m, generator=gen, device="cuda")
        down = x >= a + b
        right = ((x >= a) & ~down) | (x >= a + b + c)
        u.mul_(2).add_(down)
        v.mul_(2).add_(right)
    return n, u, v


def _csr(case, seed):
    """(row_ptr, col, w or None): symmetric, sorted, without duplicates or self-loops, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, u, v = _edges(case, gen)
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.cat([u * n + v, v * n + u])
    del u, v, keep
    key = torch.sort(key)[0]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    key = key[first]
    del first
    row_ptr = torch.searchsorted(key, torch.arange(n + 1, dtype=torch.int64, device="cuda") * n)
    w = None
    if case["weighted"]:  # symmetric weights in [1, 100]
        x, y = key // n, key % n
        h = (torch.minimum(x, y) * 0x9E3779B1 + torch.maximum(x, y) * 0x85EBCA77 + int(seed)) & 0x7FFFFFFF
        h = (h * 0x27D4EB2F) >> 13
        w = (1 + h % 100).to(torch.int32)
        del x, y, h
    col = (key % n).to(torch.int32)
    return n, row_ptr, col, w


def prepare(case, seed):
    n, row_ptr, col, w = _csr(case, seed)
    graph = n2v.Graph(row_ptr, col, w, tune=n2v.default_tune(chunk_walkers=1 << 18) if case["cuda_graph"] else None)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    walks = case["walks"]
    state = {"case": case, "graph": graph, "seed": int(seed) * 1_000_003 + 17}
    if case["call"] == "serve":
        rng = np.random.default_rng(int(seed) + 2)
        mix = np.random.default_rng(case["jobs"])  # the jobs' sizes and lengths belong to the case
        jobs = []
        for j in range(case["jobs"]):
            size = int(round(math.exp(mix.uniform(0.0, math.log(max(walks, 2))))))
            length = int(mix.choice([10, 20, 40, 80]))
            p, q = np.exp(rng.uniform(math.log(0.25), math.log(4.0), 2))
            jobs.append((rng.integers(0, n, max(1, min(size, walks))).astype(np.int32), length, float(p), float(q),
                         int(seed) + j))
        state["jobs"] = jobs
        state["server"] = n2v.Server(graph, 1 << 30)
        return state
    if walks >= n:  # every vertex, in order
        starts = torch.arange(n, dtype=torch.int32, device="cuda").repeat((walks + n - 1) // n)[:walks].contiguous()
    else:
        starts = torch.randint(0, n, (walks,), generator=gen, device="cuda", dtype=torch.int32)
    state["starts"] = starts
    if case["call"] == "to_host":
        state["out"] = torch.empty((walks * case["r"], case["l"]), dtype=torch.int32).pin_memory()
    if case["cuda_graph"]:  # a recorded call has its own stream and keeps its buffers
        state["stream"] = torch.cuda.Stream()
        state["out"] = torch.empty((walks * case["r"], case["l"]), dtype=torch.int32, device="cuda")
        need = n2v.n2v_walk_ws_bytes(graph.handle, walks * case["r"], case["l"], n2v.N2V_PERSISTENT)
        state["ws"] = torch.empty(need // 8 + 32, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
    return state


# --------------------------------------------------------------------------
# one pass

def _serve(state):
    server, left, rows = state["server"], {}, [None] * len(state["jobs"])
    for i, (starts, l, p, q, seed) in enumerate(state["jobs"]):
        left[server.submit(starts, l, p, q, seed)] = i
    while left:
        server.step()
        for jid in server.poll():
            rows[left.pop(jid)] = server.rows(jid).clone()
            server.release(jid)
    return rows


def run(state):
    case, graph = state["case"], state["graph"]
    if case["call"] == "serve":
        return _serve(state)
    job = (graph, state["starts"], case["r"], case["l"], case["p"], case["q"], state["seed"])
    if case["call"] == "to_host":
        ring = max(1, min(1 << 16, case["walks"] * case["r"]))
        return n2v.walk_to_host(*job, ring_walks=ring, out=state["out"])
    if case["cuda_graph"]:
        here = torch.cuda.current_stream()
        state["stream"].wait_stream(here)
        n2v.walk(*job, out=state["out"], ws=state["ws"], stream=state["stream"], cuda_graph=True)
        here.wait_stream(state["stream"])
        return state["out"]
    return n2v.walk(*job, approx=(case["eps"], case["popular"]) if case["eps"] >= 0 else None)


def work(case):
    """The graph's bytes, or what the steps can touch of it where that is less, the starts and the rows."""
    n = ER_N if case["graph"] == "er" else 1 << case["scale"]
    nnz = 2 * ER_M if case["graph"] == "er" else 2 * case["ef"] * n
    walks, l = case["walks"] * case["r"], case["l"]
    if case["call"] == "serve":  # log-uniform job sizes in [1, walks], lengths 10, 20, 40, 80
        walks, l = max(1, int(case["jobs"] * walks / math.log(max(walks, 3)))), 37
    entry = 8 if case["weighted"] else 4
    touched = walks * l * (16 + entry * nnz / n)
    return {"bytes": min(8 * n + entry * nnz, touched) + 4 * walks + 4 * walks * l, "flops": 0}


# --------------------------------------------------------------------------
# the rows themselves, in Python integers, for the smallest jobs

def _draw(seed, walk, k):
    x = [k, walk & 0xFFFFFFFF, walk >> 32, 0]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        m0, m1 = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [(m1 >> 32) ^ x[1] ^ k0, m1 & 0xFFFFFFFF, (m0 >> 32) ^ x[3] ^ k1, m0 & 0xFFFFFFFF]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return (x[1] << 32) | x[0]


def exact(case, seed):
    walks, l = case["walks"] * case["r"], case["l"]
    if case["call"] != "walk" or case["eps"] >= 0 or walks * l > 2000:
        return None
    n, row_ptr, col, w = _csr(case, seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    if case["walks"] >= n:
        starts = np.arange(case["walks"]) % n
    else:
        starts = torch.randint(0, n, (case["walks"],), generator=gen, device="cuda", dtype=torch.int32).cpu().numpy()
    rp, col = row_ptr.cpu().numpy(), col.cpu().numpy()
    w = None if w is None else w.cpu().numpy()
    ap, aq = (int(np.rint(65536.0 / case[x])) for x in ("p", "q"))
    key = int(seed) * 1_000_003 + 17
    out = np.full((walks, l), -1, dtype=np.int32)
    for i in range(walks):
        t, v = -1, int(starts[i % len(starts)])
        for k in range(l):
            nv = col[rp[v]:rp[v + 1]]
            wt = np.ones(len(nv), dtype=np.uint64) if w is None else w[rp[v]:rp[v + 1]].astype(np.uint64)
            if k:
                a = np.where(nv == t, ap, np.where(np.isin(nv, col[rp[t]:rp[t + 1]]), 65536, aq))
                wt = wt * a.astype(np.uint64)
            c = np.cumsum(wt)
            if len(c) == 0 or c[-1] == 0:
                break
            r = (_draw(key, i, k) * int(c[-1])) >> 64
            t, v = v, int(nv[np.searchsorted(c, r, side="right")])
            out[i, k] = v
    return out
