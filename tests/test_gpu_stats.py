"""The stats build counts each step under the way it was taken (needs a GB300).

On a complete bipartite graph every step after the first is at one side from the other, so the
lengths of both lists, the keys and the search are known for every step.
"""
import json
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

REPO = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import json, sys
import numpy as np
from paper_1805_00280_gb300 import graphs as G, n2v
x, y, weighted = (int(a) for a in sys.argv[1:])
a, b = (m.ravel() for m in np.meshgrid(np.arange(x), np.arange(x, x + y), indexing="ij"))
row_ptr = np.concatenate([np.arange(x) * y, x * y + np.arange(y + 1) * x]).astype(np.int64)
col = np.concatenate([b, np.tile(np.arange(x), y)]).astype(np.int32)
w = (1 + np.arange(len(col)) % 9).astype(np.uint32) if weighted else None
graph = n2v.Graph.from_csr(G.CSR(row_ptr, col, w, "bipartite"))
n2v.n2v_step_stats(reset=True)
n2v.walk(graph, np.arange(x + y, dtype=np.int32), 1, 11, 0.5, 2.0, 3)
print(json.dumps(n2v.n2v_step_stats()))
"""


# x vertices of y neighbours and y of x; the mode of a step at one of the x and at one of the y:
# 0, 1 searched in global memory and 3, 2 in staged samples, by keys N(v), N(t)
@pytest.mark.parametrize("x,y,weighted,at_x,at_y", [
    (70, 100, 1, 2, 3),   # more than a weighted batch (64 keys): the shorter list gives the keys
    (70, 100, 0, 3, 3),   # one batch (128 keys): N(v) does
    (70, 3000, 1, 1, 0),  # weighted, beyond the ratio whose samples are staged
    (70, 3000, 0, 2, 3),  # top samples staged
])
def test_steps_are_counted_by_the_way_they_were_taken(x, y, weighted, at_x, at_y):
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    r = subprocess.run([sys.executable, "-c", CODE, str(x), str(y), str(weighted)], cwd=REPO,
                       env=dict(os.environ, N2V_STATS="1"), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-3000:]
    got = json.loads(r.stdout.strip().splitlines()[-1])
    want = {f"mode{m}_{f}": 0 for m in range(5) for f in ("steps", "short_sum", "long_sum")}
    for m, dv, dt in ((at_x, y, x), (at_y, x, y)):  # ten steps a walk, five at either side
        steps, keys = 5 * (x + y), dv if m in (0, 3) else dt
        want[f"mode{m}_steps"] += steps
        want[f"mode{m}_short_sum"] += steps * keys
        want[f"mode{m}_long_sum"] += steps * (dv + dt - keys)
    assert {k: got[k] for k in want} == want
