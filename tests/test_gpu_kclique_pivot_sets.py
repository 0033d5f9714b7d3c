"""Pivoting on candidate sets of more than 64 vertices whose pivot has many non-neighbours (GPU).

Such a node splits its branch range over child tasks, which read the node's set from the scratch
arena.  The arena is the caller's and zeroed, so a set that was never written reads as empty.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,p", [(110, 0.85), (150, 0.75), (200, 0.7)])
@pytest.mark.parametrize("k,queues", [(4, 1), (5, 4)])
def test_split_nodes_count_their_whole_set(n, p, k, queues):
    n, e = inputs.random_graph(n, p, seed=11)
    off, adj = oracle.orient(n, e)
    sets = [np.intersect1d(adj[off[u]:off[u + 1]], adj[off[v]:off[v + 1]]).size
            for u in range(n) for v in adj[off[u]:off[u + 1]]]
    assert max(sets) > 64   # the multi-word path runs
    pool, scratch = 64 << 20, 256 << 20
    cfg = runner.make_config(scratch_bytes=scratch)
    need = G.gtap_arena_bytes(G.GTAP_MODE_THREAD, queues, pool, cfg)
    arena = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    base = (arena.data_ptr() + 255) // 256 * 256
    r = runner.kclique(runner.DeviceGraph(n, e), k, n_queues=queues, route=1 if queues > 1 else 0,
                       scratch_bytes=scratch, algorithm=G.GTAP_KCLIQUE_PIVOT, pool_bytes=pool, device_arena=base,
                       arena_bytes=need)
    assert r.values == [oracle.kclique(n, e, k)]
