"""k-clique tasks that no warp request serves run in full batches (GPU).

The triangle count and pivoting use one lane a task: a step of a warp takes up to 32 of them.  Range
tasks fork by eight down to single edges' ranges, so all but the first few steps find full queues.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("algorithm", [G.GTAP_KCLIQUE_ORIENT, G.GTAP_KCLIQUE_PIVOT])
@pytest.mark.parametrize("queues", [1, 4])
def test_triangle_tasks_fill_the_warp(algorithm, queues):
    n, e = inputs.rmat_graph(13, 16, seed=5)
    r = runner.kclique(runner.DeviceGraph(n, e), 3, n_queues=queues, route=1 if queues > 1 else 0, algorithm=algorithm)
    assert r.values == [oracle.kclique(n, e, 3)]
    assert r.stats["tasks_executed"] > 16 * r.stats["steps"]


def test_branches_of_sets_beyond_the_warp_buffer_fill_the_warp():
    # DAG edges of K_700 that leave vertex 0 towards the next 100: sets of 599 to 698 members, past
    # the 512 a warp holds
    n = 700
    u, v = np.triu_indices(n, k=1)
    g = runner.DeviceGraph(n, np.stack([u, v], axis=1).astype(np.int32))
    r = runner.kclique(g, 4, n_queues=4, route=1, ranges=[(0, 100)], grid_blocks=8)
    assert r.values == [sum((n - 1 - w) * (n - 2 - w) // 2 for w in range(1, 101))]
    assert r.stats["tasks_executed"] > 8 * r.stats["steps"]


def test_triangle_tasks_beside_tasks_for_the_warp_are_held_few_at_a_time():
    # a full batch claimed for triangles could hold 4-clique tasks, which the warp serves one by one
    n, e = inputs.rmat_graph(12, 16, seed=5)
    g = runner.DeviceGraph(n, e)
    with runner.Context(G.GTAP_MODE_THREAD, 4, scratch_bytes=1 << 30) as c:
        t = c.register("kclique")
        handles = [c.spawn(t, g.args(k, 64, 1)) for k in (3, 4)]
        c.run()
        assert [c.result_u64(h) for h in handles] == [oracle.kclique(n, e, k) for k in (3, 4)]
        assert c.stats()["tasks_executed"] <= 2 * c.stats()["steps"]
