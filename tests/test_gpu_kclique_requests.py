"""k-clique counts where the warp-served passes change path (GPU).

Complete graphs have closed-form counts, C(n, k), and candidate sets of every size up to n - 2: around
the row limit of 64, the powers of two of the search, and the 512 members a warp's set buffer holds.
"""
import math

import numpy as np
import pytest

from paper_2604_05982_gb300 import runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _complete(n):
    u, v = np.triu_indices(n, k=1)
    return runner.DeviceGraph(n, np.stack([u, v], axis=1).astype(np.int32))


@pytest.mark.parametrize("n,k", [(3, 3), (4, 4), (35, 4), (66, 4), (67, 4), (131, 4), (258, 4), (259, 4), (514, 4), (515, 4),
                                 (300, 3), (66, 5), (131, 5), (70, 6)])
@pytest.mark.parametrize("thr,queues", [(64, 4), (2, 1)])
def test_complete_graph_counts(n, k, thr, queues):
    if thr == 2 and k > 4:
        thr = 32
    r = runner.kclique(_complete(n), k, split_threshold=thr, n_queues=queues, route=1 if queues > 1 else 0)
    assert r.values == [math.comb(n, k)]


def test_several_small_graphs_in_one_launch():
    # lanes of one warp serve requests of different graphs and clique sizes
    ns = [5, 20, 64, 65, 66, 90, 129]
    gs = [_complete(n) for n in ns]
    for k in (4, 5):
        assert runner.kclique(gs, k, n_queues=4, route=1).values == [math.comb(n, k) for n in ns]
