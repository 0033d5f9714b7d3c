"""Octree refinement with any number of blocks, bit for bit against the oracle's tree (GPU).

No block waits for one that has not started: a single block refines everything, and a grid of many
more blocks than the GPU holds at a time (2048 threads an SM) ends.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("blocks", [1, 2, 7, 151, 6000])
@pytest.mark.parametrize("n,leaf", [(1, 64), (65, 64), (5000, 3)])
def test_refinement_by_any_number_of_blocks(blocks, n, leaf):
    pos, q = inputs.fmm_points(n, "plummer", seed=n)
    cells, ref_order = oracle.fmm_tree(pos, leaf_size=leaf)
    with runner.Fmm(order=1, leaf_size=leaf, theta=0.5, mixed=True) as f:
        assert G.load_library().gtap_debug_fmm_refine_blocks(G._P(f.plan), blocks) == 0
        for _ in range(2):
            f.build(pos, q)
            info, geom, order = f.tree()
            assert np.array_equal(order, ref_order.astype(np.int32))
            assert np.array_equal(info[:, :3], cells[:, 1:4].astype(np.int32))
            assert np.array_equal(info[:, 3], (cells[:, 0].astype(np.int32) << 8) | cells[:, 4].astype(np.int32))
            assert np.array_equal(geom[:, :3], cells[:, 5:8])
