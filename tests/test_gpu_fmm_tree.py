"""Octree build where its kernels change shape, bit for bit against the oracle's tree (GPU).

Around the radix tiles (1024 keys, 4096 from 2^18 points up), many points of one code (equal keys
keep input order), and leaf sizes that give one cell, a deep chain, or more cells than the first
capacity guess.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(pos, q, leaf):
    with runner.Fmm(order=1, leaf_size=leaf, theta=0.5, mixed=True) as f:
        f.build(pos, q)
        info, geom, order = f.tree()
    cells, ref_order = oracle.fmm_tree(pos, leaf_size=leaf)
    assert np.array_equal(order, ref_order.astype(np.int32))
    assert np.array_equal(info[:, :3], cells[:, 1:4].astype(np.int32))
    assert np.array_equal(info[:, 3], (cells[:, 0].astype(np.int32) << 8) | cells[:, 4].astype(np.int32))
    assert np.array_equal(geom[:, :3], cells[:, 5:8])


@pytest.mark.parametrize("n", [1023, 1024, 1025, 5000, (1 << 18) - 1, 1 << 18, (1 << 18) + 4097])
def test_tree_around_radix_tiles(n):
    pos, q = inputs.fmm_points(n, "plummer", seed=n)
    _check(pos, q, 64)


def test_tree_equal_codes_keep_input_order():
    # 40 points at each of 300 places, interleaved: equal codes everywhere, each place one leaf
    pos, _ = inputs.fmm_points(300, "uniform", seed=2)
    pos = np.tile(pos, (40, 1))
    _check(pos, np.ones(len(pos)), 40)


@pytest.mark.parametrize("n,leaf", [(50, 64), (2, 1), (3000, 1)])
def test_tree_shapes(n, leaf):
    pos, q = inputs.fmm_points(n, "uniform", seed=7)
    if n == 2:
        pos = np.array([[0.0, 0.0, 0.0], [1.0, 1.0, 1.0]]) * 2.0 ** -20 + [[0.5, 0.5, 0.5], [0.5, 0.5, 0.5]]
        pos = np.concatenate([pos, [[0.0, 0.0, 0.0], [1.0, 1.0, 1.0]]])   # a close pair: a chain of one-child cells
        q = np.ones(4)
    _check(pos, q, leaf)
