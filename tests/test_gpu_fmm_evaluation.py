"""FMM evaluation kernels where their work split changes, against the FP64 oracle FMM (GPU).

Near lists longer than one run (small leaves, skewed sets), leaves of one point, point counts
around the 4-lane groups and the point pairs of the P2P kernels, and every register order of M2L.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mixed,tol", [(False, 1e-12), (True, 1e-5)])
@pytest.mark.parametrize("n,dist,leaf,order", [(3, "uniform", 1, 2), (257, "uniform", 1, 2), (4097, "plummer", 3, 2),
                                               (30001, "plummer", 5, 4), (9001, "plummer", 64, 5),
                                               (12289, "uniform", 33, 6)])
def test_evaluation_splits(n, dist, leaf, order, mixed, tol):
    pos, q = inputs.fmm_points(n, dist, seed=n)
    ref = oracle.fmm(pos, q, p=order, theta=0.5, leaf_size=leaf)
    with runner.Fmm(order=order, leaf_size=leaf, theta=0.5, mixed=mixed) as f:
        phi = f.run(pos, q).cpu().numpy()
    assert np.linalg.norm(phi - ref) <= tol * np.linalg.norm(ref)
