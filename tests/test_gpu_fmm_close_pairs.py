"""Mixed FMM with two points closer than FP32 resolves on either side of a leaf face (GPU).

The points are distinct, so their potentials are large but finite, as the FP64 oracle has them.
"""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n,gap", [(600, 1e-10), (600, 1e-13), (5000, 1e-12)])
def test_pair_across_the_mid_plane(n, axis, gap):
    pos, q = inputs.fmm_points(n, "uniform", seed=n)
    pos[0], pos[1] = 0.0, 1.0              # the cube is [0, 1]^3, its mid-planes are leaf faces
    pos[2] = pos[3] = [0.3, 0.3, 0.3]
    pos[2, axis], pos[3, axis] = 0.5 - gap / 2, 0.5 + gap / 2
    q[2], q[3] = 0.75, -0.5
    ref = oracle.fmm(pos, q, p=6, theta=0.5, leaf_size=64)
    with runner.Fmm(order=6, leaf_size=64, theta=0.5, mixed=True) as f:
        phi = f.run(pos, q).cpu().numpy()
    assert np.isfinite(phi).all()
    # the tolerance of the mixed form against the oracle in the other tests, for the pair and for the rest
    assert np.abs(phi[2:4] / ref[2:4] - 1).max() <= 1e-5
    rest = np.delete(np.arange(n), [2, 3])
    assert np.linalg.norm(phi[rest] - ref[rest]) <= 1e-5 * np.linalg.norm(ref[rest])
