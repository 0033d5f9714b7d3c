"""FMM near field on exceptional values, and tree sizes and orders at the ends of their ranges (GPU)."""
import numpy as np
import pytest

import oracle
from paper_2604_05982_gb300 import inputs, runner

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# The FP64 reciprocal square root starts from the FP32 approximation for arguments with a biased
# exponent in [897, 1150] and takes the library's elsewhere: both sides of the window's ends, odd and
# even exponents, arguments that are subnormal, zero (the square underflows) and infinite (it overflows).
GAPS = [2.0 ** -63, 2.0 ** -63 * (1 - 2.0 ** -30), 2.0 ** 64, 2.0 ** 64 * (1 - 2.0 ** -30), 1.0, 3.0, 0.1, 1.5e-5, 7.7e11,
        1.4142135623730951, 2.0 ** -520 * 1.25, 2.0 ** -511, 1e-170, 1e150, 2e160]


@pytest.mark.parametrize("gap", GAPS)
def test_two_points_fp64(gap):
    pos = np.array([[0.0, 0.0, 0.0], [gap, 0.0, 0.0]])
    q = np.array([1.0, -2.0])
    with runner.Fmm(order=2, leaf_size=64, theta=0.5, mixed=False) as f:
        phi = f.run(pos, q).cpu().numpy()
    with np.errstate(all="ignore"):
        inv = 1.0 / np.sqrt(np.float64(gap) * np.float64(gap))
    want = np.array([-2.0, 1.0]) * inv
    if np.isfinite(inv) and inv != 0.0:
        # half an ulp of the last step, a quarter from the rounded residual, two roundings of the
        # reference: below two ulps
        assert np.abs(phi / want - 1).max() <= 2.0 ** -51
    else:
        assert np.array_equal(phi, want)


@pytest.mark.parametrize("mixed,tol", [(False, 1e-12), (True, 1e-5)])
@pytest.mark.parametrize("n", [40, 100, 131])
def test_an_infinite_charge_stays_where_it_belongs(n, mixed, tol):
    # at most two levels: every pair is near, no expansion is used
    pos, q = inputs.fmm_points(n, "uniform", seed=n)
    j = n // 2
    clean = oracle.fmm(pos, np.where(np.arange(n) == j, 0.0, q), p=2, theta=0.5, leaf_size=64)
    q[j] = np.inf
    with runner.Fmm(order=2, leaf_size=64, theta=0.5, mixed=mixed) as f:
        phi = f.run(pos, q).cpu().numpy()
    assert np.isposinf(np.delete(phi, j)).all()
    assert abs(phi[j] - clean[j]) <= tol * abs(clean[j])


def test_more_cells_than_the_first_capacity():
    # pairs 2^-20 apart: leaves of one point at the end of chains of one-child cells, more cells than the
    # build's first guess of 2 * (8 n / (leaf + 1)) + 64, so it starts again with twice the room
    m = 3000
    at, _ = inputs.fmm_points(m, "uniform", seed=4)
    at = (np.floor(at * 2.0 ** 18) + 0.25) / 2.0 ** 18
    pos = np.concatenate([at, at + 0.9 * 2.0 ** -20, [[0.0, 0.0, 0.0], [1.0, 1.0, 1.0]]])
    cells, ref_order = oracle.fmm_tree(pos, leaf_size=1)
    assert len(cells) > 2 * (8 * len(pos) // 2) + 64
    with runner.Fmm(order=1, leaf_size=1, theta=0.5, mixed=False) as f:
        for _ in range(2):   # (the second build starts with the grown capacity)
            f.build(pos, np.ones(len(pos)))
            info, geom, order = f.tree()
            assert np.array_equal(order, ref_order.astype(np.int32))
            assert np.array_equal(info[:, :3], cells[:, 1:4].astype(np.int32))
            assert np.array_equal(info[:, 3], (cells[:, 0].astype(np.int32) << 8) | cells[:, 4].astype(np.int32))
            assert np.array_equal(geom[:, :3], cells[:, 5:8])


@pytest.mark.parametrize("mixed,tol", [(False, 1e-12), (True, 1e-5)])
@pytest.mark.parametrize("order", [1, 3, 7, 8])
def test_orders_against_the_oracle(order, mixed, tol):
    pos, q = inputs.fmm_points(6001, "plummer", seed=order)
    ref = oracle.fmm(pos, q, p=order, theta=0.5, leaf_size=32)
    with runner.Fmm(order=order, leaf_size=32, theta=0.5, mixed=mixed) as f:
        phi = f.run(pos, q).cpu().numpy()
    assert np.linalg.norm(phi - ref) <= tol * np.linalg.norm(ref)
