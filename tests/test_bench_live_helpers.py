"""bench.py's helpers that feed the reported FMM roofline and launch counts (no GPU)."""
import importlib.util
import os
from math import comb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_harmonic_m2l_flops_closed_form():
    # Pairs of coefficients: sum of (2 k1 + 1)(2 k2 + 1) over k1 + k2 <= p, the x^p coefficient of
    # (1 + x)^2 / (1 - x)^5; one FMA each.  Recurrence of order k, index (a, b, c) with c in {0, 1}: two
    # flops per first-order and per second-order term and one more where there is a second-order term;
    # the components number 2k (c = 0) and 3k - 2 (c = 1), those above one 2(k-1) and 2(k-2), the
    # coefficients with one k + 1 less (1, 1) at k = 2, and k less (1, 1, 1) at k = 3.  Each order
    # adds 4 factors' flops less the constant ones (2) and 2 per z = 2 entry (k - 1 of them), and the
    # displacement 7 + 2p.
    b = _bench()
    for p in range(1, 7):
        pairs = comb(p + 4, 4) + 2 * comb(p + 3, 4) + comb(p + 2, 4)
        assert pairs == sum((2 * i + 1) * (2 * j + 1) for i in range(p + 1) for j in range(p + 1 - i))
        rec = 7 + 2 * p
        for k in range(1, p + 1):
            second = 2 * (k - 1) + 2 * max(k - 2, 0)
            with_second = {1: 0, 2: 2, 3: 4 + 2}.get(k, 2 * k + 1)
            rec += 2 + 2 * (5 * k - 2) + 2 * second + with_second + 2 * (k - 1)
        assert b.m2l_flops_per_pair_harmonic(p) == rec + 2 * pairs, p
    assert b.m2l_flops_per_pair_harmonic(6) == 1452


def test_fmm_launches_of_the_bench_sets():
    b = _bench()
    # tree: box, codes, 8 radix passes, refinement, gather, check, leaf-local coordinates (mixed);
    # upward: P2M and a launch per level above the leaves'; traversal: constants, reset, run, report;
    # evaluation: two groupings of 5, fold and M2L, L2L per level, runs, P2P, L2P
    assert b._fmm_launches_per_instance(6, True) == 14 + 6 + 4 + (10 + 2 + 5 + 3)
    assert b._fmm_launches_per_instance(10, False) == 13 + 10 + 4 + (10 + 2 + 9 + 3)
    assert b._fmm_launches_per_instance(1, True) == 14 + 1 + 4 + (10 + 2 + 0 + 3)
