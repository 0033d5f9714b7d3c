"""An idle warp whose fullest queue was stolen (GPU).

Worker 0 of an 8-warp block starts with all the work: 256 leaves in its first class and 31 leaves of
ten times their length in its second.  It pops 32 of the short ones; the seven other warps steal 32
each, from the fuller class every time, which empties the first.  So worker 0's next look at that
class fails although the second holds tasks.  It must not run them with the block's probe token: the
warps that are idle meanwhile probe, steal and watch the deadline only with that token.
"""
import pytest

from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import runner

pytestmark = pytest.mark.gpu

WARPS = 8
ITERS = 400000


def _leaf(iters):
    return G.gtap_bintree_args(0, iters, 1, 0, 0, 0)


def _context(policy, roots):
    c = runner.Context(G.GTAP_MODE_THREAD, 2, grid_blocks=1, steal_policy=policy)
    t = c.register("bintree")
    for iters, q in roots:
        c.spawn(t, _leaf(iters), queue=q)   # roots 0, 8, 16, ... are worker 0's
        for _ in range(WARPS - 1):
            c.spawn(t, _leaf(0))
    return c


@pytest.mark.parametrize("policy", [G.GTAP_STEAL_FILL, G.GTAP_STEAL_EMPTY])
def test_idle_warps_watch_the_deadline(policy):
    with _context(policy, [(ITERS, 0)] * 32) as c:
        c.run()
        assert c.stats()["n_workers"] == WARPS
        one = c.stats()["kernel_ms"]   # one step of the short leaves
    with _context(policy, [(ITERS, 0)] * 256 + [(10 * ITERS, 1)] * 31) as c:
        # the short leaves end after one step's time, the long ones after eleven
        G.gtap_set_timeout(c.ctx, int(3e6 * one))
        assert c.run(raise_on_error=False) == G.GTAP_ERR_TIMEOUT
        assert c.stats()["kernel_ms"] > 5 * one   # a step in flight is not interrupted
