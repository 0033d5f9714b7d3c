"""gtap_config.idle_backoff_ns governs every idle warp of a block, not the probing one alone (GPU)."""
import pytest

from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import runner

pytestmark = pytest.mark.gpu


def _idle_rounds_per_ms(backoff):
    # one long leaf on a block of eight warps: one idle warp probes, six wait for its turn
    r = runner.bintree(0, 1000000, grid_blocks=1, idle_backoff_ns=backoff)
    assert r.stats["n_workers"] == 8
    return r.stats["idle_iterations"] / r.stats["kernel_ms"]


def test_short_backoff_shortens_every_idle_sleep():
    # The waiting warps sleep up to 512 ns instead of 6400 (about 0.7 against 6.4 us a round, six
    # warps), the probing one 32 instead of 512 (0.6 to 0.8 against 1.1 us a round): 10 rounds a us against 2.
    # With the probing warp alone on the shorter sleep it would be 2.7 against 2.
    assert _idle_rounds_per_ms(32) > 2.5 * _idle_rounds_per_ms(512)
