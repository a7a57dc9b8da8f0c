"""GPU: sweeps that start early beside the running one spread over the SMs.

The tiles of the first job of each pair take one SM each (a half to a fifth of
the GPU); the second job has twice as many (four times for the stars), and still
no SM needs two of one sweep, or only the larger job needs two.  With the early
blocks crowded on a few SMs a sweep lasts twice as long.  Times are the least of
several device-timed runs; the bars lie midway between an even spread (1.1, 1.1,
and at most 0.6) and a crowded one (1.8, 1.5, 0.9)."""
import pytest

from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

pytestmark = pytest.mark.gpu
STEPS = 48


def _time(obj):
    import torch

    best = float("inf")
    for k in range(7):
        obj.init_random_phase(3) if isinstance(obj, spinrp.State) else obj.init_random_phase()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        obj.evolve(0.02, STEPS)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b)) if k > 1 else best
    obj.close()
    return best


def _state(J, ht, prec):
    return spinrp.State(spinrp.System(J, ht), prec, series_cap=STEPS + 1)


def _batch(Js, ht, prec):
    return spinrp.Batch([spinrp.System(J, ht) for J in Js], list(range(len(Js))), prec, series_cap=STEPS + 1)


def test_four_stars_cost_little_more_than_one():
    """complex64 stars of 17 spins: 32 blocks, and 128."""
    one = _time(_state(W.star_dipolar(17, 1), W.DIPOLAR, "c64"))
    four = _time(_batch([W.star_dipolar(17, 1 + k) for k in range(4)], W.DIPOLAR, "c64"))
    assert four <= 1.4 * one, (four, one)


def test_two_chains_cost_little_more_than_one_c128():
    """complex128 chains of 18 spins: 128 blocks of which three fit an SM, and 256."""
    one = _time(_state(W.chain(18, 0.9), W.XY, "c128"))
    two = _time(_batch([W.chain(18, 0.9 + 0.1 * k) for k in range(2)], W.XY, "c128"))
    assert two <= 1.3 * one, (two, one)


def test_half_the_state_takes_half_the_time_c128():
    """complex128 chains of 19 spins (a tile an SM) against 20 (two)."""
    small = _time(_state(W.chain(19, 0.9), W.XY, "c128"))
    large = _time(_state(W.chain(20, 0.9), W.XY, "c128"))
    assert small <= 0.75 * large, (small, large)


def test_all_site_sweep_shares_an_sm_c128():
    """complex128 chain of 20 spins, 256 blocks: the readout sweep (one of a step's two)
    with two blocks an SM takes the step to 1.4 times, one at a time to 1.66."""
    J = W.chain(20, 0.9)
    plain = _time(_state(J, W.XY, "c128"))
    sites = _time(_state(J, W.XY, "c128").set_sites(True))
    assert sites <= 1.53 * plain, (sites, plain)
