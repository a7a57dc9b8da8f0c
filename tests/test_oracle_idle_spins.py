"""Oracle: couplings of fewer spins than the state has leave the others idle."""
import numpy as np
import pytest

import oracle
from paper_0710_3747_gb300 import workloads as W


@pytest.mark.parametrize("htype", [oracle.XY, oracle.DIPOLAR])
@pytest.mark.parametrize("idle", [1, 2])
def test_smaller_couplings_are_padded(htype, idle):
    a, b = oracle.couplings(W.ladder(4, 1.0, 0.5), htype)
    M = 8 + idle
    wide = [np.pad(x, (0, idle)) for x in (a, b)]
    psi0 = oracle.init_random_phase(M, 8)
    got, want = psi0.copy(), psi0.copy()
    P, N = oracle.evolve(got, a, b, 0.07, 3)
    Pw, Nw = oracle.evolve(want, *wide, 0.07, 3)
    assert np.array_equal(got, want) and np.array_equal(P, Pw) and np.array_equal(N, Nw)
    Pa, _ = oracle.evolve_all_sites(psi0.copy(), a, b, 0.07, 3)
    assert np.array_equal(Pa[:, 0], P)
    x = psi0.copy()
    oracle.diag(x, a, 0.3)
    y = psi0.copy()
    oracle.diag(y, wide[0], 0.3)
    assert np.array_equal(x, y)


def test_larger_couplings_are_refused():
    a, b = oracle.couplings(W.ladder(4, 1.0, 0.5), oracle.XY)
    with pytest.raises(ValueError):
        oracle.evolve(oracle.init_random_phase(7, 1), a, b, 0.1, 1)
