"""GPU: register programs at their edges against the oracle -- walks over the
register-bit pairs, the tabulated diagonal op, and passes whose first and last
phase move the tile between registers and the state.

Random coupling graphs (sparse ones give passes of one phase, relabelled or
not, and phases of one gate; dense ones full walks), tiles of 2^10..2^14
amplitudes, five and six register bits, so 5..9 thread-index bits and zero to
six outer spins.  Tolerances: |dP| <= 1e-5 at every step and amplitudes within
1.3e-4 of the typical amplitude 2^{-(M-1)/2}, the bars of the other complex64
tests (rounding 6e-8 per gate, at most about 10^3 gates on an amplitude).
"""
import numpy as np
import pytest

import oracle
from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _graph(seed):
    rng = np.random.default_rng([0x9A7, seed])
    M = int(rng.integers(11, 17))
    J = np.triu(rng.normal(size=(M, M)) * (rng.random((M, M)) < (0.12, 0.3, 1.0)[seed % 3]), 1)
    J[0, 1] = 0.8
    a = np.triu(rng.normal(size=(M, M)) * (rng.random((M, M)) < 0.5), 1)
    return M, J + J.T, a + a.T, (W.XY, W.GENERIC, W.DIPOLAR, W.ISOTROPIC)[seed % 4]


@pytest.mark.parametrize("rb", [5, 6])
@pytest.mark.parametrize("seed", range(12))
def test_random_graphs_match_oracle(seed, rb):
    M, J, a, ht = _graph(seed)
    dt, steps, phase = 0.03, 4, 91 + seed
    a = a if ht == W.GENERIC else None
    Pw, Nw, psi = oracle.run(J, ht, phase, dt, steps, a_generic=a)
    for K in sorted({max(5 + rb, 10 + seed % 3), min(14, M)}):
        s = spinrp.System(J, ht, a)
        s.set_tile("c64", min(K, M))
        s.set_regbits(rb)
        s.plan_check("c64")
        st = spinrp.State(s, "c64", series_cap=steps + 1).init_random_phase(phase)
        st.evolve(dt, 1).evolve(dt, steps - 1)
        assert np.max(np.abs(st.polarization() - Pw)) <= 1e-5
        assert np.max(np.abs(st.norm_series() - Nw)) <= 1e-5
        assert np.max(np.abs(st.amplitudes() - psi)) <= 1.3e-4 * 2.0 ** (-(M - 1) / 2)
        st.close()
