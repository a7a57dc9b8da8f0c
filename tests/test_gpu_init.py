"""GPU: the initial states over the sizes where the index map of the kernel
changes (fewer states than threads, no loop bits, one to four loop bits) and
layouts that put spin 1 anywhere, every amplitude against the oracle.

The product state's reference sums its phases exactly, as 64-bit fixed-point
turns (u_l has 53 bits): in FP64 the sum of 23 phases is itself off by more
than a rounding of the amplitude.

Tolerances: an amplitude is 2^{-(M-1)/2} times a cosine and a sine, each within
2e-7 (complex64: angle, function and product roundings of 6e-8) or 1e-15
(complex128) of its value.
"""
import numpy as np
import pytest

import oracle
from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _product(M, seed):
    turns = np.zeros(1, dtype=np.uint64)  # of the up spins' phases, spins 2..M
    for spin in range(1, M):
        t = np.uint64(int(oracle.product_uniform(seed, spin) * 2**53) << 11)
        turns = np.concatenate([turns, turns - t])
    ang = turns.astype(np.int64).astype(np.float64) * (2 * np.pi / 2**64)
    psi = np.zeros(1 << M, dtype=np.complex128)
    psi[1::2] = 2.0 ** (-(M - 1) / 2) * np.exp(1j * ang)
    return psi


@pytest.mark.parametrize("kind", ["entangled", "product"])
@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("M,K", [(2, 0), (8, 0), (9, 7), (10, 8), (18, 10), (19, 9), (20, 10), (22, 12), (23, 11), (24, 12)])
def test_initial_states(M, K, prec, kind):
    J = W.star_gaussian(M, 3) if M < 20 else W.chain(M, 0.7)[::-1, ::-1].copy()
    s = spinrp.System(J, spinrp.XY)
    s.set_tile(prec, K)
    st = spinrp.State(s, prec, series_cap=1)
    init, ref = ((st.init_random_phase, oracle.init_random_phase) if kind == "entangled"
                 else (st.init_product_phase, _product))
    init(2**61 + 17 * M)
    got, want = st.amplitudes(), ref(M, 2**61 + 17 * M)
    tol = (2e-7 if prec == "c64" else 1e-15 * max(1, M)) * 2.0 ** (-(M - 1) / 2)
    assert np.max(np.abs(got - want)) <= tol
    assert st.polarization()[0] == 1.0
    assert abs(st.norm_series()[0] - 1.0) <= (1e-6 if prec == "c64" else 1e-13)
    st.close()
