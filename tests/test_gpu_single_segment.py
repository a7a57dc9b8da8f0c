"""GPU: plans of one sweep per step with spins outside the tile (Ising systems,
and flip-flop bonds that fit one tile under S^zS^z couplings of every spin)
against the oracle.  The first sweep of a call applies the diagonal op twice,
for dt/2 and for dt, so the outer spins' share is needed for both.

Tolerances are the bars of the other tests: complex64 |dP| <= 1e-5 and
amplitudes within 1.3e-4 of the typical amplitude 2^{-(M-1)/2} (rounding 6e-8 an
op, far fewer than 10^3 of them here), complex128 1e-10 and 1e-10.
"""
import numpy as np
import pytest

import oracle
from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DT, PHASE, THREADS = 0.05, 31, 16


def _dense(M, rng):
    a = np.triu(rng.normal(size=(M, M)), 1)
    return a + a.T


def _system(kind, M, seed=0):
    """(J, family, S^zS^z couplings): no bonds, or bonds among spin 1 and a few others."""
    rng = np.random.default_rng([0x51, M, seed])
    if kind == "ising":
        return _dense(M, rng), W.ISING, None
    on = [0] + sorted(rng.choice(np.arange(1, M), size=5, replace=False).tolist())
    J = np.zeros((M, M))
    for x, y in zip(on, on[1:]) if kind == "path" else [(p, q) for p in on for q in on if p < q]:
        J[x, y] = J[y, x] = rng.normal() + 1.5
    return J, W.GENERIC, _dense(M, rng)


def _bars(prec, M):
    typical = 2.0 ** (-(M - 1) / 2)
    return (1e-10, 1e-10 * typical) if prec == "c128" else (1e-5, 1.3e-4 * typical)


@pytest.mark.parametrize("kind,M,prec,K,rb,orient,sites", [
    ("ising", 14, "c64", 0, 0, 0, False),
    ("ising", 15, "c64", 13, 6, 0, False),
    ("ising", 16, "c64", 14, 6, 0, True),
    ("ising", 17, "c64", 0, 0, 0, False),
    ("ising", 17, "c128", 0, 0, 0, False),
    ("ising", 13, "c64", 8, 0, 0, False),   # per-gate kernel
    ("dense", 14, "c64", 10, 5, 0, False),
    ("dense", 14, "c64", 0, 0, 0, True),
    ("dense", 17, "c64", 13, 6, 0, True),
    ("dense", 18, "c128", 0, 0, 0, False),
    ("path", 15, "c64", 12, 5, 1, False),   # oriented storage
    ("path", 16, "c64", 13, 6, 1, False),
    ("dense", 23, "c64", 13, 6, 0, False),  # pipelined sweep
    ("dense", 23, "c64", 13, 6, 0, True),
])
def test_states_match_oracle(kind, M, prec, K, rb, orient, sites):
    J, ht, a = _system(kind, M)
    s = spinrp.System(J, ht, a)
    s.set_tile(prec, K)
    s.set_regbits(rb)
    s.set_orientation(orient)
    info = s.plan_info(prec)
    assert info["segments"] == 1 and info["K"] < M
    assert bool(s.orientation(prec)) == bool(orient)
    s.plan_check(prec)
    Pw, Nw, psi = oracle.run(J, ht, PHASE, DT, 6, a_generic=a, threads=THREADS)
    st = spinrp.State(s, prec, series_cap=8).set_sites(sites)
    assert st.pipeline() == (M == 23)
    st.init_random_phase(PHASE).evolve(DT, 1).evolve(DT, 2).evolve(DT, 3)
    barP, bar = _bars(prec, M)
    assert np.max(np.abs(st.polarization() - Pw)) <= barP
    assert np.max(np.abs(st.norm_series() - Nw)) <= barP
    assert np.max(np.abs(st.amplitudes() - psi)) <= bar
    st.close()


@pytest.mark.parametrize("M,K,rb,jobs,persistent,pipelined", [
    (14, 0, 0, 5, False, 0),
    (15, 13, 6, 8, True, 0),
    (17, 13, 6, 40, False, 1),
])
def test_batches_match_oracle(M, K, rb, jobs, persistent, pipelined):
    rng = np.random.default_rng([0x52, M])
    J, ht, _ = _system("dense", M)
    systems, avals = [], []
    for _ in range(jobs):
        avals.append(_dense(M, rng))
        systems.append(spinrp.System(J, ht, avals[-1]))
        systems[-1].set_tile("c64", K)
        systems[-1].set_regbits(rb)
    b = spinrp.Batch(systems, [PHASE + k for k in range(jobs)], "c64", series_cap=8).set_persistent(persistent)
    assert b.pipeline_groups() == pipelined
    b.init_random_phase().evolve(DT, 1).evolve(DT, 5)
    for k in (0, jobs // 2, jobs - 1):
        Pw, _, _ = oracle.run(J, ht, PHASE + k, DT, 6, a_generic=avals[k], threads=THREADS)
        assert np.max(np.abs(b.polarization(k) - Pw)) <= 1e-5
    b.close()
