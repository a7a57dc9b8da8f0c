"""Performance cases: the jobs that users of this library run, through its public entry points.

A pass is one job as a program runs it on a state (or batch) that it keeps: the random-phase state is
initialised, evolved by a number of Trotter steps, and its P(t) and norm series are read back.  The sizes
come from the named workloads of ``paper_0710_3747_gb300.workloads`` (the 2x7, 2x15 ladders, the 20-spin
dipolar star, the disorder batch of 12..22 spins, the served mix of 10..28 spins, T = 5..50 at dt = 0.05),
with the long ones cut to fewer steps, which run the same kernels.

A complex64 state's amplitudes and gates are single precision, so its results are kept as float32 here, as a
program that stores many runs keeps them; a complex128 state's stay float64.
"""
import math

import numpy as np
import torch

from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W

_DEFAULTS = {"prec": "c64", "init": "entangled", "sites": False, "jobs": 0, "m_hi": 0, "resume": False}


def listed():
    return [
        # the smallest served request: a ladder that fits one tile, so latency on one SM is all there is
        {"name": "ladder10", "kind": "ladder", "M": 10, "dt": 0.05, "steps": 100},
        # the 14-spin ladder of the method's own demonstration, whole job
        {"name": "ladder14", "kind": "ladder", "M": 14, "dt": 0.05, "steps": 400},
        # the same in double precision: the job whose P(t) is wanted to 1e-10
        {"name": "ladder14_c128", "kind": "ladder", "M": 14, "dt": 0.05, "steps": 400, "prec": "c128"},
        # a served star of an odd size: all-to-all Gaussian couplings, isotropic (gates and diagonal phase), product state
        {"name": "gauss17", "kind": "gauss", "M": 17, "dt": 0.02, "steps": 100, "init": "product"},
        # the 20-spin dipolar star (L2-sized, gate arithmetic), a tenth of its 1000 steps
        {"name": "star20", "kind": "star", "M": 20, "dt": 0.02, "steps": 100},
        # the same in double precision (the FP64 units are the limit)
        {"name": "star20_c128", "kind": "star", "M": 20, "dt": 0.02, "steps": 10, "prec": "c128"},
        # a stored state is loaded, evolved under XY + Ising couplings, and every amplitude and sector weight read back
        {"name": "resume18", "kind": "xyz", "M": 18, "dt": 0.05, "steps": 40, "resume": True},
        # an odd-sized chain with the polarization of every spin after every step (spreading along the chain)
        {"name": "chain23_sites", "kind": "chain", "M": 23, "dt": 0.05, "steps": 40, "sites": True},
        # a large served star: many gates on every tile, with the diagonal phase
        {"name": "star25", "kind": "star", "M": 25, "dt": 0.05, "steps": 6},
        # a large served ladder
        {"name": "ladder26", "kind": "ladder", "M": 26, "dt": 0.05, "steps": 20},
        # the headline: 2x15 ladder, 2^30 amplitudes streaming from HBM
        {"name": "ladder30", "kind": "ladder", "M": 30, "dt": 0.05, "steps": 6},
        # disorder average: 96 dipolar stars of 12..19 spins evolved together, every job's P(t) and the ensemble
        {"name": "batch96", "kind": "star", "M": 12, "m_hi": 19, "jobs": 96, "dt": 0.02, "steps": 25},
    ]


def draw(rng):
    """Another case of the same ranges: sizes over 10..27 spins, every family, precision, initial state and readout."""
    what = rng.choice(["state", "state", "state", "state", "c128", "sites", "resume", "batch"])
    if what == "batch":
        lo = rng.randint(11, 16)
        return {"kind": rng.choice(["star", "gauss", "ladder"]), "M": lo, "m_hi": lo + rng.randint(0, 3),
                "jobs": rng.randint(8, 120), "dt": 0.02, "steps": rng.randint(10, 40)}
    kind = rng.choice(["ladder", "ladder", "star", "star", "gauss", "chain", "xyz"])
    if what == "c128":
        M = rng.randint(10, 20)
    elif what == "resume":
        M = rng.randint(10, 18)
    else:
        M = rng.randint(10, 27 if kind in ("ladder", "chain") else 24)
    # steps: a served job's 100..1000, fewer for large states (about 2^33 amplitude-bond updates at most)
    gates = 2 * _nbonds(kind, _fit(kind, M)) * 2.0 ** M
    most = max(2, min(600, int(2.0 ** (30 if what == "c128" else 33) / gates)))
    steps = max(2, int(round(math.exp(rng.uniform(math.log(max(2, most // 6)), math.log(most))))))
    if what == "sites" or kind == "xyz":
        steps = min(steps, 60)
    return {"kind": kind, "M": _fit(kind, M), "dt": rng.choice([0.02, 0.05]), "steps": steps,
            "prec": "c128" if what == "c128" else "c64", "init": rng.choice(["entangled", "entangled", "product"]),
            "sites": what == "sites", "resume": what == "resume"}


def _fit(kind, M):
    return M - M % 2 if kind in ("ladder", "xyz") else M


def _nbonds(kind, M):
    return {"ladder": 3 * (M // 2) - 2, "xyz": 3 * (M // 2) - 2, "chain": M - 1}.get(kind, M * (M - 1) // 2)


def _full(case):
    return {**_DEFAULTS, **case}


def _couplings(kind, M, rng):
    """(J, Hamiltonian family, S^zS^z couplings of a generic one) of one job."""
    if kind == "ladder":
        return W.ladder(M // 2, 1.0, float(rng.uniform(0.2, 1.0))), W.XY, None
    if kind == "chain":
        return W.chain(M, float(rng.uniform(0.6, 1.2))), W.XY, None
    if kind == "xyz":
        return (W.ladder(M // 2, 1.0, float(rng.uniform(0.2, 1.0))), W.GENERIC,
                W.ladder(M // 2, float(rng.uniform(0.2, 1.0)), 0.4))
    seed = int(rng.integers(1, 2**31))
    if kind == "gauss":
        return W.star_gaussian(M, seed), W.ISOTROPIC, None
    return W.star_dipolar(M, seed), W.DIPOLAR, None


def _jobs(case, seed):
    """[(J, family, a, phase seed)] of a case's jobs, from the seed alone."""
    rng = np.random.default_rng([0xCA5E, seed])
    if not case["jobs"]:
        sizes = [case["M"]]
    else:
        sizes = [case["M"] + k % (case["m_hi"] - case["M"] + 1) for k in range(case["jobs"])]
    return [(*_couplings(case["kind"], _fit(case["kind"], M), rng), int(rng.integers(1, 2**62))) for M in sizes]


def _loaded(case, seed):
    """A stored state: normalised complex amplitudes with spin 1 mostly up."""
    n = 1 << case["M"]
    rng = np.random.default_rng([0x10AD, seed])
    psi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    psi[0::2] *= 0.3
    return psi / np.linalg.norm(psi)


def prepare(case, seed):
    c = _full(case)
    jobs = _jobs(c, seed)
    systems = [spinrp.System(J, ht, a) for J, ht, a, _ in jobs]
    s = {"case": c, "seed": jobs[0][3]}
    if c["jobs"]:
        s["batch"] = spinrp.Batch(systems, [j[3] for j in jobs], c["prec"], series_cap=c["steps"] + 1)
        return s
    s["state"] = spinrp.State(systems[0], c["prec"], series_cap=c["steps"] + 1)
    s["state"].set_sites(c["sites"])
    if c["resume"]:
        s["psi"] = _loaded(c, seed)
    return s


def _keep(c, x):
    if c["prec"] == "c128":
        return x
    return x.astype(np.complex64 if np.iscomplexobj(x) else np.float32)


def run(s):
    c = s["case"]
    if c["jobs"]:
        b = s["batch"]
        b.init_random_phase().evolve(c["dt"], c["steps"])
        mean, spread = b.ensemble()
        every = np.stack([b.polarization(k) for k in range(b.n)])
        return {"mean": _keep(c, mean), "spread": _keep(c, spread), "P": _keep(c, every)}
    st = s["state"]
    if c["resume"]:
        st.load(s["psi"])
    elif c["init"] == "product":
        st.init_product_phase(s["seed"])
    else:
        st.init_random_phase(s["seed"])
    st.evolve(c["dt"], c["steps"])
    out = {"P": _keep(c, st.polarization(1)), "norm": _keep(c, st.norm_series())}
    if c["sites"]:
        out["sites"] = _keep(c, st.site_series())
    if c["resume"]:
        out["psi"] = _keep(c, st.amplitudes())
        out["sectors"] = _keep(c, st.sector_norms())
    return out


def work(case):
    """Bytes: the state once out (and in, when it is loaded), the series, and for a state that no on-chip memory
    holds two sweeps per Trotter step, forward and reverse half step, each reading and writing it.  Operations:
    three fused multiply-adds a plane for every amplitude pair of every gate, a complex product for the diagonal
    phase."""
    c = _full(case)
    amp = 8 if c["prec"] == "c64" else 16
    total = {"bytes": 0.0, "flops": 0.0}
    sizes = [c["M"]] if not c["jobs"] else [c["M"] + k % (c["m_hi"] - c["M"] + 1) for k in range(c["jobs"])]
    sizes = [_fit(c["kind"], M) for M in sizes]
    state = sum(amp * 2.0 ** M for M in sizes)
    for M in sizes:
        n = 2.0 ** M
        total["bytes"] += amp * n + 16.0 * (c["steps"] + 1) * (1 + M / 2 * c["sites"])
        if c["resume"]:
            total["bytes"] += 2 * 16 * n
        total["flops"] += c["steps"] * n * (6.0 * _nbonds(c["kind"], M) + (0 if c["kind"] in ("ladder", "chain") else 6.0))
    if state > 129e6:
        total["bytes"] += c["steps"] * 4.0 * state
    return total


# ---------------------------------------------------------------------------
# The same jobs in 64 bits, in plain torch: random phases, the symmetric
# second-order Trotter product bond by bond, and the readouts.
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Words 0 and 1 of Philox4x32-10 for int64 counters, key = (low, high word of seed)."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1


def _turns(w0, w1):
    return ((w0 << 21) | (w1 >> 11)).double() * 2.0 ** -53


def _initial(M, init, seed):
    dev = "cuda"
    psi = torch.zeros(1 << M, dtype=torch.complex128, device=dev)
    up = psi.view(-1, 2)[:, 1]
    if init == "product":
        q = torch.arange(M, dtype=torch.int64, device=dev)
        zero = torch.zeros_like(q)
        phi = 2 * math.pi * _turns(*_philox(q, zero, zero, zero + 1, seed))
        x = torch.arange(1 << (M - 1), dtype=torch.int64, device=dev)
        total = torch.zeros(1 << (M - 1), dtype=torch.float64, device=dev)
        for spin in range(1, M):
            total -= phi[spin] * ((x >> (spin - 1)) & 1)
        up.copy_(torch.polar(torch.full_like(total, 2.0 ** (-0.5 * (M - 1))), total))
        return psi
    step = 1 << 25
    for r0 in range(0, 1 << (M - 1), step):
        r = torch.arange(r0, min(r0 + step, 1 << (M - 1)), dtype=torch.int64, device=dev)
        zero = torch.zeros_like(r)
        ang = 2 * math.pi * _turns(*_philox(r, zero, zero, zero, seed))
        up[r0:r0 + r.numel()] = torch.polar(torch.full_like(ang, 2.0 ** (-0.5 * (M - 1))), ang)
    return psi


def _matrices(J, ht, a):
    zero = np.zeros_like(J)
    return {W.XY: (zero, J), W.DIPOLAR: (2 * J, -J), W.ISOTROPIC: (J, J), W.ISING: (J, zero)}.get(ht, (a, J))


def _weights(p, M, every):
    """(weight with spin q up for q = 1 or all, whole weight) of each job."""
    v = torch.view_as_real(p).view(p.shape[0], -1, 2, 1 << 0, 2)
    total = [v[:, :, b].square().sum((1, 2, 3)) for b in (0, 1)] if M < 28 else [
        torch.linalg.vector_norm(v[:, :, b], dim=(1, 2, 3)).square() for b in (0, 1)]
    norm = total[0] + total[1]
    ups = [total[1]]
    if every:
        prob = p.real.square() + p.imag.square()
        ups += [prob.view(p.shape[0], -1, 2, 1 << q)[:, :, 1].sum((1, 2)) for q in range(1, M)]
    return torch.stack(ups, 1), norm


def _evolve(psi, mats, dt, steps, every):
    """Evolves psi (jobs x 2^M, changed in place) and returns the weights after every step and at the start."""
    n, M = psi.shape[0], mats[0][0].shape[0]
    tau = 0.5 * dt
    dev = psi.device
    bonds = [(i, j) for i in range(M) for j in range(i + 1, M) if any(b[i, j] for _, b in mats)]
    gates = []
    for i, j in bonds:
        th = torch.tensor([0.5 * tau * b[i, j] for _, b in mats], dtype=torch.float64, device=dev).view(n, 1, 1, 1)
        gates.append((i, j, torch.cos(th), torch.complex(torch.zeros_like(th), -torch.sin(th))))
    phase = None
    if any(np.any(a) for a, _ in mats):
        theta = torch.zeros(n, 1 << M, dtype=torch.float64, device=dev)
        x = torch.arange(1 << M, device=dev)
        for i in range(M):
            for j in range(i + 1, M):
                aij = [a[i, j] for a, _ in mats]
                if any(aij):
                    sign = 1.0 - 2.0 * (((x >> i) ^ (x >> j)) & 1)
                    theta += 0.25 * torch.tensor(aij, dtype=torch.float64, device=dev).view(n, 1) * sign
        phase = torch.polar(torch.ones_like(theta), -tau * theta)
        del theta, x

    def apply(g):
        i, j, c, s = g
        v = psi.view(n, -1, 2, 1 << (j - i - 1), 2, 1 << i)
        a, b = v[:, :, 0, :, 1], v[:, :, 1, :, 0]
        if n == 1:
            c, s = float(c), complex(s.flatten()[0])
            t = a.clone()
            a.mul_(c).add_(b, alpha=s)
            b.mul_(c).add_(t, alpha=s)
        else:
            t = a * c + b * s
            b.mul_(c).add_(a * s)
            a.copy_(t)

    got = [_weights(psi, M, every)]
    for _ in range(steps):
        if phase is not None:
            psi *= phase
        for g in gates:
            apply(g)
        for g in reversed(gates):
            apply(g)
        if phase is not None:
            psi *= phase
        got.append(_weights(psi, M, every))
    ups, norms = torch.stack([u for u, _ in got]), torch.stack([w for _, w in got])
    return ups.cpu().numpy(), norms.cpu().numpy()


def exact(case, seed):
    c = _full(case)
    jobs = _jobs(c, seed)
    if c["jobs"]:
        P = np.empty((len(jobs), c["steps"] + 1))
        for M in sorted({j[0].shape[0] for j in jobs}):
            at = [k for k, j in enumerate(jobs) if j[0].shape[0] == M]
            psi = torch.stack([_initial(M, c["init"], jobs[k][3]) for k in at])
            u, w = _evolve(psi, [_matrices(*jobs[k][:3]) for k in at], c["dt"], c["steps"], False)
            P[at] = (2 * u[:, :, 0] / w - 1).T
        return {"mean": P.mean(0), "spread": P.std(0), "P": P}
    J, ht, a, phase_seed = jobs[0]
    M = J.shape[0]
    psi = torch.from_numpy(_loaded(c, seed)).cuda() if c["resume"] else _initial(M, c["init"], phase_seed)
    psi = psi.view(1, -1)
    u, w = _evolve(psi, [_matrices(J, ht, a)], c["dt"], c["steps"], c["sites"])
    out = {"P": 2 * u[:, 0, 0] / w[:, 0] - 1, "norm": w[:, 0]}
    if c["sites"]:
        out["sites"] = 2 * u[:, 0] / w - 1
    if c["resume"]:
        out["psi"] = psi[0].cpu().numpy()
        ones = np.array([bin(k).count("1") for k in range(1 << M)])
        out["sectors"] = np.bincount(ones, np.abs(out["psi"]) ** 2, M + 1)
    return out
