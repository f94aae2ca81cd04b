"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one call of a user's program: a batch of systems (lattice, size,
temperatures, couplings, paths), a schedule of sweeps, a precision and the
options in use.  Kinds:

  run       a kept handle (mp.Simulation): one full run and every system's estimates
  call      the whole one-shot call (mp.simulate): create, run, estimates, destroy
  gradient  mp.autograd.observables forward and backward at many (beta, h) pairs

prepare() makes what the program has in hand (the handle of a batch for one
seed), run() is one pass, exact() the same numbers from plain torch in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1305_6758_gb300 as mp
from paper_1305_6758_gb300 import autograd as mp_autograd

# Estimates that are results: without the echoes of the inputs, the run's own
# clock and the largest rounding residue of |S| (a column of the records too).
RESULTS = [f for f in mp.EST_FIELDS
           if f not in ("n_paths", "N", "T", "n_meas", "attempts", "norm_max", "elapsed_s")]
LATTICES = {"sc": mp.SC, "chain": mp.CHAIN, "ising": mp.ISING}
# Operations (integer and floating, all lanes) that one attempted update needs:
# Philox4x32-10 and the uniforms 46, the trial direction 9, the spin 6, three
# loads and three adds (less one add) per neighbour, the energy change 8, the
# accept test 5, the measurement 2; an Ising flip shares a Philox call of four.
OPS = {"sc": 109.0, "chain": 85.0, "ising": 25.0}


def listed():
    return [
        # the plain method as first stated: one small lattice in FP64, long schedule
        dict(name="plain_fp64", kind="run", lattice="sc", L="4", paths="256", T0=1.5, T1=1.5, nT=1,
             J=1.0, h=0.0, n_therm=1000, n_meas=1000, fp64=True, flags=0),
        # the headline scan: L = 16 over 21 temperatures, the GPU full for the whole call (a
        # shorter schedule than a production scan's: time is proportional to the sweeps)
        dict(name="scan_L16", kind="run", lattice="sc", L="16", paths="4096", T0=0.5, T1=2.5, nT=21,
             J=1.0, h=0.0, n_therm=50, n_meas=50, fp64=False, flags=0),
        # finite-size scaling at T_C: uneven sizes in one launch, one of them on two-CTA clusters
        dict(name="batch_uneven", kind="run", lattice="sc", L="8,12,16,20,24,32",
             paths="8192,4096,2048,1024,512,256", T0=1.44, T1=1.44, nT=1, J=1.0, h=0.0, n_therm=60,
             n_meas=60, fp64=False, flags=0),
        # large lattices near T_C, streamed from HBM
        dict(name="large_L64", kind="run", lattice="sc", L="64", paths="1024", T0=1.40, T1=1.48, nT=3,
             J=1.0, h=0.0, n_therm=10, n_meas=20, fp64=False, flags=0),
        # the paper's search for T_C (its Sec. 5): Binder cumulants of L = 20 and 30 after 200
        # sweeps, one output per path
        dict(name="binder_L20_L30", kind="run", lattice="sc", L="20,30", paths="800,800", T0=1.44,
             T1=1.45, nT=2, J=1.0, h=0.0, n_therm=199, n_meas=1, fp64=False, flags=0),
        # the FP64 form that FP32 results are held against
        dict(name="fp64_L16", kind="run", lattice="sc", L="16", paths="1024", T0=0.5, T1=2.5, nT=3,
             J=1.0, h=0.0, n_therm=20, n_meas=20, fp64=True, flags=0),
        # an ordinary small study (the paper's Sec. 4): L = 10, 1000 paths, half of them from the
        # ordered state
        dict(name="two_start_L10", kind="run", lattice="sc", L="10", paths="1000", T0=1.0, T1=1.0, nT=1,
             J=1.0, h=0.0, n_therm=500, n_meas=1, fp64=False, flags=mp.FLAG_TWO_START),
        # the smallest call: one lattice, few paths, everything from create to destroy
        dict(name="call_L8", kind="call", lattice="sc", L="8", paths="64", T0=1.44, T1=1.44, nT=1, J=1.0,
             h=0.0, n_therm=20, n_meas=20, fp64=False, flags=0),
        # fitting couplings: observables and their gradients at 22 (beta, h) pairs
        dict(name="gradient_L16", kind="gradient", lattice="sc", L="16", paths="4096", b0=0.6, b1=0.8,
             nb=11, h1=0.01, J=1.0, n_therm=20, n_meas=20, fp64=False),
        # the same on the 64-spin open chain, where the answer is known in closed form
        dict(name="gradient_chain64", kind="gradient", lattice="chain", L="64", paths="4096", b0=0.6,
             b1=0.8, nb=11, h1=0.01, J=1.0, n_therm=250, n_meas=250, fp64=False),
        # the Ising model of the paper's appendix, around its T_C
        dict(name="ising_L60", kind="run", lattice="ising", L="60", paths="10000", T0=1.0, T1=3.0, nT=4,
             J=1.0, h=0.0, n_therm=50, n_meas=100, fp64=False, flags=0),
        # the paper's literal order, N attempts at random sites per sweep
        dict(name="random_order_L10", kind="run", lattice="sc", L="10", paths="10000", T0=1.0, T1=1.0,
             nT=1, J=1.0, h=0.0, n_therm=10, n_meas=10, fp64=False, flags=mp.FLAG_RANDOM_SITE),
    ]


# ---------------------------------------------------------------- drawing --
# Attempts per pass of a drawn case, by the kernel family it runs on: from a
# small call to no more than the family's listed case.
RANGES = {
    "sc": (2e6, 2e10), "batch": (1e7, 8e9), "stream": (2e7, 5e9), "fp64": (2e6, 3e8),
    "chain": (1e6, 2.5e9), "ising": (2e7, 2e10), "random": (1e6, 1.8e8), "call": (1e5, 1e8),
    "gradient": (5e7, 1e10),
}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    return 2 * rng.randint(lo // 2, hi // 2)


def _schedule(rng, sites, attempts):
    """Paths, thermalisation and measurement sweeps for about so many attempts of all systems."""
    paths = max(1, min(int(_log(rng, 8, 10000)), int(attempts / sites / _log(rng, 6, 200))))
    sweeps = max(4, min(3000, int(attempts / sites / paths)))
    n_meas = 1 if rng.random() < 0.3 else max(1, int(sweeps * rng.uniform(0.2, 0.8)))
    return paths, sweeps - n_meas, n_meas


def draw(rng):
    fam = rng.choice(sorted(RANGES))
    attempts = _log(rng, *RANGES[fam])
    nT = rng.choice([1, 1, 2, 3, 5, 21])
    T0 = rng.uniform(0.5, 2.0)
    case = dict(kind="run", lattice="sc", T0=T0, T1=T0 + rng.uniform(0.05, 0.6), nT=nT,
                J=rng.choice([1.0, 1.0, 1.0, -1.0, 0.7]), h=rng.choice([0.0, 0.0, 0.01, 0.3]), fp64=False,
                flags=rng.choice([0, 0, mp.FLAG_TWO_START]))
    if fam in ("sc", "call"):
        sizes = [_even(rng, 4, 26 if fam == "sc" else 16)]
    elif fam == "batch":
        sizes = sorted(rng.sample([6, 8, 10, 12, 14, 16, 18, 20, 22, 24, 26, 30, 32], rng.randint(2, 5)))
    elif fam == "stream":
        sizes = [rng.choice([28, 30, 34, 36, 40, 44, 48, 50, 56, 60, 64])]
    elif fam == "fp64":
        case["fp64"] = True
        sizes = [_even(rng, 4, 20)] if rng.random() < 0.7 else [_even(rng, 22, 46)]
        if rng.random() < 0.25:
            case["lattice"] = "chain"
            sizes = [rng.randint(8, 512)]
    elif fam == "chain":
        case["lattice"] = "chain"
        sizes = [int(_log(rng, 3, 2000))]
    elif fam == "ising":
        case["lattice"] = "ising"
        sizes = [_even(rng, 8, 128)]
    elif fam == "random":
        case["flags"] = mp.FLAG_RANDOM_SITE
        sizes = [_even(rng, 4, 16)]
        if rng.random() < 0.2:
            case["lattice"] = "chain"
            sizes = [rng.randint(8, 512)]
    else:  # gradient
        lattice = rng.choice(["sc", "chain"])
        L = _even(rng, 4, 20) if lattice == "sc" else rng.randint(8, 256)
        nb = rng.randint(1, 11)
        sites = L ** 3 if lattice == "sc" else L
        paths, n_therm, n_meas = _schedule(rng, 2 * nb * sites, min(attempts, RANGES["chain"][1] if lattice == "chain"
                                                                    else attempts))
        b0 = rng.uniform(0.4, 0.8)
        return dict(kind="gradient", lattice=lattice, L=str(L), paths=str(max(2, paths)), b0=b0,
                    b1=b0 + rng.uniform(0.05, 0.4), nb=nb, h1=rng.choice([0.01, 0.2]), J=1.0, n_therm=n_therm,
                    n_meas=n_meas, fp64=False)
    if fam == "call":
        case.update(kind="call", nT=1, flags=0)
    n = len(sizes)
    power = {"sc": 3, "chain": 1, "ising": 2}[case["lattice"]]
    # smaller lattices of a batch get more paths, as in a finite-size study
    share = [max(sizes) ** power / s ** power for s in sizes]
    share = [min(32.0, v) for v in share]
    sites = sum(v * s ** power for v, s in zip(share, sizes)) * case["nT"]
    paths, case["n_therm"], case["n_meas"] = _schedule(rng, sites, attempts)
    case["L"] = ",".join(str(s) for s in sizes)
    case["paths"] = ",".join(str(max(2, int(paths * share[k]))) for k in range(n))
    return case


# ------------------------------------------------------------------- path --
def _lin(a, b, n):
    return [a + (b - a) * k / (n - 1) if n > 1 else a for k in range(n)]


def _systems(case):
    """The batch of a case: every size at every temperature (or every (beta, h) pair)."""
    lat = LATTICES[case["lattice"]]
    sizes = [int(v) for v in case["L"].split(",")]
    paths = [int(v) for v in case["paths"].split(",")]
    if case["kind"] == "gradient":
        return [mp.System(L, 1.0 / b, case["J"], h, P, lat)
                for L, P in zip(sizes, paths) for h in (0.0, case["h1"]) for b in _lin(case["b0"], case["b1"], case["nb"])]
    return [mp.System(L, T, case["J"], case["h"], P, lat)
            for L, P in zip(sizes, paths) for T in _lin(case["T0"], case["T1"], case["nT"])]


def prepare(case, seed):
    precision = mp.FP64 if case["fp64"] else mp.FP32
    state = dict(case=case, seed=seed, systems=_systems(case))
    if case["kind"] == "run":
        state["sim"] = mp.Simulation(state["systems"], case["n_therm"], case["n_meas"], seed=seed,
                                     precision=precision, flags=case["flags"])
    elif case["kind"] == "gradient":
        state["beta"] = torch.tensor([1.0 / s.T for s in state["systems"]], dtype=torch.float64, requires_grad=True)
        state["h"] = torch.tensor([s.h for s in state["systems"]], dtype=torch.float64, requires_grad=True)
        # the loss's weights of <e> and <|m|> at each point
        gen = torch.Generator().manual_seed(seed)
        state["w"] = torch.rand(2, len(state["systems"]), generator=gen, dtype=torch.float64) + 0.5
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "call":
        s = state["systems"][0]
        est = mp.simulate(s.L, s.T, J=s.J, h=s.h, n_paths=s.n_paths, n_therm=case["n_therm"],
                          n_meas=case["n_meas"], seed=state["seed"],
                          precision=mp.FP64 if case["fp64"] else mp.FP32)
        return {"estimates": {f: est[f] for f in RESULTS}}
    if case["kind"] == "gradient":
        s = state["systems"][0]
        state["beta"].grad = state["h"].grad = None
        e, m = mp_autograd.observables(state["beta"], state["h"], L=s.L, n_paths=s.n_paths, n_therm=case["n_therm"],
                                       n_meas=case["n_meas"], J=s.J, lattice=s.lattice, seed=state["seed"],
                                       precision=mp.FP64 if case["fp64"] else mp.FP32)
        (state["w"][0] * e + state["w"][1] * m).sum().backward()
        return {"e": e.detach(), "m": m.detach(), "grad_beta": state["beta"].grad, "grad_h": state["h"].grad}
    sim = state["sim"]
    sim.run()
    est = [sim.estimates(k) for k in range(len(state["systems"]))]
    # the handle's record buffer is overwritten by its next run: keep these
    return {"records": sim.device_records().clone(),
            "estimates": {f: np.array([e[f] for e in est]) for f in RESULTS}}


def _attempts(case):
    return sum(s.N * s.n_paths for s in _systems(case)) * (case["n_therm"] + case["n_meas"])


def work(case):
    systems = _systems(case)
    out = 8.0 * len(RESULTS) * len(systems)
    if case["kind"] == "run":
        out += 8.0 * mp.NREC * sum(s.n_paths for s in systems)
    return {"bytes": out, "flops": OPS[case["lattice"]] * _attempts(case)}


# ------------------------------------------------------------------ exact --
# The method in plain torch, 64 bits: the same counters and uniforms (the FP32
# form's are the 23-bit ones), every other number in float64.
_M0, _M1, _MASK = 0xD2511F53, 0xCD9E8D57, 0xFFFFFFFF
_TAG_UPDATE, _TAG_INIT, _TAG_SITE, _TAG_ISING = 0, 1, 2, 4


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of int64 tensors holding 32-bit words."""
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = c0 * _M0, c2 * _M1  # wraps: the low 64 bits are the product
        c0, c1, c2, c3 = (((p1 >> 32) & _MASK) ^ c1 ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ c3 ^ k1, p0 & _MASK)
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c0, c1, c2, c3


def _uniform(r, fp64):
    return (r.double() + 0.5) * 2.0 ** -32 if fp64 else ((r >> 9).double() * 2.0 + 1.0) * 2.0 ** -24


def _direction(r0, r1, fp64):
    z = 2.0 * _uniform(r0, fp64) - 1.0
    rad, phi = ((1.0 - z) * (1.0 + z)).sqrt(), 2.0 * math.pi * _uniform(r1, fp64)
    return torch.stack([rad * phi.cos(), rad * phi.sin(), z])


def _geometry(lattice, L):
    """(neighbours (sites, k), site N standing for none; colour (sites,)) of a lattice."""
    if lattice == mp.CHAIN:
        i = np.arange(L)
        return np.stack([np.where(i > 0, i - 1, L), np.where(i < L - 1, i + 1, L)], 1), i % 2
    d = 3 if lattice == mp.SC else 2
    i = np.arange(L ** d)
    c = [(i // L ** k) % L for k in range(d)]
    nb = [i + ((c[k] + s) % L - c[k]) * L ** k for k in range(d) for s in (1, -1)]
    return np.stack(nb, 1), sum(c) % 2


def _records(case, systems, seed, group, dev):
    """Per-path records of the systems in `group` (one lattice and size)."""
    fp64, flags = case["fp64"], case.get("flags", 0)
    s0 = systems[group[0]]
    N, ising = s0.N, s0.lattice == mp.ISING
    nb, colour = _geometry(s0.lattice, s0.L)
    nb = torch.from_numpy(nb).to(dev)
    each = [systems[k].n_paths for k in group]
    path = torch.cat([torch.arange(n, device=dev) for n in each])[:, None]
    many = torch.tensor(each, device=dev)
    col = lambda v, dtype: torch.tensor(v, dtype=dtype, device=dev).repeat_interleave(many)[:, None]  # noqa: E731
    sysw = col([k << 8 for k in group], torch.int64)
    beta, J, h = (col([f(systems[k]) for k in group], torch.float64)
                  for f in (lambda s: 1.0 / s.T, lambda s: s.J, lambda s: s.h))
    ordered = (path >= col([n - n // 2 for n in each], torch.int64)) & bool(flags & mp.FLAG_TWO_START)
    out = []
    step = max(1, (1 << 24) // N)
    for a in range(0, len(path), step):
        cut = slice(a, a + step)
        out.append(_walk(case, N, s0.L, nb, torch.from_numpy(colour).to(dev), path[cut], sysw[cut], beta[cut], J[cut], h[cut], ordered[cut],
                         seed, fp64, ising, bool(flags & mp.FLAG_RANDOM_SITE)))
    return torch.cat(out)


def _walk(case, N, L, nb, colour, path, sysw, beta, J, h, ordered, seed, fp64, ising, random_site):
    dev, P, f64 = path.device, len(path), torch.float64
    i = torch.arange(N, device=dev)[None]
    zero = torch.zeros((), dtype=torch.int64, device=dev)
    r = _philox(i + 0 * path, zero, path, sysw | _TAG_INIT, seed)
    if ising:
        S = 1.0 - 2.0 * (~ordered & (r[0] >> 31 == 1)).double()[None]
    else:
        S = torch.where(ordered, torch.tensor([0.0, 0.0, 1.0], dtype=f64, device=dev)[:, None, None], _direction(r[0], r[1], fp64))
    S = torch.cat([S, torch.zeros(S.shape[0], P, 1, dtype=f64, device=dev)], 2)  # site N: no neighbour
    acc = torch.zeros(P, 20, dtype=f64, device=dev)
    accepted = torch.zeros(P, dtype=f64, device=dev)
    rows = torch.arange(P, device=dev)
    bonds = nb[:, 1:2] if nb.shape[1] == 2 else nb[:, 0::2]
    sites = [torch.nonzero(colour == c)[:, 0] for c in (0, 1)]

    def field(S, at):
        f = S.index_select(2, nb[at, 0])
        for k in range(1, nb.shape[1]):
            f = f + S.index_select(2, nb[at, k])
        return f

    sweeps = case["n_therm"] + case["n_meas"]
    for s in range(sweeps):
        sw = zero + s
        if random_site:
            r = _philox(i + 0 * path, sw, path, sysw | _TAG_SITE, seed)
            at = ((r[3] * 2 + 1) * N) >> 33
            t, u = _direction(r[0], r[1], fp64), _uniform(r[2], fp64)
            for a in range(N):
                j = at[:, a]
                f = S[:, rows[:, None], nb[j]].sum(2)
                d = t[:, :, a] - S[:, rows, j]
                dE = -J[:, 0] * (d * f).sum(0) - h[:, 0] * d[2]
                ok = (dE <= 0) | (u[:, a] < (-beta[:, 0] * dE).exp())
                S[:, rows, j] = torch.where(ok, t[:, :, a], S[:, rows, j])
                accepted += ok
        for c, at in enumerate([] if random_site else sites):
            f, old = field(S, at), S.index_select(2, at)
            if ising:
                x, y = at % L, at // L
                w = torch.stack(_philox(torch.arange((L // 2) * ((L + 3) // 4), device=dev)[None] + 0 * path, sw, path,
                                        sysw | (_TAG_ISING + c), seed))
                u = _uniform(w[y % 4, :, x // 2 + (L // 2) * (y // 4)].T, True)
                dE = 2.0 * old[0] * (J * f[0] + h)
                ok, new = (dE <= 0) | (u < (-beta * dE).exp()), -old
            else:
                r = _philox(at[None] + 0 * path, sw, path, sysw | _TAG_UPDATE, seed)
                new = _direction(r[0], r[1], fp64)
                d = new - old
                dE = -J * (d * f).sum(0) - h * d[2]
                ok = (dE <= 0) | (_uniform(r[2], fp64) < (-beta * dE).exp())
            S[:, :, at] = torch.where(ok, new, old)
            accepted += ok.sum(1)
        if s < case["n_therm"]:
            continue
        eb = sum((S[:, :, :N] * S.index_select(2, bonds[:, k])).sum((0, 2)) for k in range(bonds.shape[1]))
        M = torch.cat([torch.zeros(3 - S.shape[0], P, dtype=f64, device=dev), S.sum(2)])
        mx, my, mz = M / N
        e = (-J[:, 0] * eb - h[:, 0] * M[2]) / N
        m2 = mx * mx + my * my + mz * mz
        m = m2.sqrt()
        now = torch.stack([e, e * e, m, m2, m2 * m2, mx, my, mz, mz * mz, mz.abs(), e * m, e * mz, m * mz], 1)
        acc[:, :13] += now / case["n_meas"]
        acc[:, 13:17] = torch.stack([mx, my, mz, e], 1)
    acc[:, mp.REC["acc"]] = accepted / (float(sweeps) * N)
    acc[:, mp.REC["norm"]] = 0.0 if ising else (S[:, :, :N].square().sum(0).sqrt() - 1.0).abs().amax(1)
    return acc


def _derived(mu, N, beta):
    e, e2, m, m2, m4, mz, mz2, em, emz, mmz = (mu[..., mp.REC[f]] for f in ("e", "e2", "m", "m2", "m4", "mz", "mz2", "em", "emz", "mmz"))
    return dict(chi=N * beta * (m2 - m * m), cv=N * beta ** 2 * (e2 - e * e), binder=1.0 - m4 / (3.0 * m2 * m2),
                de_dbeta=-N * (e2 - e * e), dm_dbeta=-N * (em - m * e), dmz_dbeta=-N * (emz - mz * e),
                de_dh=beta * N * (emz - e * mz) - mz, dm_dh=beta * N * (mmz - m * mz), dmz_dh=beta * N * (mz2 - mz * mz))


def _estimates(rec, s):
    """One system's estimates from its records (paths, 20)."""
    P, beta = rec.shape[0], 1.0 / s.T
    mean = rec.mean(0)
    se = rec.std(0) / math.sqrt(P)
    est = {}
    for f in ("e", "e2", "m", "m2", "m4", "mx", "my", "mz", "mz2", "amz", "acc"):
        est[f], est[f + "_se"] = mean[mp.REC[f]], se[mp.REC[f]]
    full, loo = _derived(mean, s.N, beta), _derived((rec.sum(0) - rec) / (P - 1), s.N, beta)
    for f in full:
        est[f] = full[f]
        est[f + "_se"] = ((P - 1) / P * (loo[f] - loo[f].mean()).square().sum()).sqrt()
    est["cv_m"] = est["m_se"] / est["m"]
    q = torch.special.ndtri((torch.arange(P, device=rec.device, dtype=torch.float64) + 0.5) / P)
    dq = q - q.mean()
    for f in ("e", "m", "mx", "my", "mz", "amz"):
        dx = rec[:, mp.REC[f]].sort().values - mean[mp.REC[f]]
        sxx = dx.square().sum()
        est["r_" + f] = (dx * dq).sum() ** 2 / (sxx * dq.square().sum()) if P >= 3 and sxx > 0 else torch.tensor(math.nan)
    half, z = P - P // 2, []
    for f in ("e", "m"):
        a, b = rec[:half, mp.REC[f]], rec[half:, mp.REC[f]]
        for n, v in (("a", a), ("b", b)):
            est["%s_%s" % (f, n)] = v.mean()
            est["%s_%s_se" % (f, n)] = v.std() / math.sqrt(len(v)) if len(v) > 1 else torch.tensor(math.nan)
        z.append((est[f + "_a"] - est[f + "_b"]).abs().cpu() / (est[f + "_a_se"].cpu() ** 2 + est[f + "_b_se"].cpu() ** 2).sqrt())
    est["start_z"] = torch.fmax(z[0], z[1])
    return {f: float(est[f]) for f in RESULTS}


def exact(case, seed):
    systems = _systems(case)
    rate = {"sc": 5e8, "chain": 5e8, "ising": 1.5e9}[case["lattice"]]  # attempts/s of this plain form
    steps = case["n_therm"] + case["n_meas"]
    if case.get("flags", 0) & mp.FLAG_RANDOM_SITE:
        steps *= max(s.N for s in systems) / 6
    if _attempts(case) / rate + steps * 2e-3 * len(set(s.L for s in systems)) > 15.0 or min(s.n_paths for s in systems) < 2:
        return None
    # In the FP32 form an accept test that falls on the other side of its rounding makes the rest
    # of that path another sample of the same distribution: long paths have no value of their own
    # in 64 bits, and of short ones the quantities that are zero by symmetry but for noise have none.
    single = not case["fp64"] and case["lattice"] != "ising"
    if single and max(s.N for s in systems) * (case["n_therm"] + case["n_meas"]) > 1e6:
        return None
    noise = ("mx", "my", "mz", "dmz_dbeta", "de_dh", "dm_dh", "r_e", "r_m", "r_mx", "r_my", "r_mz", "r_amz", "start_z")
    value = lambda f, v: None if single and f in noise else v  # noqa: E731
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rec = [None] * len(systems)
    for L in sorted(set(s.L for s in systems)):
        group = [k for k, s in enumerate(systems) if s.L == L]
        rows = _records(case, systems, seed, group, dev).split([systems[k].n_paths for k in group])
        for k, v in zip(group, rows):
            rec[k] = v
    if case["kind"] == "gradient":
        d = [_derived(v.mean(0), s.N, 1.0 / s.T) for v, s in zip(rec, systems)]
        gen = torch.Generator().manual_seed(seed)
        w = torch.rand(2, len(systems), generator=gen, dtype=torch.float64) + 0.5
        pick = lambda f: torch.stack([x[f].cpu() for x in d])  # noqa: E731
        mean = torch.stack([v.mean(0).cpu() for v in rec])
        return {"e": mean[:, mp.REC["e"]], "m": mean[:, mp.REC["m"]],
                "grad_beta": w[0] * pick("de_dbeta") + w[1] * pick("dm_dbeta"),
                "grad_h": None if single else w[0] * pick("de_dh") + w[1] * pick("dm_dh")}
    est = [_estimates(v, s) for v, s in zip(rec, systems)]
    if case["kind"] == "call":
        return {"estimates": {f: value(f, est[0][f]) for f in RESULTS}}
    return {"records": torch.cat(rec), "estimates": {f: value(f, np.array([e[f] for e in est])) for f in RESULTS}}
