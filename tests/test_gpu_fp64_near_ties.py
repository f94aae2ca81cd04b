"""The FP64 form's accept test on moves whose energy change is nearly zero.

A saved state is rewritten so that every site of colour 0 holds a spin a tiny
rotation away from the trial spin that its next attempt will draw: dE between
1e-10 and 1e-5, of either sign, at temperatures where beta dE is far below, near
and far above one.  The accepted moves must be those of a plain FP64
evaluation.  Left out are moves whose FP64 decision itself hangs on rounding:
dE has some ten roundings of numbers up to 6 (1e-14), the exponent as many of
its own size.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402

SEED, HEADER, STATE = 23, 64, 256


def _geometry(lattice, L):
    """Sites of colour 0 with their half indices, and their neighbours."""
    if lattice == mp.CHAIN:
        sites = list(range(0, L, 2))
        return sites, [[j for j in (i - 1, i + 1) if 0 <= j < L] for i in sites]
    sites, nbs = [], []
    for z in range(L):
        for y in range(L):
            for x in range(L):
                if (x + y + z) % 2 == 0:
                    sites.append(x + L * (y + L * z))
                    nbs.append([(x + d) % L + L * (y + L * z) for d in (1, -1)]
                               + [x + L * ((y + d) % L + L * z) for d in (1, -1)]
                               + [x + L * (y + L * ((z + d) % L)) for d in (1, -1)])
    return sites, nbs


def _view(blob, path, n_paths, N):
    """One path's spins in a checkpoint: per colour the (x, y) pairs, then z."""
    NH = (N + 1) // 2
    S = (NH + 1) & ~1
    stride = (STATE + 6 * S * 8 + 255) // 256 * 256
    assert len(blob) == HEADER + n_paths * stride
    a = np.frombuffer(blob, np.float64, 6 * S, HEADER + path * stride + STATE).reshape(2, 3 * S)
    return a, S


def _load(a, S, site, colour):
    h = site >> 1
    return np.array([a[colour, 2 * h], a[colour, 2 * h + 1], a[colour, 2 * S + h]])


@pytest.mark.parametrize("lattice,L,P", [(mp.SC, 6, 40), (mp.SC, 4, 100), (mp.CHAIN, 2, 2000)])
@pytest.mark.parametrize("T,J,h", [(1e-7, 1.0, 0.0), (1e-10, -1.0, 0.0), (1e-30, 1.0, 0.5), (1e-9, 0.0, 1.0),
                                   (1e-5, 1.0, 0.0), (3e-5, 1.0, 0.3), (2e-4, -1.0, 0.0), (0.5, 1.0, 0.2)])
def test_near_ties_are_decided_in_fp64(lattice, L, P, T, J, h):
    rng = np.random.default_rng(5)
    sites, nbs = _geometry(lattice, L)
    N = L ** 3 if lattice == mp.SC else L
    colour = (lambda i: (i % L + i // L % L + i // (L * L)) % 2) if lattice == mp.SC else (lambda i: i % 2)
    system = mp.System(L, T, J=J, h=h, n_paths=P, lattice=lattice)
    with mp.Simulation([system], 1, 3, seed=SEED, precision=mp.FP64) as sim:
        sim.run_sweeps(1)
        blob = bytearray(sim.checkpoint())
        want = {}
        for p in range(P):
            a, S = _view(blob, p, P, N)
            for i, nb in zip(sites, nbs):
                t = O.trial(i, 1, p, 0, SEED)
                w = J * sum(_load(a, S, j, colour(j)) for j in nb) + h * np.array([0.0, 0.0, 1.0])
                perp = w - (w @ t) * t
                size = np.linalg.norm(perp)
                if size < 1e-3:
                    continue
                eta = rng.choice([-1.0, 1.0]) * 10.0 ** rng.uniform(-10.0, -5.0)
                s = t + eta / size * perp / size
                s = np.rint(s / np.linalg.norm(s) * 2.0**53) / 2.0**53
                k = i >> 1
                a[0, 2 * k], a[0, 2 * k + 1], a[0, 2 * S + k] = s
                dE = -(t - s) @ w
                u = (O.philox(i, 1, p, 0, SEED, 0)[2] + 0.5) / 2.0**32
                x = dE / T
                if abs(dE) > 1e-13 and (dE < 0 or abs(np.log(u) + x) > 1e-6 + 1e-13 / T):
                    want[p, i] = (t, s, dE < 0 or np.log(u) < -x)
        sim.restore(bytes(blob))
        sim.run_sweeps(1)
        after = sim.checkpoint()
    wrong = 0
    for (p, i), (t, s, accept) in want.items():
        a, S = _view(after, p, P, N)
        got = _load(a, S, i, 0)
        wrong += not np.abs(got - (t if accept else s)).max() < 1e-13
    assert len(want) > 100
    assert wrong == 0, f"{wrong} of {len(want)}"
