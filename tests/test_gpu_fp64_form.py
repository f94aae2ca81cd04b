"""The FP64 form's accept test where its FP32 stage cannot decide, against the oracle.

Trajectories differ from the oracle's only by rounding (1e-12) and every accept
decision is the same, at temperatures from T -> 0 (every test undecided or
frozen) to T -> infinity, strong fields, either sign of J and J = 0.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


@pytest.mark.parametrize("T,J,h", [(1e-300, 1.0, 0.0), (1e-3, 1.0, 0.1), (0.05, -1.0, 0.0), (0.5, 1.0, 50.0),
                                   (1.5, 0.0, 0.3), (1.5, 0.0, 0.0), (2.0, -0.7, -2.0), (1e6, 1.0, 1.0)])
@pytest.mark.parametrize("lattice,L,P", [(mp.SC, 2, 5), (mp.SC, 6, 8), (mp.SC, 22, 2), (mp.CHAIN, 33, 6)])
def test_accept_decisions_match_the_oracle(T, J, h, lattice, L, P):
    s = mp.System(L, T, J, h, P, lattice)
    with mp.Simulation([s], 1, 5, seed=7, precision=mp.FP64, keep_spins=True) as sim:
        sim.run()
        rec, spins = sim.paths(0), np.stack([sim.spins(0, p) for p in range(P)])
    ref, rspins = O.run([O.System(L=L, T=T, J=J, h=h, n_paths=P, lattice=lattice)], 1, 5, seed=7, want_spins=True)
    np.testing.assert_array_equal(rec[:, 17], ref[0][:, 17])  # acceptance
    np.testing.assert_allclose(spins, rspins[0], rtol=0, atol=1e-12)
    np.testing.assert_allclose(rec[:, :17], ref[0][:, :17], rtol=1e-10, atol=1e-13 * max(1.0, abs(h)))
