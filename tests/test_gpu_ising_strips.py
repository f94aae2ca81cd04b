"""The Ising kernel's strips against the oracle, bit for bit, where they can go wrong.

Whole and ragged last row blocks (L % 4 = 0 and 2), one block only (L = 2, 4),
segments of every length (thread counts from one warp to 1024), the largest
lattice, thresholds that include 0 and 2^32 (the 64-bit test, low T) or not, and
a schedule cut at a checkpoint (saved spins are +-1 bytes).
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


@pytest.mark.parametrize("T,J,h", [(2.269, 1.0, 0.0), (0.2, 1.0, 0.0), (0.25, -1.0, 0.4)])
@pytest.mark.parametrize("L,P,tp", [(2, 5, 0), (4, 5, 0), (6, 5, 32), (14, 4, 64), (16, 4, 0), (34, 3, 96),
                                    (62, 3, 32), (100, 2, 128), (256, 1, 0), (254, 1, 1024)])
def test_ising_strips_match_the_oracle(L, P, tp, T, J, h):
    s = [mp.System(L, T, J, h, P, mp.ISING)]
    ref, rsp = O.run([O.System(L=L, T=T, J=J, h=h, n_paths=P, lattice=O.ISING)], 2, 3, seed=3, want_spins=True)
    with mp.Simulation(s, 2, 3, seed=3, keep_spins=True, threads_per_path=tp) as sim:
        sim.run()
        rec, spins = sim.paths(0), np.stack([sim.spins(0, p) for p in range(P)])
    np.testing.assert_array_equal(spins, rsp[0])
    np.testing.assert_array_equal(rec[:, 17], ref[0][:, 17])
    np.testing.assert_allclose(rec[:, :17], ref[0][:, :17], rtol=1e-12, atol=1e-14)
    with mp.Simulation(s, 2, 3, seed=3, threads_per_path=tp) as sim:
        sim.run_sweeps(1)
        blob = sim.checkpoint()
    with mp.Simulation(s, 2, 3, seed=3, threads_per_path=tp) as sim:
        sim.restore(blob)
        sim.run_sweeps(4)
        np.testing.assert_allclose(sim.paths(0)[:, :17], rec[:, :17], rtol=1e-12, atol=1e-14)
