"""Acceptance counts of long Ising schedules.

The counts of a warp are moved to the path's total every 2^15 sweeps, so that no
schedule overflows them: exact totals on either side of that, in one call and in
several, with one warp per path and more, against the oracle.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


@pytest.mark.parametrize("L,tp", [(2, 32), (6, 32), (6, 64)])
@pytest.mark.parametrize("T,J,h", [(2.5, 1.0, 0.2), (1.0, 0.0, 0.0)])
@pytest.mark.parametrize("n_therm,n_meas", [(32767, 1), (32768, 1), (32760, 70000)])
def test_acceptance_of_a_long_schedule(L, tp, T, J, h, n_therm, n_meas):
    s = [mp.System(L, T, J, h, 3, mp.ISING)]
    ref = O.run([O.System(L=L, T=T, J=J, h=h, n_paths=3, lattice=O.ISING)], n_therm, n_meas, seed=3)[0][:, 17]
    if J == 0.0 and h == 0.0:
        assert (ref == 1.0).all()
    with mp.Simulation(s, n_therm, n_meas, seed=3, threads_per_path=tp) as sim:
        sim.run()
        np.testing.assert_array_equal(sim.paths(0)[:, 17], ref)
        for part in (32767, 2, 3, 10**6):
            if sim.progress() < n_therm + n_meas:
                sim.run_sweeps(part)
        np.testing.assert_array_equal(sim.paths(0)[:, 17], ref)
