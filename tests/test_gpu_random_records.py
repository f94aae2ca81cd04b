"""Random-site records: rounding of the per-site values, and placement of the lattices.

The FP32 form's final e, m_x, m_y, m_z are its FP32 sums divided by N, rounded
once in FP64: each equals fl(f / N) for a number f of FP32.  A path's record does
not depend on where its lattice lies (shared memory, or HBM when the batch holds
a system too large for it).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def _records(systems, precision, n_therm=2, n_meas=3):
    with mp.Simulation(systems, n_therm, n_meas, seed=5, precision=precision, flags=mp.FLAG_RANDOM_SITE) as sim:
        sim.run()
        return sim.paths(0)


@pytest.mark.parametrize("lattice,L,P", [(mp.SC, 6, 50), (mp.SC, 10, 50), (mp.CHAIN, 33, 200), (mp.CHAIN, 9, 5000)])
def test_fp32_final_values_are_correctly_rounded(lattice, L, P):
    s = mp.System(L, 1.2, J=0.9, h=0.1, n_paths=P, lattice=lattice)
    got = _records([s], mp.FP32)[:, 13:17]
    sums = got * s.N  # an FP32 number but for the last bits of FP64
    np.testing.assert_array_equal(sums.astype(np.float32).astype(np.float64) / s.N, got)


@pytest.mark.parametrize("precision", [mp.FP32, mp.FP64])
@pytest.mark.parametrize("lattice,L,P", [(mp.SC, 4, 40), (mp.SC, 10, 30), (mp.SC, 14, 6), (mp.CHAIN, 33, 40)])
def test_records_do_not_depend_on_the_placement(lattice, L, P, precision):
    s = mp.System(L, 1.2, J=-0.9, h=0.1, n_paths=P, lattice=lattice)
    np.testing.assert_array_equal(_records([s], precision), _records([s, mp.System(28, 1.0, n_paths=1)], precision))
