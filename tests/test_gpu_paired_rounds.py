"""Thermalisation sweeps that take their rounds two at a time (FP32, chunks of
two planes: L = 10, 22, 26).

The arithmetic of a site does not depend on the order of the sites of its
colour, so spins after thermalisation agree bit for bit with those of the
mixed-size kernel, which takes one round at a time: with an odd and an even
number of rounds, with whole and ragged last rounds, and with a single round.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def _states(systems, tp):
    paths = systems[0].n_paths
    with mp.Simulation(systems, 7, 1, seed=5, precision=mp.FP32, keep_spins=True, threads_per_path=tp) as sim:
        sim.run()
        return np.stack([sim.spins(0, p) for p in range(paths)]), sim.paths(0)[:, 17]


@pytest.mark.parametrize("L,tp", [(10, 32), (10, 64), (10, 96), (10, 160), (10, 0), (22, 96), (22, 256), (22, 0),
                                  (26, 160), (26, 384), (26, 0)])
@pytest.mark.parametrize("J,h", [(1.0, 0.0), (-0.7, 0.2)])
def test_paired_rounds_equal_single_rounds(L, tp, J, h):
    system = mp.System(L, 1.3, J=J, h=h, n_paths=3)
    spins, accepted = _states([system], tp)
    ref, ref_accepted = _states([system, mp.System(8, 1.0, n_paths=1)], 0)
    np.testing.assert_array_equal(spins, ref)
    np.testing.assert_array_equal(accepted, ref_accepted)
