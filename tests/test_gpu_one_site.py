"""The one-site form where threads have no site (L = 2, 4, short chains).

Threads without a site of a colour must not touch its spins, which the others
write.  The site arithmetic does not depend on the form, so spins and
acceptances equal those of the kernel for batches of uneven sizes, which takes
the general walk, bit for bit.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def _run(systems, precision):
    n = systems[0].n_paths
    with mp.Simulation(systems, 9, 2, seed=4, precision=precision, keep_spins=True) as sim:
        sim.run()
        return np.stack([sim.spins(0, p) for p in range(n)]), sim.paths(0)[:, 17]


@pytest.mark.parametrize("precision", [mp.FP64, mp.FP32])
@pytest.mark.parametrize("lattice,L,P", [(mp.SC, 2, 40), (mp.SC, 4, 9), (mp.CHAIN, 2, 33), (mp.CHAIN, 5, 3),
                                         (mp.CHAIN, 63, 4), (mp.CHAIN, 64, 700)])
def test_one_site_form_equals_the_general_walk(lattice, L, P, precision):
    system = mp.System(L, 0.8, J=-0.9, h=0.2, n_paths=P, lattice=lattice)
    other = mp.System(6, 1.0, n_paths=1)
    spins, acc = _run([system], precision)
    ref, ref_acc = _run([system, other], precision)
    np.testing.assert_array_equal(spins, ref)
    np.testing.assert_array_equal(acc, ref_acc)
