"""One ensemble split by path ids, with the planner's own layouts.

A part of an ensemble may get other threads per path than the whole (the planner
goes by the paths per SM).  A path's record is the same bit for bit all the same:
FP32 sums keep the order of a number of threads that depends on the lattice
alone, FP64 and Ising sums are exact integers rounded once and then added over
the sweeps in one order.  Random-site paths take a thread or a warp each.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402

CASES = [  # (lattice, L, paths of the whole, paths of the part, flags)
    (mp.SC, 4, 5000, 60, 0), (mp.SC, 6, 4000, 60, 0), (mp.SC, 8, 3000, 60, 0), (mp.SC, 12, 1200, 40, 0),
    (mp.SC, 14, 600, 40, 0), (mp.SC, 16, 500, 40, 0), (mp.SC, 18, 320, 30, 0), (mp.CHAIN, 64, 5000, 40, 0),
    (mp.CHAIN, 1001, 600, 20, 0), (mp.SC, 24, 320, 20, mp.FLAG_STREAM),
    (mp.SC, 2, 5000, 60, mp.FLAG_RANDOM_SITE), (mp.CHAIN, 16, 5000, 60, mp.FLAG_RANDOM_SITE),
    (mp.CHAIN, 9, 5000, 60, mp.FLAG_RANDOM_SITE),
    (mp.ISING, 6, 5000, 60, 0), (mp.ISING, 34, 5000, 60, 0), (mp.ISING, 60, 6000, 60, 0), (mp.ISING, 100, 3000, 60, 0),
    (mp.ISING, 200, 700, 30, 0),
]


def _records(lattice, L, n, begin, flags, precision):
    systems = [mp.System(L, 1.3, J=0.9, h=0.1, n_paths=n, lattice=lattice, path_begin=begin)]
    with mp.Simulation(systems, 3, 37, seed=9, precision=precision, flags=flags) as sim:
        sim.run()
        return sim.paths(0)


@pytest.mark.parametrize("precision", [mp.FP32, mp.FP64])
@pytest.mark.parametrize("lattice,L,whole,part,flags", CASES)
def test_a_part_reproduces_its_paths_of_the_whole(lattice, L, whole, part, flags, precision):
    begin = 13
    ref = _records(lattice, L, whole, 0, flags, precision)[begin:begin + part]
    np.testing.assert_array_equal(_records(lattice, L, part, begin, flags, precision), ref)


@pytest.mark.parametrize("lattice,L", [(mp.SC, 8), (mp.SC, 16), (mp.ISING, 60)])
def test_exact_sums_do_not_depend_on_the_threads(lattice, L):
    recs = []
    for tp in (32, 96, 256):
        systems = [mp.System(L, 1.3, J=0.9, h=0.1, n_paths=5, lattice=lattice)]
        with mp.Simulation(systems, 2, 33, seed=9, precision=mp.FP64, threads_per_path=tp) as sim:
            sim.run()
            recs.append(sim.paths(0))
    np.testing.assert_array_equal(recs[0], recs[1])
    np.testing.assert_array_equal(recs[0], recs[2])
