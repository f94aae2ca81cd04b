"""The random-site kernels at the sizes where their mapping changes, against the oracle path by path.

A warp takes 32 attempts at a time (sweeps of fewer, of 32 and of 33 attempts,
and lattices so small that almost every attempt waits for an earlier one), its
lattice in shared memory or in HBM (FP64 from L = 14), with site masks shared
modulo 512; many paths of at most 16 sites run one to a thread.  FP64: equal
to rounding.  FP32: rounding can flip a borderline accept, after which that
path is another sample; fewer than one path in 50 is let off.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402

BATCHES = [
    [(mp.CHAIN, 2, 5), (mp.CHAIN, 3, 5), (mp.CHAIN, 31, 4), (mp.CHAIN, 32, 4), (mp.CHAIN, 33, 4)],
    [(mp.SC, 2, 6), (mp.SC, 4, 6), (mp.SC, 10, 4)],
    [(mp.CHAIN, 513, 3), (mp.SC, 14, 2)],
    [(mp.SC, 28, 1), (mp.CHAIN, 9, 3)],
    [(mp.SC, 2, 4870), (mp.CHAIN, 16, 3)],
    [(mp.CHAIN, 2, 2), (mp.CHAIN, 16, 4900)],
]


@pytest.mark.parametrize("precision", [mp.FP64, mp.FP32])
@pytest.mark.parametrize("batch", BATCHES)
def test_random_site_matches_oracle(batch, precision):
    systems = [mp.System(L, 1.2, J=-1.0 if L % 3 else 1.0, h=0.1, n_paths=P, lattice=lat) for lat, L, P in batch]
    osys = [O.System(L=s.L, T=s.T, J=s.J, h=s.h, n_paths=s.n_paths, lattice=s.lattice) for s in systems]
    ref, rspins = O.run(osys, 2, 3, seed=5, order_mode=O.ORDER_RANDOM, want_spins=True, two_start=True)
    with mp.Simulation(systems, 2, 3, seed=5, precision=precision, keep_spins=True,
                       flags=mp.FLAG_RANDOM_SITE | mp.FLAG_TWO_START) as sim:
        sim.run()
        for k, s in enumerate(systems):
            rec = sim.paths(k)
            last = sim.spins(k, s.n_paths - 1)
            if precision == mp.FP64:
                np.testing.assert_array_equal(rec[:, 17], ref[k][:, 17])
                np.testing.assert_allclose(rec[:, :17], ref[k][:, :17], rtol=1e-10, atol=1e-13)
                np.testing.assert_allclose(last, rspins[k][-1], rtol=0, atol=1e-12)
            else:
                off = np.abs(rec[:, :17] - ref[k][:, :17]).max(1) > 1e-5
                assert off.sum() <= max(1, s.n_paths // 50)
