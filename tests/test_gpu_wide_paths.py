"""Paths with more threads than the number that orders their FP32 sums.

With threads_per_path given, exactly that many threads run a path and add up
its sums; by default the planner may launch more, which changes no bit of the
records: the sums are then made by the same number of threads in the same
order after the sweep.  Sizes: every column chunk, one and several paths per
SM, sum orders of one and of several warps, schedules that are all
measurement, all but one thermalisation, and longer than a ring of partial
sums (16 sweeps), with the unit tables and without.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def _run(systems, n_therm, n_meas, flags, tp):
    with mp.Simulation(systems, n_therm, n_meas, seed=11, keep_spins=True, threads_per_path=tp, flags=flags) as sim:
        plan = sim.system_plan(0)
        sim.run()
        return plan, [sim.paths(k) for k in range(len(systems))], [sim.spins(0, p) for p in range(2)]


@pytest.mark.parametrize("L,paths", [(6, 3), (6, 700), (8, 5), (10, 3), (10, 400), (12, 4), (12, 450), (14, 200),
                                     (16, 3), (18, 310), (20, 2), (20, 700), (22, 3), (24, 2), (26, 2)])
@pytest.mark.parametrize("n_therm,n_meas", [(0, 3), (6, 1), (3, 37)])
def test_wide_paths_equal_narrow_paths(L, paths, n_therm, n_meas):
    systems = [mp.System(L, 1.4, J=0.9, h=0.1, n_paths=paths)]
    plan, recs, spins = _run(systems, n_therm, n_meas, 0, 0)
    for flags in (0, mp.FLAG_DEVICE_UNITS):
        _, ref, ref_spins = _run(systems, n_therm, n_meas, flags, plan["threads_per_path"])
        np.testing.assert_array_equal(recs[0], ref[0])
        np.testing.assert_array_equal(spins, ref_spins)
    _, dev, _ = _run(systems, n_therm, n_meas, mp.FLAG_DEVICE_UNITS, 0)
    np.testing.assert_array_equal(recs[0], dev[0])


def test_wide_paths_in_a_batch_and_in_parts():
    """A batch of uneven sizes against its first system alone, and a run in
    parts that stop within a ring (which rounds its sums in other groups)."""
    systems = [mp.System(20, 1.4, h=0.1, n_paths=3), mp.System(12, 1.2, n_paths=4), mp.System(10, 1.1, n_paths=2)]
    _, recs, _ = _run(systems, 5, 21, 0, 0)
    _, alone, _ = _run(systems[:1], 5, 21, 0, 160)
    np.testing.assert_allclose(recs[0], alone[0], rtol=2e-6, atol=2e-7)
    with mp.Simulation(systems, 5, 21, seed=11) as sim:
        for part in (3, 4, 9, 10):
            sim.run_sweeps(part)
        parts = [sim.paths(k) for k in range(3)]
    for a, b in zip(recs, parts):
        np.testing.assert_allclose(a, b, rtol=2e-6, atol=2e-7)
