"""cta_threads without threads_per_path: the default threads per path fit the CTA.

The planner gives paths more threads where a launch has few of them, but not more
than the CTA that the caller asks for; what it picks changes no record.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


@pytest.mark.parametrize("lattice,L,P,precision,cta", [
    (mp.SC, 10, 64, mp.FP32, 128), (mp.SC, 10, 64, mp.FP32, 32), (mp.SC, 20, 64, mp.FP32, 256),
    (mp.SC, 20, 64, mp.FP32, 160), (mp.SC, 16, 40, mp.FP32, 128), (mp.SC, 16, 3000, mp.FP64, 128),
    (mp.SC, 16, 40, mp.FP64, 128), (mp.SC, 20, 40, mp.FP64, 256), (mp.SC, 8, 40, mp.FP64, 32),
    (mp.ISING, 60, 100, mp.FP32, 128), (mp.ISING, 60, 100, mp.FP32, 256), (mp.ISING, 256, 20, mp.FP32, 256),
    (mp.ISING, 100, 1000, mp.FP32, 96)])
def test_defaults_fit_the_given_cta(lattice, L, P, precision, cta):
    recs = []
    for c in (cta, 0):
        s = mp.System(L, 1.3, J=0.9, h=0.1, n_paths=P, lattice=lattice)
        with mp.Simulation([s], 2, 19, seed=6, precision=precision, cta_threads=c) as sim:
            if c:
                assert sim.plan()["cta_threads"] == c
            sim.run()
            recs.append(sim.paths(0))
    np.testing.assert_array_equal(recs[0], recs[1])


def test_a_cta_below_the_threads_that_order_fp32_sums_is_refused():
    with pytest.raises(mp.MPError) as ei:
        mp.Simulation([mp.System(20, 1.0, n_paths=64)], 1, 1, cta_threads=128)
    assert ei.value.status == mp.MP_EINVAL


@pytest.mark.parametrize("L,paths", [(10, 3), (16, 3), (20, 2)])
def test_few_fp32_paths_get_more_threads_than_order_their_sums(L, paths):
    with mp.Simulation([mp.System(L, 1.4, n_paths=paths)], 20, 20) as sim:
        plan, system = sim.plan(), sim.system_plan(0)
        # the CTA has no threads beyond its paths'
        assert plan["cta_threads"] > system["paths_per_cta"] * system["threads_per_path"]
