"""A run captured in a CUDA graph of the caller's and replayed.

A handle without its own graph may be captured.  What it reports after a replay
is the replayed run's, whatever ran in between: its estimates are those of its
records, and a replay that was canceled says so.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


@pytest.mark.parametrize("n_systems", [1, 20])
def test_estimates_follow_a_replayed_run(n_systems):
    stream = torch.cuda.Stream()
    systems = [mp.System(4, 1.0 + 0.1 * k, n_paths=40) for k in range(n_systems)]
    with mp.Simulation(systems, 4, 6, seed=1, graph=False, stream=stream) as sim:
        sim.run()
        first = [sim.estimates(k) for k in range(n_systems)]
        first_paths = sim.paths(n_systems - 1)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            sim.run()
        sim.set_seed(2)
        sim.run()
        second = [sim.estimates(k) for k in range(n_systems)]
        assert all(a["e"] != b["e"] for a, b in zip(first, second))
        with torch.cuda.stream(stream):
            graph.replay()
        for k in range(n_systems):
            got = sim.estimates(k)
            assert [got[f] for f in mp.EST_FIELDS[:52]] == pytest.approx(
                [first[k][f] for f in mp.EST_FIELDS[:52]], rel=0, abs=0, nan_ok=True)
        np.testing.assert_array_equal(sim.paths(n_systems - 1), first_paths)
        sim.cancel()
        with torch.cuda.stream(stream):
            graph.replay()  # nothing clears the flag: the replay stops at its first poll
        with pytest.raises(mp.MPError) as ei:
            sim.estimates(0)
        assert ei.value.status == mp.MP_ECANCELED
        sim.run()  # a direct run clears it
        assert sim.estimates(0)["e"] == second[0]["e"]
