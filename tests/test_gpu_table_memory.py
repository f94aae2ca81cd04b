"""Device memory of a batch of many systems of one size: they share their unit
tables, so what a system adds is its paths' records, not a table (281 KB at L = 26)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def _bytes(n, flags):
    before = torch.cuda.memory_allocated()
    with mp.Simulation([mp.System(26 - 2 * (k % 2), 1.0 + 1e-3 * k, n_paths=1) for k in range(n)], 1, 1, flags=flags) as sim:
        used = torch.cuda.memory_allocated() - before
        if n < 10:
            sim.run()
            assert sim.estimates(n - 1)["n_paths"] == 1
    return used


@pytest.mark.parametrize("flags", [0, mp.FLAG_AUTOTUNE])
def test_systems_of_one_size_share_their_tables(flags):
    few, many = _bytes(4, flags), _bytes(404, flags)
    assert (many - few) / 400 < 4096


def test_the_autotuner_has_room_for_every_table():
    """While it tries a count on the first system of a size, the others of that
    size have the default's: a candidate that found no room would be passed over."""
    systems = [mp.System(L, 1.2, n_paths=2) for L in (10, 12, 10, 12, 10)]
    with mp.Simulation(systems, 3, 3, flags=mp.FLAG_AUTOTUNE) as sim:
        tp = [sim.system_plan(k)["threads_per_path"] for k in range(5)]
        assert tp[0] == tp[2] == tp[4] and tp[1] == tp[3]
        sim.run()
        recs = [sim.paths(k) for k in range(5)]
    with mp.Simulation(systems, 3, 3, flags=mp.FLAG_DEVICE_UNITS) as sim:
        sim.run()
        for k, r in enumerate(recs):
            assert abs(sim.paths(k)[:, 13:16] - r[:, 13:16]).max() < 1e-5
