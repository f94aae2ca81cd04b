"""Every mp_estimates call synchronises the handle's stream, as the header says, also
one that is served from the copy an earlier call made."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def test_each_call_waits_for_the_stream():
    stream = torch.cuda.Stream()
    x = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    with mp.Simulation([mp.System(4, 1.0, n_paths=8), mp.System(4, 1.2, n_paths=8)], 2, 3, stream=stream) as sim:
        sim.run()
        sim.estimates(0)
        for k in (1, 0):
            done = torch.cuda.Event()
            with torch.cuda.stream(stream):
                y = x
                for _ in range(20):  # some milliseconds of the caller's own work
                    y = (y @ x).clamp_(-1.0, 1.0)
                done.record()
            assert sim.estimates(k)["n_paths"] == 8
            assert done.query()
