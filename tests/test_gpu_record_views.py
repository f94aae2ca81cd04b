"""device_records() gives a view of its own on every call: what a caller does to
one view's shape or flags does not show in the next."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1305_6758_gb300 as mp  # noqa: E402


def test_views_are_independent():
    with mp.Simulation([mp.System(4, 1.5, n_paths=6)], 1, 2) as sim:
        sim.run()
        sim.estimates()
        view = sim.device_records()
        view.t_()
        view.requires_grad_()
        again = sim.device_records()
        assert again.shape == (6, mp.NREC) and again.is_contiguous() and not again.requires_grad
        assert again.data_ptr() == view.data_ptr()
