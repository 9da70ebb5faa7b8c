"""The spot-intensity loss at its degenerate sizes: the intensity of a single
spot over its own mean is 1 whatever the field, so the loss is (1 - t)^2 and its
gradient exactly 0."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_single_spot_has_no_gradient():
    from paper_2505_08777_gb300.autograd import spot_intensity_loss
    rng = np.random.default_rng(8)
    t = torch.tensor([0.7], device="cuda")
    for z in rng.normal(size=(200, 2)) * 10.0 ** rng.uniform(-6, 6, (200, 1)):
        E = torch.tensor([complex(*z)], dtype=torch.complex64, device="cuda", requires_grad=True)
        loss = spot_intensity_loss(E, t)
        (g,) = torch.autograd.grad(loss, [E])
        assert g.abs().item() == 0.0
        assert abs(loss.item() - 0.09) <= 1e-7
