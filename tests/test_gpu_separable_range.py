"""The separable transforms over the range of floats: they are linear, so input
times a power of two gives exactly the output times it, as long as no partial sum
leaves the normal numbers."""
import pytest

torch = pytest.importorskip("torch")

from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [104, 90, -90, -104])
def test_scaled_inputs(k):
    from paper_2505_08777_gb300 import Hologram
    p = random_problem(17, 640, 610, 70, list(range(2, 12)))
    amp, C = torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda()
    amp = 0.5 + 0.5 * amp / amp.max()                    # no value far below the others
    ph = torch.from_numpy(p.phase0).cuda()
    y = torch.polar(torch.linspace(0.5, 1.0, p.N), torch.arange(p.N, dtype=torch.float32)).cuda()
    f = 2.0**k
    h, hk = Hologram(amp, C, noll=p.noll), Hologram(amp * f, C, noll=p.noll)
    assert h.launch_info()["kernels"] & 48 == 48
    g, gk = torch.view_as_real(h.adjoint(y)[0]), torch.view_as_real(h.adjoint(y * f)[0])
    keep = g.abs() * f >= 2.0**-124
    assert torch.equal(gk[keep], g[keep] * f) and keep.float().mean() > 0.9
    E, Ek = torch.view_as_real(h.forward(ph)), torch.view_as_real(hk.forward(ph))
    keep = E.abs() * f >= 2.0**-124
    assert torch.isfinite(Ek).all() and torch.allclose(Ek[keep] / f, E[keep], rtol=2e-6, atol=0) and keep.any()
    h.check()
    hk.check()
