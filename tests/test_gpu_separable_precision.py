"""How exact the separable kernels' gradients and loops are, against the float64
oracle, tighter than the transforms' common tolerances.

Moments of one gradient, per term: two sine / cosine pairs 2 x 3.4e-7, D phase
products reduced modulo a turn 2 pi D 2^-25 = 1.9e-6 at D = 10 (2.6e-6 at 14),
mixed terms dropped 1e-6, u^4 taken as u^2 - 1/8 1e-6, which add up to 4.6e-6
(5.3e-6): 5e-6 of the norm up to D = 10, 6e-6 at D = 14.

Weights of a spot after one iteration: w T / |E_n| of a field whose error is at
most 1e-5 of its largest value, so 1e-5 max|E| / |E_n| of the weight, and the same
of the norm at most: twice that. The field after it: the transforms' 1e-4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import REL_TOL, assert_close, oracle_inputs  # noqa: E402
from oracle import grad as ograd, transform, wgs  # noqa: E402
from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu

LOW = list(range(2, 12))


def _holo(p, bits):
    from paper_2505_08777_gb300 import Hologram
    h = Hologram(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), noll=p.noll)
    assert h.launch_info()["kernels"] & bits == bits
    return h


@pytest.mark.parametrize("nx,ny,N,noll,tol", [
    (905, 903, 161, LOW, 5e-6),
    (901, 930, 20, [2, 3, 4, 5, 6], 5e-6),
    (930, 901, 33, list(range(2, 16)), 6e-6),
])
def test_moments(nx, ny, N, noll, tol):
    p = random_problem(nx + ny + N, nx, ny, N, noll, defocus_max=5.0)
    Z, C, A = oracle_inputs(p)
    E = transform.forward(transform.field(A, p.phase0), C, Z, workers=8)
    gE = ograd.grad_E(E, p.target).astype(np.complex64)
    dph_ref, dC_ref = ograd.backward(A, p.phase0, C, Z, gE.astype(np.complex128))
    h = _holo(p, 16 | 32 | 64)
    dph, dC = h.grad(torch.from_numpy(p.phase0).cuda(), torch.from_numpy(gE).cuda())
    h.check()
    dph, dC = dph.cpu().numpy().astype(np.float64).ravel(), dC.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(dC - dC_ref) <= tol * np.linalg.norm(dC_ref)
    assert np.linalg.norm(dph - dph_ref) <= tol * np.linalg.norm(dph_ref)


@pytest.mark.parametrize("nx,ny,N,noll", [
    (577, 562, 65, LOW),
    (560, 731, 130, [2, 3, 4, 5, 6]),
    (803, 801, 7, LOW),
    (640, 700, 300, LOW),
])
def test_one_iteration(nx, ny, N, noll):
    p = random_problem(nx + ny - N, nx, ny, N, noll, defocus_max=5.0, target_range=(0.5, 1.0))
    Z, C, A = oracle_inputs(p)
    E0 = np.abs(transform.forward(transform.field(A, p.phase0), C, Z, workers=8))
    ref = wgs.run(A, p.phase0, C, Z, p.target, 1, workers=8)
    h = _holo(p, 128 | 256)
    ph, w = torch.from_numpy(p.phase0).cuda().clone(), torch.from_numpy(p.target).cuda().clone()
    E, met = h.wgs(ph, w, torch.from_numpy(p.target).cuda(), 1)
    h.check()
    off = np.abs(w.cpu().numpy().astype(np.float64) - ref.weights) / ref.weights
    assert np.all(off <= 2e-5 * E0.max() / E0)
    assert_close(E.cpu().numpy(), ref.E, REL_TOL, "field")
    assert abs(float(met[0]) - ref.uniformity) <= REL_TOL
