"""Errors that all pixels share. A spot without tilt and aberrations sums the
nearfield itself, so whatever the pixels' phase factors are off by on average over
a turn adds up over them, where the field's own sum grows with their root only.
For a random field of M pixels: 1e-6 for all errors that differ from pixel to
pixel (3.5e-7 of a turn's rounding, split operands and accumulation) and 2e-9
sqrt(M) for a mean of 2e-9 (cosine 5e-10, the rest of the rounding as much again).
Phases of many turns count as their remainders, which the product with 1 / 2 pi in
two pieces keeps to 2^-25 turns: the same bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import oracle_inputs, rel_err  # noqa: E402
from oracle import transform  # noqa: E402
from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(nx, ny, N, noll):
    p = random_problem(nx + ny + N, nx, ny, N, noll)
    p.coeff[N // 2] = 0.0                                # the spot that sums the field
    p.coeff = np.ascontiguousarray(p.coeff)
    return p


def _holo(p, bits):
    from paper_2505_08777_gb300 import Hologram
    h = Hologram(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), noll=p.noll)
    assert h.launch_info()["kernels"] & bits == bits
    return h


@pytest.mark.parametrize("nx,ny,N,noll", [(901, 888, 17, list(range(2, 12))), (512, 775, 33, [2, 3, 4, 5, 6]),
                                          (450, 431, 70, list(range(2, 12)))])
def test_random_field_and_unwrapped_phase(nx, ny, N, noll):
    p = _problem(nx, ny, N, noll)
    Z, C, A = oracle_inputs(p)
    h = _holo(p, 16)
    rng = np.random.default_rng(N)
    bound = 1e-6 + 2e-9 * np.sqrt(nx * ny)
    f = (p.amp * (rng.normal(size=(ny, nx)) + 1j * rng.normal(size=(ny, nx)))).astype(np.complex64)
    E = h.forward_field(torch.from_numpy(f).cuda()).cpu().numpy()
    ref = transform.forward(f.astype(np.complex128).ravel(), C, Z, workers=8)
    assert rel_err(E, ref) <= bound
    assert abs(E[N // 2] - ref[N // 2]) <= bound * np.sqrt(np.mean(np.abs(ref) ** 2))
    ph = rng.uniform(-500.0, 500.0, (ny, nx)).astype(np.float32)
    E = h.forward(torch.from_numpy(ph).cuda()).cpu().numpy()
    ref = transform.forward(transform.field(A, ph), C, Z, workers=8)
    assert rel_err(E, ref) <= bound
    h.check()
