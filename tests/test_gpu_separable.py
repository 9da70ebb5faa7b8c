"""GPU parity of the separable tile transforms (csrc/sep_forward.cu,
csrc/sep_adjoint.cu) at the sizes where the automatic choice takes them:
remainders of 32 and 128 spots, ragged last tiles, row strips from 1 to 32
(coefficients scaled), bases of degree 2 and 4, few spots on a large grid,
bands, and the same calls under capture.

Tolerance of a transform at the workloads' coefficients (scale <= 1), per
term: D products reduced modulo a turn, 2 pi D 2^-25 <= 2.6e-6 for D <= 14;
mixed terms dropped 1e-6; two sine / cosine pairs 2 * 2^-21 = 1e-6; split
operands and accumulation 1e-6: 5.6e-6 if all add up, 1e-5 taken. Stronger
coefficients lose fp32 bits in the phase itself: the transforms' 1e-4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import GRAD_TOL, REL_TOL, assert_close, oracle_inputs  # noqa: E402
from oracle import grad as ograd, transform  # noqa: E402
from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu

LOW = list(range(2, 12))
CASES = [
    # (nx, ny, N, noll, scale of the coefficients)
    (417, 403, 65, LOW, 0.05),
    (403, 417, 64, list(range(2, 16)), 1.0),
    (561, 577, 129, LOW, 1.0),
    (640, 560, 97, LOW, 6.0),
    (560, 575, 160, LOW, 30.0),
    (803, 801, 7, LOW, 1.0),
    (233, 201, 231, [2, 3, 4, 5, 6], 1.0),
    (930, 901, 67, LOW, 1.0),
    (577, 590, 172, LOW, 6.0),
    (901, 930, 20, [2, 3, 4, 5, 6], 1.0),
    (905, 903, 161, LOW, 1.0),
]


def _holo(p):
    from paper_2505_08777_gb300 import Hologram
    return Hologram(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), noll=p.noll)


def _problem(nx, ny, N, noll, scale):
    p = random_problem(nx + ny + N, nx, ny, N, noll, defocus_max=5.0)
    p.coeff = np.ascontiguousarray(p.coeff * np.float32(scale))
    rng = np.random.default_rng(N)
    y = (rng.normal(size=N) + 1j * rng.normal(size=N)).astype(np.complex64)
    return p, y


@pytest.mark.parametrize("nx,ny,N,noll,scale", CASES)
def test_separable_transforms_match_oracle(nx, ny, N, noll, scale):
    from paper_2505_08777_gb300.shard import band_holograms
    p, y = _problem(nx, ny, N, noll, scale)
    tol = 1e-5 if scale <= 1.0 else REL_TOL
    Z, C, A = oracle_inputs(p)
    h = _holo(p)
    ph, yt = torch.from_numpy(p.phase0).cuda(), torch.from_numpy(y).cuda()
    f = transform.field(A, p.phase0)
    E_ref, g_ref = transform.forward(f, C, Z, workers=8), transform.adjoint(y.astype(np.complex128), C, Z, workers=8)
    E = h.forward(ph)
    assert_close(E.cpu().numpy(), E_ref, tol, "forward")
    x = torch.from_numpy(f.reshape(ny, nx).astype(np.complex64)).cuda()
    assert_close(h.forward_field(x).cpu().numpy(), E_ref, tol, "forward of a field")
    g = h.adjoint(yt)[0]
    assert_close(g.cpu().numpy(), g_ref, tol, "adjoint")
    # the same calls under capture: the same kernels in the same order
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            E2, g2 = h.forward(ph), h.adjoint(yt)[0]
        graph.replay()
    torch.cuda.current_stream().wait_stream(s)
    assert torch.equal(E2, E) and torch.equal(g2, g)
    # bands: rows of tiles of the same grid
    cut = (ny // 2) // 32 * 32
    blocks = [(0, cut), (cut, ny)]
    bands = band_holograms(torch.from_numpy(p.amp).cuda(), torch.from_numpy(p.coeff).cuda(), p.noll, ny, blocks)
    E3 = sum(b.forward(ph[r0:r1].contiguous()).cpu().numpy().astype(np.complex128) for b, (r0, r1) in zip(bands, blocks))
    assert_close(E3, E_ref, tol, "summed band forwards")
    assert_close(torch.cat([b.adjoint(yt)[0] for b in bands], 0).cpu().numpy(), g_ref, tol, "tiled band adjoints")
    # the sweep's shared nearfield image against a forward of its own per offset
    I = h.zsub_sweep(ph, 1, [-0.5, 0.25])
    Cs = torch.from_numpy(p.coeff).cuda()
    Cs[:, 1] -= 0.25                              # phase + delta Z_d: kernels with C_d - delta
    from paper_2505_08777_gb300 import Hologram
    E4 = Hologram(torch.from_numpy(p.amp).cuda(), Cs, noll=p.noll).forward(ph)
    assert_close(I[1].cpu().numpy(), (E4.abs() ** 2).cpu().numpy(), 1e-6, "sweep")   # the same kernels
    for q in [h] + bands:
        q.check()


@pytest.mark.parametrize("nx,ny,N,noll,scale", [CASES[2], CASES[4], CASES[6], *CASES[7:]])
def test_separable_gradient_matches_oracle(nx, ny, N, noll, scale):
    p, _ = _problem(nx, ny, N, noll, scale)
    Z, C, A = oracle_inputs(p)
    h = _holo(p)
    E = transform.forward(transform.field(A, p.phase0), C, Z, workers=8)
    gE = ograd.grad_E(E, p.target).astype(np.complex64)
    dph_ref, dC_ref = ograd.backward(A, p.phase0, C, Z, gE.astype(np.complex128))
    dph, dC = h.grad(torch.from_numpy(p.phase0).cuda(), torch.from_numpy(gE).cuda())
    dph, dC = dph.cpu().numpy().astype(np.float64).ravel(), dC.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(dph - dph_ref) <= GRAD_TOL * np.linalg.norm(dph_ref)
    assert np.linalg.norm(dC - dC_ref) <= GRAD_TOL * np.linalg.norm(dC_ref)
