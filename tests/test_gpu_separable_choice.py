"""Where the automatic choice takes the separable transforms: not for one or two
spots, and not where the coefficients that a handle is created with need many
row strips. A handle that it leaves to the other kernels returns bit for bit
what their forced variant returns (1: few spots, 2 from 256); one created with
weak aberrations keeps the separable kernels when stronger ones are set, up to
the 32 strips of a tile, within the transforms' tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import REL_TOL, assert_close, oracle_inputs  # noqa: E402
from oracle import transform  # noqa: E402
from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu

LOW = list(range(2, 12))


def _problem(nx, ny, N, noll, scale):
    p = random_problem(nx + 3 * ny + N, nx, ny, N, noll, defocus_max=5.0)
    p.coeff = np.ascontiguousarray(p.coeff * np.float32(scale))
    y = torch.polar(torch.ones(N), torch.arange(N, dtype=torch.float32)).cuda()
    return p, torch.from_numpy(p.phase0).cuda(), y


def _holo(p, coeff, variant=0):
    from paper_2505_08777_gb300 import Hologram
    h = Hologram(torch.from_numpy(p.amp).cuda(), torch.from_numpy(coeff).cuda(), noll=p.noll)
    h.set_variant(variant)
    return h


def _calls(h, ph, y):
    dph, dC = h.grad(ph, y)
    x, w, t = ph.clone(), torch.ones(len(y), device="cuda"), torch.ones(len(y), device="cuda")
    E, met = h.wgs(x, w, t, 2)
    assert h.graph_kernels(2) == h.wgs_launches(2)
    h.check()
    return h.forward(ph), h.adjoint(y)[0], h.zsub_sweep(ph, 1, [0.5, -0.5]), dph, dC, x, w, E


@pytest.mark.parametrize("nx,ny,N,noll,scale,variant", [
    (901, 930, 1, LOW, 1.0, 1),
    (930, 901, 2, LOW, 1.0, 1),
    (3000, 2000, 2, [2, 3, 4, 5, 6], 1.0, 1),
    (577, 590, 260, LOW, 30.0, 2),
])
def test_left_to_the_other_kernels(nx, ny, N, noll, scale, variant):
    p, ph, y = _problem(nx, ny, N, noll, scale)
    got, want = (_calls(_holo(p, p.coeff, v), ph, y) for v in (0, variant))
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("nx,ny,N,noll,other", [(901, 930, 11, LOW, True), (901, 930, 12, LOW, False),
                                                (1030, 1000, 23, [2, 3, 4, 5, 6], True),
                                                (1030, 1000, 24, [2, 3, 4, 5, 6], False)])
def test_a_field_on_few_spots(nx, ny, N, noll, other):
    p, ph, _ = _problem(nx, ny, N, noll, 0.1)
    Z, C, A = oracle_inputs(p)
    f = torch.polar(torch.from_numpy(p.amp).cuda(), ph)
    h = _holo(p, p.coeff)
    assert h.launch_info()["kernels"] & 16
    E = h.forward_field(f)
    assert torch.equal(E, _holo(p, p.coeff, 1).forward_field(f)) == other
    ref = transform.forward(f.cpu().numpy().astype(np.complex128).ravel(), C, Z, workers=8)
    assert_close(E.cpu().numpy(), ref, 1e-5, "field")
    h.check()


@pytest.mark.parametrize("nx,ny,N,scale", [(577, 590, 100, 30.0), (640, 600, 97, 6.0), (905, 903, 161, 30.0)])
def test_stronger_coefficients_set_later(nx, ny, N, scale):
    p, ph, y = _problem(nx, ny, N, LOW, scale)
    Z, C, A = oracle_inputs(p)
    h = _holo(p, np.ascontiguousarray(p.coeff / np.float32(100.0)))
    other = _holo(p, p.coeff, 2)
    h.set_coefficients(torch.from_numpy(p.coeff).cuda())
    E, g = h.forward(ph), h.adjoint(y)[0]
    assert not torch.equal(g, other.adjoint(y)[0])      # another kernel's rounding
    assert_close(E.cpu().numpy(), transform.forward(transform.field(A, p.phase0), C, Z, workers=8), REL_TOL, "forward")
    assert_close(g.cpu().numpy(), transform.adjoint(y.cpu().numpy().astype(np.complex128), C, Z, workers=8), REL_TOL,
                 "adjoint")
    h.check()


def test_a_handle_without_memory_for_them_serves_on_the_other_kernels():
    from paper_2505_08777_gb300 import _lib
    lib = _lib.load()
    sizes, refuse = [], set()
    stream = torch.cuda.current_stream().cuda_stream

    def alloc(ctx, n, s):
        sizes.append(n)
        if len(sizes) - 1 in refuse:
            return None
        return torch.cuda.caching_allocator_alloc(n, 0, stream)

    hooks = _lib.ALLOC_FN(alloc), _lib.FREE_FN(lambda ctx, p, s: torch.cuda.caching_allocator_delete(p))
    p, ph, y = _problem(905, 903, 300, LOW, 1.0)
    assert lib.ash_set_allocator(*hooks, None) == 0
    try:
        full = _holo(p, p.coeff)
        block = sizes[-1]                               # taken last
        E_sep, full_bytes = full.forward(ph), full.workspace_bytes()
        full.close()
        count = len(sizes)
        sizes.clear()
        refuse.add(count - 1)
        h = _holo(p, p.coeff)
        assert len(sizes) == count and sizes[-1] == block
        assert h.workspace_bytes() == full_bytes - block
        got = _calls(h, ph, y)
        h.close()
    finally:
        torch.cuda.synchronize()
        lib.ash_set_allocator(_lib.ALLOC_FN(0), _lib.FREE_FN(0), None)
    want = _calls(_holo(p, p.coeff, 2), ph, y)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert_close(E_sep.cpu().numpy(), want[0].cpu().numpy(), 1e-5, "separable forward")


# launch-info bits: 16 / 32 / 64 separable forward, adjoint, moments; 128 / 256 forward and adjoint of a loop
@pytest.mark.parametrize("nx,ny,N,noll,scale,bits", [
    (417, 403, 65, LOW, 0.05, 16),
    (399, 700, 65, LOW, 0.05, 0),
    (561, 577, 129, LOW, 0.05, 16 | 32 | 128 | 256),
    (577, 590, 260, LOW, 30.0, 0),
    (640, 700, 63, LOW, 0.05, 0),
    (803, 801, 7, LOW, 0.1, 16 | 32 | 128 | 256),
    (905, 903, 161, LOW, 0.1, 16 | 32 | 64 | 128 | 256),
    (901, 930, 2, LOW, 1.0, 0),
    (901, 930, 3, LOW, 0.1, 0),
    (901, 930, 4, LOW, 0.1, 32 | 64 | 256),
    (901, 930, 6, LOW, 0.1, 16 | 32 | 64 | 128 | 256),
    (1030, 1030, 15, [2, 3, 4, 5, 6], 1.0, 32 | 64 | 256),
    (233, 201, 231, [2, 3, 4, 5, 6], 1.0, 16 | 32),
    (901, 930, 20, [2, 3, 4, 5, 6], 1.0, 16 | 32 | 64 | 128 | 256),
    (600, 600, 70, list(range(2, 17)), 0.05, 0),          # degree 5
])
def test_launch_info_tells_the_choice(nx, ny, N, noll, scale, bits):
    p, _, _ = _problem(nx, ny, N, noll, scale)
    h = _holo(p, p.coeff)
    assert h.launch_info()["kernels"] & ~15 == bits
    h.set_variant(2)
    assert h.launch_info()["kernels"] & ~15 == 0


@pytest.mark.parametrize("nx,ny,N,scale", [(905, 903, 161, 7.5), (620, 610, 260, 2.2)])
def test_forward_alone_beside_the_other_adjoint(nx, ny, N, scale):
    # strips enough for the adjoint's line, not for the forward's
    p, ph, y = _problem(nx, ny, N, LOW, scale)
    Z, C, A = oracle_inputs(p)
    h = _holo(p, p.coeff)
    assert h.launch_info()["kernels"] & ~15 == 16 | 128
    got = _calls(h, ph, y)
    assert_close(got[0].cpu().numpy(), transform.forward(transform.field(A, p.phase0), C, Z, workers=8), REL_TOL, "forward")
    assert torch.equal(got[1], _holo(p, p.coeff, 2 if N >= 256 else 1).adjoint(y)[0])
