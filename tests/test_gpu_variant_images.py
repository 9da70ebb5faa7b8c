"""The tensor-core kernels' spot images (variant 2) on a handle whose automatic
choice does not read them: coefficients set in any variant, by calls and by
replays of captured graphs, reach every later call of every variant. Each
forward is compared bit for bit with that of a handle of its own, created with
the same coefficients."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from workloads import random_problem  # noqa: E402

pytestmark = pytest.mark.gpu

NOLL = list(range(2, 12))


@pytest.fixture(scope="module")
def setup():
    p = random_problem(77, 905, 903, 70, NOLL)
    ph = torch.from_numpy(p.phase0).cuda()
    amp = torch.from_numpy(p.amp).cuda()
    rng = np.random.default_rng(5)
    Cs = [torch.from_numpy((p.coeff + rng.normal(size=p.coeff.shape)).astype(np.float32)).cuda() for _ in range(4)]
    return amp, ph, Cs


def _holo(amp, C, variant=0):
    from paper_2505_08777_gb300 import Hologram
    h = Hologram(amp, C, noll=NOLL)
    h.set_variant(variant)
    return h


def _capture(fn):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = fn()
    torch.cuda.current_stream().wait_stream(s)
    return g, out


def _want(amp, ph, C, variant=2):
    return _holo(amp, C, variant).forward(ph)


def test_replayed_forward_sees_coefficients_set_in_another_variant(setup):
    amp, ph, Cs = setup
    h = _holo(amp, Cs[0], 2)
    h.forward(ph)
    graph, E = _capture(lambda: h.forward(ph))
    h.set_variant(0)
    h.set_coefficients(Cs[1])
    graph.replay()
    assert torch.equal(E, _want(amp, ph, Cs[1]))


def test_replayed_coefficients_reach_a_later_variant(setup):
    amp, ph, Cs = setup
    h = _holo(amp, Cs[0])
    C = Cs[1].clone()
    h.forward_coeff(C, ph)
    graph, E = _capture(lambda: h.forward_coeff(C, ph))
    h.set_variant(2)
    assert torch.equal(h.forward(ph), _want(amp, ph, Cs[1]))
    h.set_variant(0)
    C.copy_(Cs[2])
    graph.replay()
    assert torch.equal(E, _want(amp, ph, Cs[2], 0))
    h.set_variant(2)
    assert torch.equal(h.forward(ph), _want(amp, ph, Cs[2]))
    # also while the variant stays, and by a forward captured in it
    later, E2 = _capture(lambda: h.forward(ph))
    C.copy_(Cs[3])
    graph.replay()
    assert torch.equal(h.forward(ph), _want(amp, ph, Cs[3]))
    C.copy_(Cs[1])
    graph.replay()
    later.replay()
    assert torch.equal(E2, _want(amp, ph, Cs[1]))


def test_captured_but_not_replayed_coefficients_do_not_count(setup):
    amp, ph, Cs = setup
    h = _holo(amp, Cs[0])
    h.set_coefficients(Cs[1])
    _capture(lambda: h.forward_coeff(Cs[2], ph))
    h.set_variant(2)
    assert torch.equal(h.forward(ph), _want(amp, ph, Cs[1]))
    # the loops' graphs: their kernels alone, on the coefficients of now
    h.set_variant(0)
    h.set_coefficients(Cs[3])
    h.set_variant(2)
    t = torch.ones(Cs[0].shape[0], device="cuda")
    got, want = [], []
    for q, out in ((h, got), (_holo(amp, Cs[3], 2), want)):
        x, w = ph.clone(), t.clone()
        E, _ = q.wgs(x, w, t, 2)
        assert q.graph_kernels(2) == q.wgs_launches(2)
        out += [x, w, E]
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_variant_change_inside_a_capture(setup):
    # no synchronisation in the call, so that the capture stays valid
    amp, ph, Cs = setup
    h = _holo(amp, Cs[0])

    def both():
        h.set_variant(2)
        return h.forward(ph)
    graph, E = _capture(both)
    graph.replay()
    assert torch.equal(E, _want(amp, ph, Cs[0]))
    h.set_variant(0)
    h.set_coefficients(Cs[1])
    graph.replay()
    assert torch.equal(E, _want(amp, ph, Cs[1]))


def test_images_reach_the_calls_that_read_them():
    # a separable forward beside a tensor-core adjoint, moment pass and loop
    p = random_problem(78, 470, 450, 300, NOLL)
    ph, amp = torch.from_numpy(p.phase0).cuda(), torch.from_numpy(p.amp).cuda()
    C1 = torch.from_numpy((p.coeff * np.float32(0.5)).astype(np.float32)).cuda()
    y = torch.polar(torch.ones(p.N), torch.arange(p.N, dtype=torch.float32)).cuda()
    t = torch.ones(p.N, device="cuda")
    fresh = _holo(amp, C1)

    def loop(h):
        x, w = ph.clone(), t.clone()
        h.wgs(x, w, t, 2)
        assert h.graph_kernels(2) == h.wgs_launches(2)
        return x
    calls = [lambda h: h.adjoint(y)[0], lambda h: h.grad(ph, y)[1], loop,
             lambda h: (h.zsub_sweep(ph, 1, [0.5]), h.adjoint(y)[0])[1]]
    for call in calls:
        h = _holo(amp, torch.from_numpy(p.coeff).cuda())
        h.forward_coeff(C1, ph)
        assert torch.equal(call(h), call(fresh))
